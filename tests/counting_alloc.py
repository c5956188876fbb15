"""A device allocator for graphs (iso_alloc) that logs what is taken and can refuse
to hand out more than a number of bytes."""

from paper_1512_09090_gb300 import _lib


class CountingAlloc(_lib._TorchAlloc):
    def __init__(self, device):
        super().__init__(device)
        self.limit = None  # bytes handed out at a time, at most
        self.live = self.peak = 0
        self.size, self.log = {}, []

    def _alloc(self, ctx, size, stream):
        if self.limit is not None and self.live + size > self.limit:
            return None
        p = super()._alloc(ctx, size, stream)
        if p:
            self.size[p] = size
            self.log.append(size)
            self.live += size
            self.peak = max(self.peak, self.live)
        return p

    def _free(self, ctx, ptr, stream):
        self.live -= self.size.pop(ptr)
        super()._free(ctx, ptr, stream)


def upload(ch, monkeypatch):
    """The hierarchy on the device, with its allocator."""
    monkeypatch.setattr(_lib, "_TorchAlloc", CountingAlloc)
    dg = _lib.iso_upload_graph(ch)
    return dg, dg._alloc
