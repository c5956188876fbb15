// Read-only view of a device graph (iso_graph is defined in iso_api.cu), for
// code outside that file that launches the kernels on it: the
// allocation-free entry point.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "iso.h"

struct iso_graph_view {
    int n, L, tau_max, num_sms;
    int device;  // CUDA device the graph was uploaded to
    int64_t m;
    const uint32_t *down_off, *up_off, *pair_off;
    const int2 *down_arc, *pair_ids;
    const int4* up_arc;
    const int32_t *pair_head, *pos, *level_off, *pair_owner;
    const uint2* core_arc;
    const uint32_t* level_arc;
    const int32_t* h_level_off;
};

// Fills v from g.  ISO_E_INVAL if either is NULL.
int iso_graph_view_of(const iso_graph* g, iso_graph_view* v);
