// vb_resident.h -- the plan of the shared-memory resident Viana-Bray sweeps (vb_resident.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sg_internal.cuh"

namespace sg {

constexpr int kResMain = 12;                // warps that update vertices
constexpr int kResHelp = 6;                 // warps that work out the next sweep's acceptance
constexpr int kResThreads = 32 * (kResMain + kResHelp);
// one CTA for a graph; a cluster, each CTA with the words of its own vertices, read by the others; a
// cluster, each CTA with a copy of all words, to which every update is written
constexpr int kResSolo = 0, kResCluster = 1, kResCopies = 2;
constexpr int kResMaxCluster = 16;          // CTAs of one graph's cluster (a power of two)
constexpr int kResMaxSmem = 218 * 1024;     // dynamic shared memory of one CTA, beside its static tables

struct VbResident {
    const uint32_t* graph_class_slice;  // [n_colours n_graphs + 1] first slice of each (class, graph)
    uint32_t cluster, log_cluster;
    bool copies;
    bool wide;                          // some slice has more than 15 entries (vb_resident.cu: kResPlanes)
    int graph_slices;                   // slices of the largest graph
    int max_slices;                     // slices and entries of the fullest CTA
    uint32_t max_entries;
};

// word_slices: slices whose spin words a CTA holds
size_t vb_resident_smem(int R, int word_slices, int max_slices, int64_t max_entries);
// clusters of this plan that the GPU holds at once (0: the plan does not fit)
int vb_resident_clusters(int R, const VbResident& rs);
int vb_resident_sweeps(const VbPackedDev& d, const VbResident& rs, uint32_t t0,
                       int n_sweeps, cudaStream_t st);

}  // namespace sg
