// sk_fields_warp.h -- the order of the fields warp's work in a chain CTA of the persistent SK sweep
// (sk_persist.cu), apart from the instructions it is made of, so that it also runs on the host.
#pragma once

#ifdef __CUDACC__
#define SG_FIELDS_WARP __device__ __forceinline__
#else
#define SG_FIELDS_WARP inline
#endif

namespace sg {

constexpr int kChainStages = 3;  // staged blocks ahead of the chain

// Blocks 0 .. nk - 1 (block b = k mod nb of its sweep) go to stage k mod kChainStages: once the stage
// is released (wait_empty, phase k / kChainStages - 1) and, for k > L, the block's fields are published
// (wait_published), copy brings them into the stage.  A wait that gives up ends the work.  Either way
// every copy lands (drain) before the warp leaves.  That does not depend on whether anything has failed
// so far: the last copies are issued blocks before they are used, and a CTA whose other warps give up
// after that must not exit with a copy into its shared memory on its way.  Without a failure the
// other warps wait for the same copies.
template <class Ops>
SG_FIELDS_WARP void run_fields_warp(Ops& ops, int nk, int nb, int L) {
    int last_fill[kChainStages];
    for (int s = 0; s < kChainStages; ++s) last_fill[s] = -1;
    for (int k = 0, b = 0; k < nk; ++k, b = (b + 1 == nb) ? 0 : b + 1) {
        const int s = k % kChainStages;
        if (k >= kChainStages && !ops.wait_empty(s, (unsigned)(k / kChainStages - 1) & 1u)) break;
        if (k > L && !ops.wait_published(b, k)) break;
        ops.copy(s, b, k > L);
        last_fill[s] = k;
    }
    for (int s = 0; s < kChainStages; ++s)
        if (last_fill[s] >= 0) ops.drain(s, (unsigned)(last_fill[s] / kChainStages) & 1u);
}

}  // namespace sg
