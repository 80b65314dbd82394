// vb_resident.cu -- packed Viana-Bray sweeps of small graphs for sm_103a: one thread-block cluster per
// graph keeps the whole instance (spin words, neighbours, couplings, labels) in the shared memory
// of its CTAs and runs all the sweeps of a call in one launch.  Dynamics as in vb_sweep.cu: one
// thread per vertex for 64 lanes and R replicas (multispin coding, SI section 2), one colour class
// (an independent set) at a time.
//
// What bounds it: the latency of one class (the neighbours' words, the counting, a barrier), times
// the classes.  In shared memory a gathered word pair is 30 cycles away, or a few hundred in a
// neighbouring CTA, against about 700 in L2, and the classes are separated by a cluster barrier
// (a CTA barrier for one CTA) instead of a grid-wide one through L2.  Six of
// the 18 warps work out the acceptance of a class for the next sweep while the others update it.
//
// In a cluster the words that neighbours read are either where their owner keeps them, or every
// CTA holds a copy of all words: gathers from another CTA take about 4 cycles for each 16 bytes, so
// where the copies fit it is cheaper to send every updated slice to the other CTAs (512 bytes for two
// replicas, whole lines, about 43 cycles each) and gather at home.
//
// us a sweep, two replicas, before (grid-wide) -> now: N = 1000 18 -> 4.4 (one CTA), 2500 12.4 -> 4.9,
// bipartite 4096 9.8 -> 2.9, 6000 14 -> 6.4, 9000 15 -> 8.0.
//
// The slices (32 vertices) of a class are dealt in turn to the CTAs of the cluster, and in a CTA to
// its warps.
#include "../../include/sg.h"
#include "sg_internal.cuh"
#include "vb_bits.cuh"
#include "vb_resident.h"

namespace sg {

namespace {

// Counter planes: slices up to width 15, and wider ones (degrees up to 63).  Both take their entries in
// chunks: one at a time a class lasts as long as its widest slice (us a sweep, one at a time -> chunks:
// N = 3000, degree 16, R = 2 19.1 -> 14.4, R = 4 126 -> 38; degree 24, R = 2 114 -> 54).  Graphs without wide
// slices run kernels without their counting, whose registers would slow the others down (R = 4, N = 1500
// 8.2 us a sweep, 8.6 with it).
constexpr int kResPlanes = 4, kResWidePlanes = 6;
static_assert(SG_VB_MAX_DEGREE < (1 << kResWidePlanes), "the counter holds every degree");

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}

template <int R, int MODE>
__device__ __forceinline__ SpinWords<R> gather_near(uint32_t a) {
    SpinWords<R> s;
    if constexpr (R == 1) {
        if constexpr (MODE != kResCluster) asm volatile("ld.shared.u64 %0, [%1];" : "=l"(s.v[0]) : "r"(a));
        else asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(s.v[0]) : "r"(a));
    } else {
#pragma unroll
        for (int h = 0; h < R / 2; ++h) {
            if constexpr (MODE != kResCluster)
                asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(s.v[2 * h]), "=l"(s.v[2 * h + 1]) : "r"(a + 16 * h));
            else
                asm volatile("ld.shared::cluster.v2.u64 {%0, %1}, [%2];" : "=l"(s.v[2 * h]), "=l"(s.v[2 * h + 1]) : "r"(a + 16 * h));
        }
    }
    return s;
}

template <int R>
__device__ __forceinline__ void store_remote(uint32_t a, const SpinWords<R>& s) {
    if constexpr (R == 1) {
        asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(s.v[0]) : "memory");
    } else {
#pragma unroll
        for (int h = 0; h < R / 2; ++h)
            asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(a + 16 * h), "l"(s.v[2 * h]), "l"(s.v[2 * h + 1]) : "memory");
    }
}

// every thread's words of a class are visible to the cluster, and no thread reads on before
template <int MODE>
__device__ __forceinline__ void class_barrier_arrive() {
    if constexpr (MODE != kResSolo) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
template <int MODE>
__device__ __forceinline__ void class_barrier_wait() {
    if constexpr (MODE == kResSolo) __syncthreads();
    else asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

}  // namespace

template <int R, int MODE, bool WIDE>
__global__ void __launch_bounds__(kResThreads, 1)
    k_vb_resident(VbPackedDev d, VbResident rs, uint32_t t0, uint32_t n_sweeps) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint32_t c_lo[kVbMaxColours], c_hi[kVbMaxColours];       // slices of the graph's classes
    __shared__ uint16_t first_of[kVbMaxColours + 1][kResMaxCluster];    // local slices before a class, per CTA
    __shared__ uint32_t c_before[kVbMaxColours + 1];                    // the graph's slices before a class
    __shared__ __align__(16) uint32_t thr[R * kVbThrStride];
    uint64_t* S = reinterpret_cast<uint64_t*>(smem);                            // [slots][R]
    uint64_t* J = S + (size_t)(MODE == kResCopies ? rs.graph_slices : rs.max_slices) * 32 * R;                           // [entries]
    uint32_t* nbr = reinterpret_cast<uint32_t*>(J + rs.max_entries);            // [entries] address of the words
    uint32_t* vinfo = nbr + rs.max_entries;                                     // [slots]
    uint32_t* base = vinfo + rs.max_slices * 32;                                // [slices + 1] first entry
    uint8_t* kmins = reinterpret_cast<uint8_t*>(base + rs.max_slices + 1);      // [2][slots][R] this sweep's, the next's
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    constexpr uint32_t warps = kResThreads / 32;
    const uint32_t C = MODE == kResSolo ? 1u : rs.cluster, lc = rs.log_cluster;
    const uint32_t rank = MODE == kResSolo ? 0u : cluster_rank();
    const uint32_t g = MODE == kResSolo ? blockIdx.x : blockIdx.x >> lc;
    const uint32_t nc = (uint32_t)d.n_colours, ng = (uint32_t)d.n_graphs;
    const uint64_t seed = __ldg(d.seeds + g);

    for (uint32_t c = tid; c < nc; c += kResThreads) {
        c_lo[c] = __ldg(rs.graph_class_slice + c * ng + g);
        c_hi[c] = __ldg(rs.graph_class_slice + c * ng + g + 1);
    }
    for (uint32_t i = tid; i < (uint32_t)(R * kVbThrStride); i += kResThreads)
        thr[i] = __ldg(d.thr + g * (R * kVbThrStride) + i);
    __syncthreads();
    if (tid == 0) {
        uint32_t n = 0;
        for (uint32_t c = 0; c < nc; ++c) {
            c_before[c] = n;
            n += c_hi[c] - c_lo[c];
        }
    }
    if (tid < C) {
        uint32_t n = 0;
        for (uint32_t c = 0; c < nc; ++c) {
            first_of[c][tid] = (uint16_t)n;
            const uint32_t m = c_hi[c] - c_lo[c];
            n += m > tid ? (m - tid + C - 1) >> lc : 0u;
        }
        first_of[nc][tid] = (uint16_t)n;
    }
    __syncthreads();
    const uint32_t n_local = first_of[nc][rank];
    // the local slices' first entries: widths, then their running sum (warp 0)
    auto slice_of = [&](uint32_t l) -> uint32_t {
        uint32_t c = 0;
        while (l >= first_of[c + 1][rank]) ++c;
        return c_lo[c] + ((l - first_of[c][rank]) << lc) + rank;
    };
    for (uint32_t l = tid; l < n_local; l += kResThreads) {
        const uint32_t s = slice_of(l);
        base[l + 1] = __ldg(d.slice_base + s + 1) - __ldg(d.slice_base + s);
    }
    if (tid == 0) base[0] = 0u;
    __syncthreads();
    if (warp == 0) {
        uint32_t sum = 0;
        for (uint32_t l0 = 0; l0 < n_local; l0 += 32) {
            uint32_t v = l0 + lane < n_local ? base[l0 + lane + 1] : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, v, o);
                if (lane >= (uint32_t)o) v += u;
            }
            if (l0 + lane < n_local) base[l0 + lane + 1] = sum + v;
            sum += __shfl_sync(0xFFFFFFFFu, v, 31);
        }
    }
    __syncthreads();
    // the instance into shared memory, one slice per warp; a neighbour's slot becomes the address
    // of its words
    for (uint32_t l = warp; l < n_local; l += warps) {
        const uint32_t s = slice_of(l);
        const uint32_t slot = s * 32 + lane;
        vinfo[l * 32 + lane] = __ldg(d.vinfo + slot);
        if constexpr (MODE != kResCopies) {
            const SpinWords<R> w = load_words<R>(d.S + (int64_t)slot * R);
#pragma unroll
            for (int r = 0; r < R; ++r) S[(l * 32 + lane) * R + r] = w.v[r];
        }
        const uint32_t gb = __ldg(d.slice_base + s);
        for (uint32_t e = base[l] + lane; e < base[l + 1]; e += 32) {
            const uint32_t ge = gb + (e - base[l]);
            J[e] = __ldg(d.jb + ge);
            const uint32_t j = __ldg(d.col + ge), sj = j >> 5;
            uint32_t c = 0;
            while (sj < c_lo[c] || sj >= c_hi[c]) ++c;  // every neighbour lies in a class of this graph
            if constexpr (MODE == kResCopies) {
                nbr[e] = smem_addr(S + ((c_before[c] + sj - c_lo[c]) * 32 + (j & 31u)) * R);
                continue;
            }
            const uint32_t i = sj - c_lo[c], owner = i & (C - 1u);
            const uint32_t a = smem_addr(S + ((first_of[c][owner] + (i >> lc)) * 32 + (j & 31u)) * R);
            nbr[e] = MODE == kResSolo ? a : cluster_addr(a, owner);
        }
    }
    if constexpr (MODE == kResCopies) {  // all the graph's words
        for (uint32_t c = 0; c < nc; ++c)
            for (uint32_t i = tid; i < (c_hi[c] - c_lo[c]) * 32; i += kResThreads) {
                const SpinWords<R> w = load_words<R>(d.S + ((int64_t)c_lo[c] * 32 + i) * R);
#pragma unroll
                for (int r = 0; r < R; ++r) S[((size_t)c_before[c] * 32 + i) * R + r] = w.v[r];
            }
    }
    // Acceptance of the vertices of local slice l at time t: a lane flips iff its unsatisfied count u
    // reaches ceil((d - m*) / 2), m* the largest accepted m (the accepted m are a prefix 1..m*)
    auto accept = [&](uint32_t l, uint32_t t) {
        const uint32_t vi = vinfo[l * 32 + lane];
        const int deg = vi == kInactive ? 0 : (int)(vi >> kDegShift);
        const uint4 rnd = philox4x32_10(make_uint4(vi & kOrigMask, t, 0u, 0u), (uint32_t)seed,
                                        (uint32_t)(seed >> 32));
        uint32_t packed = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t r32 = uint4_word(rnd, r);
            const uint4 th = *reinterpret_cast<const uint4*>(thr + r * kVbThrStride);
            int ms = (int)(r32 < th.y) + (int)(r32 < th.z) + (int)(r32 < th.w);
            if (ms == 3)
                while (ms < deg && r32 < thr[r * kVbThrStride + ms + 1]) ++ms;
            ms = ms < deg ? ms : deg;
            packed |= (uint32_t)((deg - ms + 1) >> 1) << (8 * r);
        }
        uint8_t* k = kmins + ((size_t)(t & 1u) * rs.max_slices * 32 + l * 32 + lane) * R;
        if constexpr (R == 1) *k = (uint8_t)packed;
        else if constexpr (R == 2) *reinterpret_cast<uint16_t*>(k) = (uint16_t)packed;
        else *reinterpret_cast<uint32_t*>(k) = packed;
    };
    __syncthreads();  // the labels are in place
    for (uint32_t l = warp; l < n_local; l += warps) accept(l, t0);
    __syncthreads();
    class_barrier_arrive<MODE>();

    for (uint32_t t = t0, te = t0 + n_sweeps; t != te; ++t)
        for (uint32_t c = 0; c < nc; ++c) {
            const uint32_t l_end = first_of[c + 1][rank];
            class_barrier_wait<MODE>();
            if (warp >= kResMain) {
                // the next sweep's acceptance of this class, beside its update of this sweep
                for (uint32_t l = first_of[c][rank] + warp - kResMain; l < l_end; l += warps - kResMain)
                    accept(l, t + 1);
            }
            for (uint32_t l = warp < kResMain ? first_of[c][rank] + warp : l_end; l < l_end; l += kResMain) {
                const uint32_t i = ((l - first_of[c][rank]) << lc) + rank;  // the slice's place in its class
                uint64_t* own = S + ((MODE == kResCopies ? c_before[c] + i : l) * 32 + lane) * R;
                SpinWords<R> si = load_words<R>(own);
                uint32_t e = base[l] + lane;
                const uint32_t end = base[l + 1];  // width = (end - base[l]) / 32
                const uint32_t vi = vinfo[l * 32 + lane];
                const uint8_t* k = kmins + ((size_t)(t & 1u) * rs.max_slices * 32 + l * 32 + lane) * R;
                int kmin[R];
                if constexpr (R == 1) {
                    kmin[0] = *k;
                } else {
                    const uint32_t packed = R == 2 ? *reinterpret_cast<const uint16_t*>(k) : *reinterpret_cast<const uint32_t*>(k);
#pragma unroll
                    for (int r = 0; r < R; ++r) kmin[r] = (int)((packed >> (8 * r)) & 255u);
                }
                // (in one CTA with four replicas the compiler orders the loads of narrow slices better beside
                // a plain loop for wide ones, which no graph of such a launch has: N = 300 4.75 us a sweep,
                // without 5.0; N = 1000 7.43, 7.66)
                constexpr bool kPlainWide = !WIDE && R == 4 && MODE == kResSolo;
                if ((!WIDE && !kPlainWide) || end - base[l] <= 32u * ((1u << kResPlanes) - 1u)) {
                    constexpr int CH = R == 4 ? 4 : 8;  // entries whose words are on their way at once
                    uint64_t p[R][kResPlanes];
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int b = 0; b < kResPlanes; ++b) p[r][b] = 0ull;
                    for (; e < end; e += 32 * CH) {
                        SpinWords<R> w[CH];
                        uint64_t Je[CH];
#pragma unroll
                        for (int u = 0; u < CH; ++u) {
                            w[u] = si;  // an absent entry counts nothing
                            Je[u] = 0ull;
                            if (e + 32 * u < end) {
                                w[u] = gather_near<R, MODE>(nbr[e + 32 * u]);
                                Je[u] = J[e + 32 * u];
                            }
                        }
#pragma unroll
                        for (int h = 0; h < CH; h += 4) {
                            if (e + 32 * h >= end) break;  // warp-uniform
#pragma unroll
                            for (int r = 0; r < R; ++r)
                                bitslice_add4<kResPlanes>(p[r], si.v[r] ^ w[h].v[r] ^ Je[h],
                                                          si.v[r] ^ w[h + 1].v[r] ^ Je[h + 1],
                                                          si.v[r] ^ w[h + 2].v[r] ^ Je[h + 2],
                                                          si.v[r] ^ w[h + 3].v[r] ^ Je[h + 3]);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) si.v[r] ^= at_least<kResPlanes>(p[r], kmin[r]);
                } else if constexpr (WIDE) {
                    // six planes, and of four replicas two at a time (all four would need more than the 96
                    // registers of 18 warps)
                    constexpr int RW = R == 1 ? 1 : 2, CH = 8;
#pragma unroll
                    for (int r0 = 0; r0 < R; r0 += RW) {
                        uint64_t p[RW][kResWidePlanes];
#pragma unroll
                        for (int r = 0; r < RW; ++r)
#pragma unroll
                            for (int b = 0; b < kResWidePlanes; ++b) p[r][b] = 0ull;
                        for (uint32_t i = e; i < end; i += 32 * CH) {
                            SpinWords<RW> w[CH];
                            uint64_t Je[CH];
#pragma unroll
                            for (int u = 0; u < CH; ++u) {
#pragma unroll
                                for (int r = 0; r < RW; ++r) w[u].v[r] = si.v[r0 + r];
                                Je[u] = 0ull;
                                if (i + 32 * u < end) {
                                    w[u] = gather_near<RW, MODE>(nbr[i + 32 * u] + 8 * r0);
                                    Je[u] = J[i + 32 * u];
                                }
                            }
#pragma unroll
                            for (int h = 0; h < CH; h += 4) {
                                if (i + 32 * h >= end) break;  // warp-uniform
#pragma unroll
                                for (int r = 0; r < RW; ++r)
                                    bitslice_add4<kResWidePlanes>(p[r], si.v[r0 + r] ^ w[h].v[r] ^ Je[h],
                                                                  si.v[r0 + r] ^ w[h + 1].v[r] ^ Je[h + 1],
                                                                  si.v[r0 + r] ^ w[h + 2].v[r] ^ Je[h + 2],
                                                                  si.v[r0 + r] ^ w[h + 3].v[r] ^ Je[h + 3]);
                            }
                        }
#pragma unroll
                        for (int r = 0; r < RW; ++r) si.v[r0 + r] ^= at_least<kResWidePlanes>(p[r], kmin[r0 + r]);
                    }
                } else if constexpr (kPlainWide) {
                    uint64_t p[R][kResWidePlanes];
#pragma unroll
                    for (int r = 0; r < R; ++r)
#pragma unroll
                        for (int b = 0; b < kResWidePlanes; ++b) p[r][b] = 0ull;
                    for (; e < end; e += 32) {
                        const SpinWords<R> w = gather_near<R, MODE>(nbr[e]);
#pragma unroll
                        for (int r = 0; r < R; ++r) bitslice_add<kResWidePlanes>(p[r], si.v[r] ^ w.v[r] ^ J[e]);
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) si.v[r] ^= at_least<kResWidePlanes>(p[r], kmin[r]);
                }
                if (vi != kInactive) {
#pragma unroll
                    for (int r = 0; r < R; ++r) own[r] = si.v[r];
                    if constexpr (MODE == kResCopies) {
                        const uint32_t a = smem_addr(own);
                        for (uint32_t k = 1; k < C; ++k) store_remote<R>(cluster_addr(a, (rank + k) & (C - 1u)), si);
                    }
                }
            }
            class_barrier_arrive<MODE>();
        }
    class_barrier_wait<MODE>();  // no CTA leaves while another may read its words
    for (uint32_t l = warp; l < n_local; l += warps) {
        const uint32_t s = slice_of(l);
        uint32_t at = l;
        if constexpr (MODE == kResCopies) {
            uint32_t c = 0;
            while (l >= first_of[c + 1][rank]) ++c;
            at = c_before[c] + s - c_lo[c];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) d.S[((int64_t)s * 32 + lane) * R + r] = S[(at * 32 + lane) * R + r];
    }
}

size_t vb_resident_smem(int R, int word_slices, int max_slices, int64_t max_entries) {
    return (size_t)word_slices * 32 * R * 8 + (size_t)max_entries * 12 + (size_t)max_slices * 32 * 4 +
           ((size_t)max_slices + 1) * 4 + (size_t)max_slices * 64 * R;
}

template <int R, int MODE, bool WIDE>
static cudaError_t resident_config(const VbResident& rs, int n_graphs, cudaLaunchConfig_t& cfg,
                                   cudaLaunchAttribute* attr) {
    auto kern = k_vb_resident<R, MODE, WIDE>;
    const size_t smem = vb_resident_smem(R, rs.copies ? rs.graph_slices : rs.max_slices, rs.max_slices, rs.max_entries);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kResMaxSmem);
    if (e != cudaSuccess) return e;
    if (MODE != kResSolo) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(n_graphs * (int)rs.cluster));
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = rs.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = MODE == kResSolo ? 0 : 1;
    return cudaSuccess;
}

template <int R, int MODE, bool WIDE>
static int resident_clusters(const VbResident& rs) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    int n = 0;
    if (resident_config<R, MODE, WIDE>(rs, 1, cfg, attr) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if constexpr (MODE == kResSolo) {
        int dev = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_vb_resident<R, MODE, WIDE>, kResThreads,
                                                          cfg.dynamicSmemBytes) != cudaSuccess ||
            cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return n * sms;
    }
    if (cudaOccupancyMaxActiveClusters(&n, k_vb_resident<R, MODE, WIDE>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <int R, bool WIDE>
static int resident_clusters_mode(const VbResident& rs) {
    return rs.cluster == 1 ? resident_clusters<R, kResSolo, WIDE>(rs)
           : rs.copies ? resident_clusters<R, kResCopies, WIDE>(rs)
                               : resident_clusters<R, kResCluster, WIDE>(rs);
}

int vb_resident_clusters(int R, const VbResident& rs) {
    if (vb_resident_smem(R, rs.copies ? rs.graph_slices : rs.max_slices, rs.max_slices, rs.max_entries) > (size_t)kResMaxSmem) return 0;
    switch (R) {
        case 1: return rs.wide ? resident_clusters_mode<1, true>(rs) : resident_clusters_mode<1, false>(rs);
        case 2: return rs.wide ? resident_clusters_mode<2, true>(rs) : resident_clusters_mode<2, false>(rs);
        case 4: return rs.wide ? resident_clusters_mode<4, true>(rs) : resident_clusters_mode<4, false>(rs);
        default: return 0;
    }
}

template <int R, int MODE, bool WIDE>
static int resident_launch(const VbPackedDev& d, const VbResident& rs, uint32_t t0,
                           int n_sweeps, cudaStream_t st) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    if (resident_config<R, MODE, WIDE>(rs, d.n_graphs, cfg, attr) != cudaSuccess) return -1;
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, k_vb_resident<R, MODE, WIDE>, d, rs, t0, (uint32_t)n_sweeps) ==
                   cudaSuccess ? 1 : -1;
}

template <int R, bool WIDE>
static int resident_launch_mode(const VbPackedDev& d, const VbResident& rs, uint32_t t0,
                                int n_sweeps, cudaStream_t st) {
    return rs.cluster == 1 ? resident_launch<R, kResSolo, WIDE>(d, rs, t0, n_sweeps, st)
           : rs.copies ? resident_launch<R, kResCopies, WIDE>(d, rs, t0, n_sweeps, st)
                               : resident_launch<R, kResCluster, WIDE>(d, rs, t0, n_sweeps, st);
}

int vb_resident_sweeps(const VbPackedDev& d, const VbResident& rs, uint32_t t0,
                       int n_sweeps, cudaStream_t st) {
    if (n_sweeps <= 0) return 0;
    switch (d.R) {
        case 1: return rs.wide ? resident_launch_mode<1, true>(d, rs, t0, n_sweeps, st)
                               : resident_launch_mode<1, false>(d, rs, t0, n_sweeps, st);
        case 2: return rs.wide ? resident_launch_mode<2, true>(d, rs, t0, n_sweeps, st)
                               : resident_launch_mode<2, false>(d, rs, t0, n_sweeps, st);
        case 4: return rs.wide ? resident_launch_mode<4, true>(d, rs, t0, n_sweeps, st)
                               : resident_launch_mode<4, false>(d, rs, t0, n_sweeps, st);
        default: return -1;
    }
}

}  // namespace sg
