// vb_sweep.cu -- the packed Viana-Bray sweep for sm_103a: several sweeps in one cooperative launch,
// one thread per vertex for all 64 lanes and all R replicas (multispin coding, SI section 2), one
// colour class (an independent set) at a time, the generalisation of the bipartite half-updates of
// SI section 3, with a grid-wide barrier between classes.
//
// A warp owns the same slices (32 vertices of one class, degree-sorted) in every sweep, or, far beyond L2
// and with four replicas, its first two of a class, and claims the others.  Its work is a chain of chunks of
// four (or eight) sliced-ELL entries: while the neighbours' words of one chunk are on their way from L2, the
// neighbour slots and coupling words of the next chunk (of the next slice, the next class or the next sweep)
// are already being read into registers: nothing a sweep writes, except a vertex's own words, which only
// this thread writes or, in a claimed slice, another one before a barrier that was passed.  The next slice's
// random numbers and acceptance thresholds are worked out before the barrier that admits its gathers.
//
// What bounds it.  Small and middling graphs: a class takes about 2.1 us of latencies (the stores'
// release, the barrier's way through L2 and back, a gather) before any work.  Large ones: a sweep
// of N = 2^22 (degree 4, two replicas) reads 84 bytes per vertex from HBM (33 % of its peak), gathers
// 16.8 million word pairs, each a 32-byte sector of L2 (47 %) and a tag of L1 (51 %), and issues 500
// instructions per slice (42 %).  Far beyond L2 HBM: N = 2^24 moves 5.9 GB a sweep, 64 bytes for nearly every
// gather, at 6.5 TB/s, 0.96 of the rate of a plain copy.  us a sweep, before (groups staged by bulk copies
// into shared-memory rings, a launch per sweep) -> now: N = 2^24 950 -> 903, 2^22 129 -> 122, 2^20 49 -> 37,
// bipartite 2^18 14.2 -> 9.5, N = 300007 with one replica (a launch per class) 30.8 -> 15, N = 20011 with
// four 24.9 -> 14.  Without the rings there is no pipeline to fill and drain in each class, and no launch gap.
#include <algorithm>
#include <type_traits>

#include "../../include/sg.h"
#include "sg_internal.cuh"
#include "vb_bits.cuh"

namespace sg {

namespace {

constexpr uint32_t kClaimGroups = kVbClaimGroups;

// Threads of a CTA (two CTAs share an SM), for chunks of CH entries, without and with claimed slices.
// Beyond L2 no register may spill: the spilled words go to HBM with the rest (N = 2^23, R = 2: 32 bytes a thread
// 402 us a sweep, none 286).  Four replicas with chunks of 8 need 226 registers (128 threads: N = 20011 16.1 us
// a sweep, N = 10^5 23.3; 192 threads with spills 17.4, 25.9; since, 14.0 and 18.3), with chunks of 4 157.
template <int R, int CH, bool kClaims>
struct SweepShape {
    static constexpr int threads = CH == 8 ? (R == 4 ? 128 : 256) : R == 1 ? 384 : R == 4 ? 192 : kClaims ? 256 : 320;
};

// Graphs whose thresholds are kept in shared memory, 32 KB for four replicas; a batch of more reads them through
// L1 (batches of 17 to 32 graphs gained 1.5 % from 16; more were not tried).
constexpr int kSweepTables = 32;
// Counter planes: slices up to width 15, and wider ones (degrees up to 63).  Both take their entries in
// chunks: one entry at a time, each waiting for its slot and then its words, a class lasts as long as its
// widest slice (us a sweep, one at a time -> chunks: N = 20000, degree 12, R = 2 55.8 -> 29.2, R = 4
// 102 -> 37; N = 200000, degree 16, R = 2 82.7 -> 45.7; also N = 2^23, degree 4, R = 2 297 -> 282, where a few
// slices of the first class are wider than 15).  Graphs without wide slices run kernels without their
// counting, whose registers would slow the others down (N = 30000, R = 2 13.6 us a sweep, 13.9 with it).
constexpr int kSweepPlanes = 4, kSweepWidePlanes = 6;
static_assert(SG_VB_MAX_DEGREE < (1 << kSweepWidePlanes), "the counter holds every degree");

__device__ __forceinline__ uint32_t ld_stream_u32(const uint32_t* p, uint64_t pol) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;"
                 : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint64_t ld_stream_u64(const uint64_t* p, uint64_t pol) {
    uint64_t v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u64 %0, [%1], %2;"
                 : "=l"(v) : "l"(p), "l"(pol));
    return v;
}

// spin words through L2 only: other CTAs write them within the launch
template <int R>
__device__ __forceinline__ SpinWords<R> ld_spins(const uint64_t* p, uint64_t pol) {
    SpinWords<R> s;
    if constexpr (R == 1) {
        asm volatile("ld.global.cg.L2::cache_hint.u64 %0, [%1], %2;" : "=l"(s.v[0]) : "l"(p), "l"(pol) : "memory");
    } else if constexpr (R == 2) {
        asm volatile("ld.global.cg.L2::cache_hint.v2.u64 {%0, %1}, [%2], %3;"
                     : "=l"(s.v[0]), "=l"(s.v[1]) : "l"(p), "l"(pol) : "memory");
    } else {  // a whole sector in one request (N = 2^22: 271 -> 210 us a sweep)
        asm volatile("ld.global.cg.L2::cache_hint.v4.b64 {%0, %1, %2, %3}, [%4], %5;"
                     : "=l"(s.v[0]), "=l"(s.v[1]), "=l"(s.v[2]), "=l"(s.v[3]) : "l"(p), "l"(pol) : "memory");
    }
    return s;
}

// Acceptance of one vertex: one Philox block per (vertex, sweep) serves replicas 0..3; the accepted
// m form a prefix 1..m*, so a lane flips iff its unsatisfied count u reaches ceil((d - m*) / 2).
// The first three thresholds come in one load (thr: shared or global memory); few draws pass all
// three.  Flips holds that count for each replica, at most 32, in a byte each where registers are short.
template <int R, bool kPacked>
struct Flips {
    int v[R];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = 0;
    }
    __device__ __forceinline__ void set(int r, int k) { v[r] = k; }
    __device__ __forceinline__ int from(int r) const { return v[r]; }
};
template <int R>
struct Flips<R, true> {
    uint32_t v;
    __device__ __forceinline__ void clear() { v = 0u; }
    __device__ __forceinline__ void set(int r, int k) { v = (r == 0 ? 0u : v) | (uint32_t)k << (8 * r); }
    __device__ __forceinline__ int from(int r) const { return (int)((v >> (8 * r)) & 255u); }
};

template <int R, bool kPacked>
__device__ __forceinline__ void accept_from(uint32_t vi, uint32_t t, uint64_t seed,
                                            const uint32_t* thr, Flips<R, kPacked>& flips) {
    const int deg = vi == kInactive ? 0 : (int)(vi >> kDegShift);
    const uint4 rnd = philox4x32_10(make_uint4(vi & kOrigMask, t, 0u, 0u), (uint32_t)seed,
                                    (uint32_t)(seed >> 32));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t r32 = uint4_word(rnd, r);
        const uint4 th = *reinterpret_cast<const uint4*>(thr + r * kVbThrStride);
        int ms = (int)(r32 < th.y) + (int)(r32 < th.z) + (int)(r32 < th.w);
        if (ms == 3)
            while (ms < deg && r32 < thr[r * kVbThrStride + ms + 1]) ++ms;
        ms = ms < deg ? ms : deg;
        flips.set(r, (deg - ms + 1) >> 1);
    }
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// the position of a warp in the sequence (sweep, class, slice); had: not its first slice of the class
struct Cursor {
    uint32_t sweep, cls, slice, had;
};

}  // namespace

template <int R, int kChunk, bool kWide, bool kClaims>
__global__ void __launch_bounds__(SweepShape<R, kChunk, kClaims>::threads, 2)
    k_vb_sweeps(VbPackedDev d, uint32_t t0, uint32_t n_sweeps) {
    __shared__ uint32_t cs[kVbMaxColours + 1];  // first slice of each class
    __shared__ int s_ok;
    __shared__ __align__(16) uint32_t s_thr[kSweepTables * R * kVbThrStride];
    __shared__ uint64_t s_seed[kSweepTables];
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t nc = (uint32_t)d.n_colours;
    const uint32_t gw = (tid >> 5) * gridDim.x + blockIdx.x;  // neighbouring slices on different SMs
    const uint32_t stride = (blockDim.x >> 5) * gridDim.x;
    for (uint32_t i = tid; i <= nc; i += blockDim.x) cs[i] = __ldg(d.class_slice + i);
    const bool tables = d.n_graphs <= kSweepTables;
    if (tables) {
        for (uint32_t i = tid; i < (uint32_t)(d.n_graphs * R * kVbThrStride); i += blockDim.x) s_thr[i] = __ldg(d.thr + i);
        for (uint32_t i = tid; i < (uint32_t)d.n_graphs; i += blockDim.x) s_seed[i] = __ldg(d.seeds + i);
    }
    if (tid == 0) s_ok = 1;
    __syncthreads();
    const uint32_t* thr = tables ? s_thr : d.thr;
    const uint64_t* seeds = tables ? s_seed : d.seeds;
    const uint64_t pol_keep = l2_evict_last();
    const uint64_t pol_stream = d.stream_first ? l2_evict_first() : pol_keep;

    // move to the warp's next slice, if there is one (sweep == n_sweeps: none)
    // The thin classes at the end, each at most one slice per warp of a CTA, are all the first CTA's:
    // they need no grid-wide barrier between them (two or three rounds there take longer than a
    // barrier: N = 10^5, R = 2 18.3 us a sweep against 16.4).
    const uint32_t warps = blockDim.x >> 5;
    uint32_t tail = nc;
    while (tail > 0 && cs[tail] - cs[tail - 1] <= warps) --tail;
    auto first_slice = [&](uint32_t cls) -> uint32_t {
        return cs[cls] + (cls < tail ? gw : blockIdx.x == 0 ? tid >> 5 : warps);
    };
    auto settle = [&](Cursor& c) {
        while (c.sweep < n_sweeps && c.slice >= cs[c.cls + 1]) {
            if (++c.cls == nc) {
                c.cls = 0;
                ++c.sweep;
            }
            c.slice = first_slice(c.cls);
            c.had = 0u;
        }
    };
    // Claimed slices.  Of a class of more than two slices a warp, every warp takes its first two as ever and
    // claims the others: number v of group g is slice 2 stride + v kClaimGroups + g.  The claim is asked for
    // a slice before it is needed.  Every warp of a group ends a class with one claim that fails, so a class
    // moves its counter by the same amount in every sweep.  Counters of odd and even sweeps: a warp may
    // ask for a class's next sweep before others have ended it in this one, but not two sweeps ahead.
    const uint32_t group = blockIdx.x % kClaimGroups;
    const uint32_t group_warps = warps * ((gridDim.x - group + kClaimGroups - 1u) / kClaimGroups);
    uint32_t claim = 0u;  // lane 0
    auto claims = [&](const Cursor& c) -> bool {
        return kClaims && gridDim.x >= kClaimGroups && c.sweep < n_sweeps && c.had > 0u && c.cls < tail &&
               cs[c.cls + 1] - cs[c.cls] > 2u * stride + kClaimGroups;
    };
    auto ask = [&](const Cursor& c) {
        if (claims(c) && lane == 0)
            claim = atomicAdd(d.claims + (group * 2u + (c.sweep & 1u)) * kVbMaxColours + c.cls, 1u);
    };
    auto claimed_slice = [&](const Cursor& c) -> uint32_t {
        const uint32_t size = cs[c.cls + 1] - cs[c.cls];
        const uint32_t a_sweep = (size - 2u * stride - group + kClaimGroups - 1u) / kClaimGroups + group_warps;
        const uint32_t v = __shfl_sync(0xFFFFFFFFu, claim, 0) - (c.sweep >> 1) * a_sweep;
        return v < size ? cs[c.cls] + 2u * stride + v * kClaimGroups + group : cs[c.cls + 1];
    };
    auto load_meta = [&](const Cursor& c) -> uint4 {
        return c.sweep < n_sweeps ? __ldg(d.slice_meta + c.slice) : make_uint4(0u, 0u, 0u, 0u);
    };

    // the next slice: position, {first entry, width, graph}, label and degree, own words, the
    // first chunk's neighbour slots and couplings
    Cursor nx{0u, 0u, first_slice(0), 0u};
    settle(nx);
    uint4 nm = load_meta(nx);
    Cursor nn = nx;  // the one after, of which only the meta data is read ahead
    auto step = [&](Cursor& c) {
        if constexpr (kClaims) {
            if (claims(c)) {
                c.slice = claimed_slice(c);
            } else {
                c.slice += c.cls < tail ? stride : warps;
                c.had = 1u;
            }
            settle(c);
            ask(c);
        } else {
            c.slice += c.cls < tail ? stride : warps;
            settle(c);
        }
    };
    step(nn);
    uint4 nnm = load_meta(nn);
    auto load_vi = [&](const Cursor& c) -> uint32_t {
        return c.sweep < n_sweeps ? ld_stream_u32(d.vinfo + (int64_t)c.slice * 32 + lane, pol_stream) : kInactive;
    };
    uint32_t nvi = load_vi(nx), nnvi = load_vi(nn);
    SpinWords<R> nsi;
    uint32_t col[kChunk];
    uint64_t J[kChunk];
    Flips<R, kClaims> nflips;
    nflips.clear();
#pragma unroll
    for (int e = 0; e < kChunk; ++e) {
        col[e] = 0u;
        J[e] = 0ull;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        nsi.v[r] = 0ull;
    }
    auto load_chunk = [&](uint32_t idx, uint32_t n) {
#pragma unroll
        for (int e = 0; e < kChunk; ++e) {
            J[e] = 0ull;
            if ((uint32_t)e < n) {
                col[e] = ld_stream_u32(d.col + idx + 32 * e, pol_stream);
                J[e] = ld_stream_u64(d.jb + idx + 32 * e, pol_stream);
            }
        }
    };
    auto load_slice = [&] {
        if (nx.sweep < n_sweeps) {
            const int64_t slot = (int64_t)nx.slice * 32 + lane;
            nsi = ld_spins<R>(d.S + slot * R, pol_keep);
            load_chunk(nm.x + lane, nm.y);
        }
    };
    auto next_acceptance = [&] {
        if (nx.sweep < n_sweeps)
            accept_from(nvi, t0 + nx.sweep, seeds[nm.z], thr + nm.z * (R * kVbThrStride), nflips);
    };
    load_slice();

    const uint32_t nq = n_sweeps * nc;
    uint32_t sweep = 0, cls = 0, phase = 0;  // phases: spans between grid-wide barriers
    bool ok = true;
    for (uint32_t q = 0; q < nq; ++q) {
        // beside claims there are registers to work out the next acceptance while gathers are on their way, but
        // for wide slices it waits (512 graphs of 84 M vertices 3.12 ms, for all slices early 3.38)
        auto next_early = [&] {
            if constexpr (kClaims) {
                if (nx.sweep == sweep && nx.cls == cls) next_acceptance();
            }
        };
        if (nx.sweep == sweep && nx.cls == cls) next_acceptance();
        if (phase > 0 && cls <= tail && gridDim.x > 1) {
            // admitted once every CTA has written the classes before (bounded).  Acquiring polls: the
            // words are read from L2 and the tables from shared memory, so nothing is lost with the L1,
            // and a fence after relaxed polls costs 0.3 to 0.4 us more (of 2.2 us between two classes
            // that hold one gather and one store, 152 CTAs; flags polled by every CTA 6.5, eight
            // counters 2.3).
            if (tid == 0) {
                const uint32_t target = phase * gridDim.x;
                int pass = ld_acquire_u32(d.gbar) >= target;
                if (!pass && d.stage_wait_ns) {
                    const uint64_t ns0 = global_ns();
                    for (uint32_t it = 1;; ++it) {
                        if (ld_acquire_u32(d.gbar) >= target) {
                            pass = 1;
                            break;
                        }
                        if ((it & 255u) == 0u && global_ns() - ns0 > d.stage_wait_ns) break;
                    }
                }
                if (!pass) {
                    atomicOr(d.err, 8);
                    s_ok = 0;
                }
            }
            __syncthreads();
            ok = s_ok != 0;
            if (!ok) break;  // uniform over the CTA
        }
        while (nx.sweep == sweep && nx.cls == cls) {
            const uint32_t slice = nx.slice, vi = nvi;
            SpinWords<R> si = nsi;
            const Flips<R, kClaims> flips = nflips;
            uint32_t left = nm.y, idx = nm.x + lane;
            auto advance = [&] {
                nx = nn;
                nm = nnm;
                nvi = nnvi;
                if constexpr (!kClaims) step(nn);
                load_slice();
                if constexpr (kClaims) step(nn);  // may wait for its claim
                nnm = load_meta(nn);
                nnvi = load_vi(nn);
            };
            auto count = [&](auto planes) {
                constexpr int P = decltype(planes)::value;
                uint64_t p[R][P];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int b = 0; b < P; ++b) p[r][b] = 0ull;
                for (;;) {
                    SpinWords<R> g[kChunk];
                    uint64_t Jc[kChunk];
#pragma unroll
                    for (int e = 0; e < kChunk; ++e) {
                        g[e] = si;  // an absent entry counts nothing: x = 0
                        Jc[e] = J[e];
                        if ((uint32_t)e < left) g[e] = ld_spins<R>(d.S + (int64_t)col[e] * R, pol_keep);
                    }
                    const bool last = left <= (uint32_t)kChunk;
                    if (!last) {
                        left -= kChunk;
                        idx += 32 * kChunk;
                        load_chunk(idx, left);
                    } else {
                        advance();
                        if constexpr (kClaims && P == kSweepPlanes) next_early();
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        uint64_t x[kChunk];
#pragma unroll
                        for (int e = 0; e < kChunk; ++e) x[e] = si.v[r] ^ g[e].v[r] ^ Jc[e];
                        bitslice_add4<P>(p[r], x[0], x[1], x[2], x[3]);
                        if constexpr (kChunk == 8) bitslice_add4<P>(p[r], x[4], x[5], x[6], x[7]);
                    }
                    if (last) break;
                }
#pragma unroll
                for (int r = 0; r < R; ++r) si.v[r] ^= at_least<P>(p[r], flips.from(r));
            };
            if (!kWide || left < (1u << kSweepPlanes)) count(std::integral_constant<int, kSweepPlanes>{});
            else if constexpr (kWide) {
                count(std::integral_constant<int, kSweepWidePlanes>{});
                if constexpr (kClaims) next_early();
            }
            // a warp's only slice comes next again: its words were read ahead of this update
            if (nx.slice == slice) nsi = si;
            if (vi != kInactive)
                store_words_keep<R>(d.S + ((int64_t)slice * 32 + lane) * R, si, pol_keep);
            if constexpr (!kClaims) {
                if (nx.sweep == sweep && nx.cls == cls) next_acceptance();
            }
        }
        __syncthreads();  // this CTA's words of the class are written
        if (tail <= cls && cls + 1 < nc) {  // the tail goes on
            ++cls;
            continue;
        }
        ++phase;
        if (tid == 0 && gridDim.x > 1)
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(d.gbar) : "memory");
        if (++cls == nc) {
            cls = 0;
            ++sweep;
        }
    }
    // the last CTA to leave rearms the counters for the next launch (every CTA leaves, also after
    // a wait that gave up, and none looks at the arrivals any more once it has counted itself out)
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(d.gbar + 1, 1u) == gridDim.x - 1) {
            atomicExch(d.gbar, 0u);
            atomicExch(d.gbar + 1, 0u);
            if constexpr (kClaims)
                for (uint32_t g = 0; g < 2u * kClaimGroups; ++g)
                    for (uint32_t c = 0; c < nc; ++c) d.claims[g * kVbMaxColours + c] = 0u;
        }
    }
}

template <int R, int CH>
static int sweep_warps(int sms) { return SweepShape<R, CH, false>::threads / 32 * 2 * sms; }

template <int R, int CH, bool kWide, bool kClaims>
static int launch_sweeps(const VbPackedDev& d, int max_class_slices, int sms, uint32_t t0,
                         int n_sweeps, cudaStream_t st) {
    constexpr int threads = SweepShape<R, CH, kClaims>::threads, warps = threads / 32;
    auto kern = k_vb_sweeps<R, CH, kWide, kClaims>;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0) != cudaSuccess ||
        per_sm < 1)
        return -1;
    if (per_sm > 2) per_sm = 2;
    // as many CTAs as the largest class fills; below one per SM four slices each (a barrier of few
    // CTAs is no dearer, and their warps share the schedulers less)
    int64_t grid = ((int64_t)max_class_slices + warps - 1) / warps;
    if (grid < sms) grid = std::min<int64_t>(sms, ((int64_t)max_class_slices + 3) / 4);
    grid = std::min<int64_t>(grid, (int64_t)sms * per_sm);
    if (grid < 1 || max_class_slices <= warps) grid = 1;  // the first CTA does it all
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, d, t0, (uint32_t)n_sweeps) == cudaSuccess ? 1 : -1;
}

// Chunks of 8 entries where every warp has at most one slice of a class: the class then takes as long
// as its widest slice, and fewer rounds of gathers count for more than warps in flight (R = 2,
// N = 65536: 15.6 us a sweep, 16.6 with chunks of 4; R = 4, N = 60000: 23.3, 27.1).  Beyond that the
// registers are better spent on more warps (R = 2, bipartite N = 2^18: 10.3 us with chunks of 4,
// 11.9 with 8; Poissonian N = 2^22: 128, 145; R = 4, N = 10^6: 80, 90), except for one replica of a graph whose
// slices have eight entries or more on average (N = 2^20, mean degree 8 65, with chunks of 4 67; 12 86, 94;
// 16 111, 125; degree 6 45, 46).
// Slices are claimed far beyond L2.  There SMs differ by a fifth in what HBM gives them, and with the same slices
// for every warp a CTA stood still for 9 % of the time at the end of a class, on average (R = 2, N = 2^24
// 958 us a sweep, claimed 903; 12 2^20 581, 562; 512 graphs of 84 M vertices 3.41 ms, 3.12).  Nearer to L2 two
// replicas need the fifth warp of each scheduler as much (2^23 283, claimed 285; 2^22 122, 127); one replica
// has six and does not gain (2^24 466, claimed 647 with five); four replicas run three without spills either
// way, and claim everywhere (N = 2^20 53, claimed 54; 2^22 209, 199; 2^23 558, 526).  One counter for all CTAs is too
// few (2^24 1069), 32 are too many, as each serves few CTAs (942; 4 to 16 903 to 908).
template <int R, bool kWide>
static int launch_r(const VbPackedDev& d, int max_class_slices, uint32_t t0, int n_sweeps, cudaStream_t st) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return -1;
    if (max_class_slices <= sweep_warps<R, 8>(sms) || (R == 1 && d.n_rows >= 8u * (uint32_t)d.n_slices))
        return launch_sweeps<R, 8, kWide, false>(d, max_class_slices, sms, t0, n_sweeps, st);
    if constexpr (R >= 2) {
        if (R == 4 || d.far_beyond_l2) return launch_sweeps<R, 4, kWide, true>(d, max_class_slices, sms, t0, n_sweeps, st);
    }
    if constexpr (R <= 2) return launch_sweeps<R, 4, kWide, false>(d, max_class_slices, sms, t0, n_sweeps, st);
}

int vb_packed_sweeps(const VbPackedDev& d, int max_class_slices, uint32_t t0, int n_sweeps,
                     cudaStream_t st) {
    if (n_sweeps <= 0 || d.n_colours <= 0) return 0;
    const bool wide = d.max_width >= (1u << kSweepPlanes);
    switch (d.R) {
        case 1: return wide ? launch_r<1, true>(d, max_class_slices, t0, n_sweeps, st)
                            : launch_r<1, false>(d, max_class_slices, t0, n_sweeps, st);
        case 2: return wide ? launch_r<2, true>(d, max_class_slices, t0, n_sweeps, st)
                            : launch_r<2, false>(d, max_class_slices, t0, n_sweeps, st);
        case 4: return wide ? launch_r<4, true>(d, max_class_slices, t0, n_sweeps, st)
                            : launch_r<4, false>(d, max_class_slices, t0, n_sweeps, st);
        default: return -1;
    }
}

}  // namespace sg
