// vb_measure.cu -- the packed Viana-Bray measurement for sm_103a: one launch counts, per lane,
// the spins that differ from every snapshot taken (the correlation after Eq. 1), the spins that
// differ between the replicas of a pair (the overlap of SI section 1) and the unsatisfied edges
// (the energy of Eq. 3).
//
// A job is a pass over rows of 32 spin words, one word per thread of a warp: C against snapshot w
// and q pass over the slices, E over the rows of the upper entries (each edge once; a row's own
// slice is up_row_slice, so a warp's rows need no per-slice loop and several rows' loads are in
// flight at once).  A warp takes a run of consecutive rows of one pass, adds the words with
// carry-save adders into bit-sliced counters, four rows at a time, and sums the counters of its
// 32 threads at the end of the run; the CTA adds its warps' totals into the results once.
//
// What bounds it: on large graphs the bytes (spins and snapshots once per pass, 12 bytes per edge
// and a 32-byte sector per gathered word), on small ones the latency of one run.  The run length
// therefore follows the size: as many warps as the GPU holds, up to kMeasureRun rows each (the
// sum over the 32 threads costs about as much as 30 rows' additions).
#include <algorithm>

#include "../../include/sg.h"
#include "sg_internal.cuh"
#include "vb_bits.cuh"

namespace sg {

constexpr int kMeasureRun = 63;     // rows of one run: the counters hold 6 planes
constexpr int kMeasurePlanes = 6;
constexpr int kMeasureWarps = 8;
static_assert(kMeasureRun < (1 << kMeasurePlanes), "a run fits the counters");

struct MeasureGrid {
    int run_s, run_e;   // rows of a run over slices, over upper rows
    uint32_t nb_s, nb_e;  // CTAs of one pass over the slices; of the energy pass
    uint32_t up_rows;
};

// Sum the counters of the warp's 32 threads.  The first exchange leaves each half warp with one
// 32-bit half of the words, the others add within the half warp, one more plane each; thread l
// then holds the totals of lanes 32 (l / 16) + l % 16 (c0) and 16 above it (c1).
template <int P>
__device__ __forceinline__ void warp_totals(const uint64_t (&p)[P], uint32_t lane, uint32_t& c0,
                                            uint32_t& c1) {
    uint32_t t[P + 5];
    const bool upper = (lane & 16u) != 0u;
    uint32_t carry = 0u;
#pragma unroll
    for (int b = 0; b < P; ++b) {
        const uint32_t lo = (uint32_t)p[b], hi = (uint32_t)(p[b] >> 32);
        const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, upper ? lo : hi, 16);
        const uint32_t k = upper ? hi : lo;
        t[b] = k ^ o ^ carry;
        carry = (k & o) | (carry & (k ^ o));
    }
    t[P] = carry;
#pragma unroll
    for (int step = 0; step < 4; ++step) {
        const int n = P + 1 + step;  // planes before this exchange
        carry = 0u;
#pragma unroll
        for (int b = 0; b < n; ++b) {
            const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, t[b], 8 >> step);
            const uint32_t k = t[b];
            t[b] = k ^ o ^ carry;
            carry = (k & o) | (carry & (k ^ o));
        }
        t[n] = carry;
    }
    const uint32_t sh = lane & 15u;
    c0 = c1 = 0u;
#pragma unroll
    for (int b = 0; b < P + 5; ++b) {
        c0 |= ((t[b] >> sh) & 1u) << b;
        c1 |= ((t[b] >> (sh + 16u)) & 1u) << b;
    }
}

template <int R>
__device__ __forceinline__ SpinWords<R> words_nc(const uint64_t* p) {
    SpinWords<R> s;
    if constexpr (R == 1) {
        s.v[0] = __ldg(p);
    } else {
#pragma unroll
        for (int h = 0; h < R / 2; ++h) {
            const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(p) + h);
            s.v[2 * h] = a.x;
            s.v[2 * h + 1] = a.y;
        }
    }
    return s;
}

// Count rows [a, b) of one graph into the counters (b - a <= kMeasureRun).  KIND 0: C against
// snap; 1: q; 2: E over upper rows.
template <int R, int KIND>
__device__ __forceinline__ void count_rows(const VbPackedDev& d, const uint64_t* __restrict__ snap,
                                           int64_t a, int64_t b, uint32_t lane,
                                           uint64_t (&p)[R][kMeasurePlanes]) {
    constexpr int NQ = KIND == 1 ? (R / 2 > 0 ? R / 2 : 1) : R;
    auto row = [&](int64_t s, bool in, uint64_t (&x)[NQ]) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) x[q] = 0ull;
        if (!in) return;  // warp-uniform
        if constexpr (KIND == 2) {
            const int64_t e = s * 32 + lane;
            const uint32_t j = __ldg(d.up_col + e);
            const uint64_t J = __ldg(d.up_jb + e);
            const SpinWords<R> si = words_nc<R>(d.S + ((int64_t)__ldg(d.up_row_slice + s) * 32 + lane) * R);
            const SpinWords<R> sj = gather_words<R>(d.S + (int64_t)j * R);
#pragma unroll
            for (int r = 0; r < R; ++r) x[r] = si.v[r] ^ sj.v[r] ^ J;
        } else {
            const SpinWords<R> si = words_nc<R>(d.S + (s * 32 + lane) * R);
            if constexpr (KIND == 0) {
                const SpinWords<R> sw = words_nc<R>(snap + (s * 32 + lane) * R);
#pragma unroll
                for (int r = 0; r < R; ++r) x[r] = si.v[r] ^ sw.v[r];
            } else if constexpr (R >= 2) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) x[q] = si.v[2 * q] ^ si.v[2 * q + 1];
            }
        }
    };
    for (int64_t s = a; s < b; s += 4) {
        uint64_t x[4][NQ];
#pragma unroll
        for (int u = 0; u < 4; ++u) row(s + u, s + u < b, x[u]);
#pragma unroll
        for (int q = 0; q < NQ; ++q) bitslice_add4(p[q], x[0][q], x[1][q], x[2][q], x[3][q]);
    }
}

// CTAs that share an SM (64 registers a thread for one and two replicas, 128 for four)
template <int R>
constexpr int kMeasureCtas = R == 4 ? 2 : 4;

template <int R>
__global__ void __launch_bounds__(32 * kMeasureWarps, kMeasureCtas<R>)
    k_vb_packed_measure(VbPackedDev d, VbMeasure m, MeasureGrid mg) {
    __shared__ unsigned long long acc[R * 64];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    // the energy pass first (its dependent gathers take longest), then C of each snapshot, then q
    const bool en = blockIdx.x < mg.nb_e;
    const uint32_t pb = en ? 0u : blockIdx.x - mg.nb_e;
    const int pass = en ? 0 : (int)(pb / mg.nb_s);
    const int kind = en ? 2 : (pass < m.n_c ? 0 : 1);
    const int64_t blk = en ? blockIdx.x : pb - (uint32_t)pass * mg.nb_s;
    const int run = en ? mg.run_e : mg.run_s;
    const int64_t rows = en ? (int64_t)mg.up_rows : (int64_t)d.n_slices;
    const int nq = kind == 1 ? R / 2 : R;
    const int64_t cta_lo = blk * kMeasureWarps * run;
    int64_t cta_hi = cta_lo + (int64_t)kMeasureWarps * run;
    if (cta_hi > rows) cta_hi = rows;
    const int64_t lo = cta_lo + (int64_t)warp * run;
    const int64_t hi = lo + run < cta_hi ? lo + run : cta_hi;
    int64_t* dst = kind == 0 ? m.c + pass * m.c_w : kind == 1 ? m.q : m.e;
    const int64_t st_g = kind == 0 ? m.c_g : kind == 1 ? m.q_g : m.e_g;
    const int64_t st_r = kind == 0 ? m.c_r : kind == 1 ? m.q_r : m.e_r;
    const int64_t st_k = kind == 0 ? m.c_k : kind == 1 ? m.q_k : m.e_k;
    const int shift = en ? 1 : 0;  // the energy's counts are of directed entries: twice each edge
    const uint64_t* snap = d.snap + (int64_t)(kind == 0 ? pass : 0) * d.n_slots * R;
    auto graph_of = [&](int64_t row) -> uint32_t {
        return __ldg(d.slice_graph + (en ? (int64_t)__ldg(d.up_row_slice + row) : row));
    };
    // Rows are in slot order, by class and then graph, so a CTA of a batch may span graphs and come
    // back to its first one in the next class: every row is looked at.  With one graph the warps
    // add into the CTA's totals; otherwise each adds its totals of each graph into the results.
    const uint32_t g_first = graph_of(cta_lo);
    bool same = true;
    if (d.n_graphs > 1)
        for (int64_t r = cta_lo + tid; r < cta_hi; r += 32 * kMeasureWarps) same = same && graph_of(r) == g_first;
    for (uint32_t i = tid; i < (uint32_t)R * 64u; i += 32 * kMeasureWarps) acc[i] = 0ull;
    const bool one_graph = __syncthreads_and(same) != 0;
    int64_t a = lo;
    while (a < hi) {
        uint32_t g = g_first;
        int64_t b = hi;
        if (!one_graph) {  // the rows of the run's next graph
            g = graph_of(a);
            b = a + 1;
            while (b < hi && graph_of(b) == g) ++b;
        }
        uint64_t p[R][kMeasurePlanes];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int k = 0; k < kMeasurePlanes; ++k) p[r][k] = 0ull;
        if (kind == 2) count_rows<R, 2>(d, snap, a, b, lane, p);
        else if (kind == 0) count_rows<R, 0>(d, snap, a, b, lane, p);
        else count_rows<R, 1>(d, snap, a, b, lane, p);
        const uint32_t k0 = 32u * (lane >> 4) + (lane & 15u);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r >= nq) break;
            uint32_t c0, c1;
            warp_totals<kMeasurePlanes>(p[r], lane, c0, c1);
            if (one_graph) {
                if (c0) atomicAdd(&acc[r * 64 + k0], (unsigned long long)c0);
                if (c1) atomicAdd(&acc[r * 64 + k0 + 16], (unsigned long long)c1);
            } else {
                int64_t* base = dst + g * st_g + r * st_r;
                if (c0)
                    atomicAdd((unsigned long long*)(base + k0 * st_k), (unsigned long long)c0 << shift);
                if (c1)
                    atomicAdd((unsigned long long*)(base + (k0 + 16) * st_k),
                              (unsigned long long)c1 << shift);
            }
        }
        a = b;
    }
    if (!one_graph) return;  // CTA-uniform
    __syncthreads();
    for (uint32_t i = tid; i < (uint32_t)nq * 64u; i += 32 * kMeasureWarps) {
        const unsigned long long v = acc[i];
        if (v)
            atomicAdd((unsigned long long*)(dst + g_first * st_g + (int64_t)(i >> 6) * st_r +
                                            (int64_t)(i & 63u) * st_k),
                      v << shift);
    }
}

int vb_packed_measure(const VbPackedDev& d, const VbMeasure& m, cudaStream_t st) {
    const int passes = m.n_c + (m.q && d.R >= 2 ? 1 : 0);
    const int64_t rows = (int64_t)d.n_slices * passes + (m.e ? (int64_t)d.up_rows : 0);
    if (rows == 0) return 0;
    MeasureGrid mg;
    mg.up_rows = d.up_rows;
    // Whole waves of the CTAs that the SMs hold at once.  In one or two waves the slowest run is the
    // time: a row of edges takes longer than a row of spins (its gathers wait for its slots), so its
    // runs are half as long (five snapshots, N = 2^20: 72 -> 60 us; a third as long 61, a quarter 65).
    // More waves even out by themselves (N = 2^22: 180 us, with shorter edge runs 185).
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return -1;
    const int64_t slots = (int64_t)sms * (d.R == 4 ? kMeasureCtas<4> : kMeasureCtas<2>);
    auto waves_of = [&](int64_t c) { return (c + slots * kMeasureWarps * kMeasureRun - 1) / (slots * kMeasureWarps * kMeasureRun); };
    const int64_t edge_cost = waves_of(rows) <= 2 ? 2 : 1;
    const int64_t cost = (int64_t)d.n_slices * passes + (m.e ? (int64_t)d.up_rows * edge_cost : 0);
    const int64_t waves = waves_of(cost);
    int64_t run = (cost + waves * slots * kMeasureWarps - 1) / (waves * slots * kMeasureWarps);
    auto edge_run = [&](int64_t r) { return std::max<int64_t>(1, r / edge_cost); };
    auto ctas = [&](int64_t r) {  // each pass's last CTA is part empty
        const int64_t n = r * kMeasureWarps, ne = edge_run(r) * kMeasureWarps;
        return (d.n_slices + n - 1) / n * passes + (m.e ? ((int64_t)d.up_rows + ne - 1) / ne : 0);
    };
    while (run < kMeasureRun && ctas(run) > waves * slots) ++run;
    mg.run_s = (int)run;
    mg.run_e = (int)edge_run(run);
    const int64_t per_cta = run * kMeasureWarps, per_cta_e = mg.run_e * kMeasureWarps;
    mg.nb_s = passes ? (uint32_t)((d.n_slices + per_cta - 1) / per_cta) : 1u;
    mg.nb_e = m.e ? (uint32_t)(((int64_t)d.up_rows + per_cta_e - 1) / per_cta_e) : 0u;
    const int64_t nb = (int64_t)mg.nb_e + (int64_t)mg.nb_s * passes;
    if (nb > 0x7FFFFFFF) return -1;
    switch (d.R) {
        case 1: k_vb_packed_measure<1><<<(unsigned)nb, 32 * kMeasureWarps, 0, st>>>(d, m, mg); break;
        case 2: k_vb_packed_measure<2><<<(unsigned)nb, 32 * kMeasureWarps, 0, st>>>(d, m, mg); break;
        case 4: k_vb_packed_measure<4><<<(unsigned)nb, 32 * kMeasureWarps, 0, st>>>(d, m, mg); break;
        default: return -1;
    }
    return 1;
}

}  // namespace sg
