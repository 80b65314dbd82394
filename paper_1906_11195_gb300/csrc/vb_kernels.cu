// vb_kernels.cu -- Viana-Bray Metropolis kernels for sm_103a (the packed sweeps are in
// vb_sweep.cu and vb_resident.cu).
//
// Model (Eq. 3): H = -sum_{(ij) in E} J_ij s_i s_j, J_ij = +-1.  Flipping s_i changes the
// energy by dE = 2m with m = s_i sum_j J_ij s_j = d_i - 2u_i, u_i the number of unsatisfied
// edges at i (J_ij s_i s_j = -1).  Metropolis (Methods): flip iff m <= 0 or r32 < thr[m].
// A sweep updates one colour class (an independent set) at a time, the generalisation of the
// bipartite half-updates of SI section 3.
//
// Packed kernel (multispin coding, SI section 2): bit k of a uint64 spin word is lane k (an
// independent disorder sample); one thread updates one vertex for all 64 lanes and all R
// replicas.  Per neighbour, x = S_i ^ S_j ^ J marks the unsatisfied lanes; the x words are
// summed into a bit-sliced count (carry-save adders, four words at a time, up to width 15; a
// ripple counter of 6 planes, degree <= 63, beyond).  Because thr[m] is
// non-increasing in m and the random number is shared by the 64 lanes, the accepted set
// {m <= m*} is a prefix: with m* = #{m in 1..d : r32 < thr[m]}, a lane flips iff d - 2u <= m*,
// i.e. u >= ceil((d - m*)/2): one bit-sliced compare against a per-thread constant.
#include "../../include/sg.h"
#include "sg_internal.cuh"

namespace sg {

// ---------------------------------------------------------------------------------------------
// packed: initial spins (quench from a random configuration)
// ---------------------------------------------------------------------------------------------
__global__ void k_vb_packed_init(VbPackedDev d) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= d.n_slots) return;
    const uint32_t vi = d.vinfo[slot];
    const int R = d.R;
    if (vi == kInactive) {
        for (int r = 0; r < R; ++r) d.S[slot * R + r] = 0ull;
        return;
    }
    const uint32_t g = d.slice_graph[slot >> 5];
    const uint64_t seed = d.seeds[g];
    const uint32_t orig = vi & kOrigMask;
    for (int r = 0; r < R; ++r) {
        const uint4 w = philox4x32_10(make_uint4(orig, 0u, (uint32_t)r, 1u), (uint32_t)seed,
                                      (uint32_t)(seed >> 32));
        d.S[slot * R + r] = (uint64_t)w.x | ((uint64_t)w.y << 32);
    }
}

int vb_packed_init(const VbPackedDev& d, cudaStream_t st) {
    const int bs = 256;
    const int64_t nb = (d.n_slots + bs - 1) / bs;
    k_vb_packed_init<<<(unsigned)nb, bs, 0, st>>>(d);
    return 1;
}

// ---------------------------------------------------------------------------------------------
// upper entries: one thread per slot keeps, in order, the entries whose neighbour lies in a
// later colour class (a higher slot), and pads the rest of its upper width with itself
// ---------------------------------------------------------------------------------------------
__global__ void k_vb_build_upper(VbPackedDev d) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= d.n_slots) return;
    const int64_t s = slot >> 5;
    const uint32_t l = (uint32_t)(slot & 31);
    const uint32_t base = d.slice_base[s], width = (d.slice_base[s + 1] - base) >> 5;
    const uint32_t ub = d.up_slice_base[s], uw = (d.up_slice_base[s + 1] - ub) >> 5;
    uint32_t* up_col = const_cast<uint32_t*>(d.up_col);
    uint64_t* up_jb = const_cast<uint64_t*>(d.up_jb);
    uint32_t e2 = 0;
    for (uint32_t e = 0; e < width; ++e) {
        const uint32_t idx = base + 32 * e + l;
        const uint32_t c = d.col[idx];
        if ((int64_t)c > slot && e2 < uw) {
            up_col[ub + 32 * e2 + l] = c;
            up_jb[ub + 32 * e2 + l] = d.jb[idx];
            ++e2;
        }
    }
    for (; e2 < uw; ++e2) {
        up_col[ub + 32 * e2 + l] = (uint32_t)slot;
        up_jb[ub + 32 * e2 + l] = 0ull;
    }
    uint32_t* row_slice = const_cast<uint32_t*>(d.up_row_slice);
    for (uint32_t e = l; e < uw; e += 32) row_slice[(ub >> 5) + e] = (uint32_t)s;
}

int vb_packed_build_upper(const VbPackedDev& d, cudaStream_t st) {
    if (!d.up_slice_base || d.n_slots == 0) return 0;
    const int bs = 256;
    k_vb_build_upper<<<(unsigned)((d.n_slots + bs - 1) / bs), bs, 0, st>>>(d);
    return 1;
}

// ---------------------------------------------------------------------------------------------
// snapshot copy (16-byte vectors; the regions are 256-byte aligned and a multiple of 16 bytes)
// ---------------------------------------------------------------------------------------------
__global__ void k_copy16(const uint4* __restrict__ src, uint4* __restrict__ dst, int64_t n16) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}

static int copy_bytes(const void* src, void* dst, int64_t bytes, cudaStream_t st) {
    const int64_t n16 = bytes / 16;
    const int bs = 256;
    int64_t nb = (n16 + bs - 1) / bs;
    if (nb > 152 * 16) nb = 152 * 16;
    if (nb < 1) nb = 1;
    k_copy16<<<(unsigned)nb, bs, 0, st>>>((const uint4*)src, (uint4*)dst, n16);
    return 1;
}

int vb_packed_snapshot(const VbPackedDev& d, int w, cudaStream_t st) {
    const int64_t words = d.n_slots * d.R;
    return copy_bytes(d.S, d.snap + (int64_t)w * words, words * 8, st);
}

// ---------------------------------------------------------------------------------------------
// The configuration in the caller's order: word (graph, replica, vertex) of the flat output, of
// which [lo, hi) goes to out.  One thread per slot: the words are read in slot order and scattered by
// label (within a class and degree the labels ascend), all of it in L2: the copy to the host is what
// takes the time (13.7 MB in about 90 us to memory that was touched before, 0.7 ms to fresh pages).
// Before, the words went to a host buffer and the host permuted them: N = 300007, one replica,
// a measurement and the configuration took 290 us and now take 90.
// ---------------------------------------------------------------------------------------------
__global__ void k_vb_packed_spins(VbPackedDev d, const int64_t* __restrict__ graph_words, int64_t lo,
                                  int64_t hi, uint64_t* __restrict__ out) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= d.n_slots) return;
    const uint32_t vi = d.vinfo[slot];
    if (vi == kInactive) return;
    const uint32_t g = d.slice_graph[slot >> 5];
    const int64_t first = graph_words[g], n = (graph_words[g + 1] - first) / d.R;
    int64_t o = first + (vi & kOrigMask);
    for (int r = 0; r < d.R; ++r, o += n)
        if (o >= lo && o < hi) out[o - lo] = d.S[slot * d.R + r];
}

int vb_packed_spins(const VbPackedDev& d, const int64_t* graph_words, int64_t lo, int64_t hi,
                    uint64_t* out, cudaStream_t st) {
    k_vb_packed_spins<<<(unsigned)((d.n_slots + 255) / 256), 256, 0, st>>>(d, graph_words, lo, hi, out);
    return 1;
}

// ---------------------------------------------------------------------------------------------
// plain kernel: one thread per (vertex, lane, replica), int8 spins, CSR in colour-major labels
// ---------------------------------------------------------------------------------------------
__global__ void k_vb_plain_init(VbPlainDev d) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)d.N * d.R) return;
    const int32_t v = (int32_t)(idx % d.N);
    const int32_t r = (int32_t)(idx / d.N);
    const uint4 w = philox4x32_10(make_uint4(d.orig[v], 0u, (uint32_t)r, 1u), (uint32_t)d.seed,
                                  (uint32_t)(d.seed >> 32));
    const uint64_t bits = (uint64_t)w.x | ((uint64_t)w.y << 32);
    for (int k = 0; k < d.L; ++k)
        d.s[((int64_t)r * d.L + k) * d.N + v] = ((bits >> k) & 1ull) ? (int8_t)-1 : (int8_t)1;
}

int vb_plain_init(const VbPlainDev& d, cudaStream_t st) {
    const int bs = 256;
    const int64_t n = (int64_t)d.N * d.R;
    k_vb_plain_init<<<(unsigned)((n + bs - 1) / bs), bs, 0, st>>>(d);
    return 1;
}

__global__ void k_vb_plain_colour(VbPlainDev d, int32_t v0, int32_t nv, const uint32_t* clock,
                                  uint32_t t_off) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)nv * d.R * d.L) return;
    const uint32_t t = *clock + t_off;
    const int32_t v = v0 + (int32_t)(idx % nv);
    const int32_t rk = (int32_t)(idx / nv);
    const int32_t r = rk / d.L, k = rk % d.L;
    const uint4 rnd = philox4x32_10(make_uint4(d.orig[v], t, (uint32_t)(r >> 2), 0u),
                                    (uint32_t)d.seed, (uint32_t)(d.seed >> 32));
    const uint32_t r32 = uint4_word(rnd, r & 3);
    int8_t* s = d.s + (int64_t)rk * d.N;
    int field = 0;
    for (int32_t e = d.row_ptr[v]; e < d.row_ptr[v + 1]; ++e) {
        const int J = ((d.jb[e] >> k) & 1ull) ? -1 : 1;
        field += J * s[d.col[e]];
    }
    const int m = s[v] * field;
    const bool flip = (m <= 0) || (r32 < d.thr[r * kVbThrStride + m]);
    if (flip) s[v] = (int8_t)(-s[v]);
}

int vb_plain_colour(const VbPlainDev& d, int32_t v_begin, int32_t v_end, const uint32_t* clock,
                    uint32_t t_off, cudaStream_t st) {
    const int32_t nv = v_end - v_begin;
    if (nv <= 0) return 0;
    const int bs = 256;
    const int64_t n = (int64_t)nv * d.R * d.L;
    k_vb_plain_colour<<<(unsigned)((n + bs - 1) / bs), bs, 0, st>>>(d, v_begin, nv, clock, t_off);
    return 1;
}

int vb_plain_snapshot(const VbPlainDev& d, int w, cudaStream_t st) {
    const int64_t bytes = (int64_t)d.R * d.L * d.N;
    // int8 snapshots are not 16-byte multiples in general: use a byte copy
    return cudaMemcpyAsync(d.snap + (int64_t)w * bytes, d.s, (size_t)bytes,
                           cudaMemcpyDeviceToDevice, st) == cudaSuccess ? 0 : -1;
}

// per-(replica or pair, lane) difference counts over the vertices; blockIdx.y = rq * L + k
__global__ void k_vb_plain_count(VbPlainDev d, VbCountJob job) {
    const int32_t rk = blockIdx.y;
    const int32_t rq = rk / d.L, k = rk % d.L;
    const int64_t plane = (int64_t)d.R * d.L * d.N;
    unsigned long long acc = 0;
    for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < d.N; v += gridDim.x * blockDim.x) {
        if (job.kind == 0) {
            const int64_t o = ((int64_t)rq * d.L + k) * d.N + v;
            acc += d.s[o] != d.snap[(int64_t)job.w * plane + o];
        } else if (job.kind == 1) {
            const int64_t a = ((int64_t)(2 * rq) * d.L + k) * d.N + v;
            const int64_t b = ((int64_t)(2 * rq + 1) * d.L + k) * d.N + v;
            acc += d.s[a] != d.s[b];
        } else {
            const int8_t* s = d.s + ((int64_t)rq * d.L + k) * d.N;
            for (int32_t e = d.row_ptr[v]; e < d.row_ptr[v + 1]; ++e) {
                const int J = ((d.jb[e] >> k) & 1ull) ? -1 : 1;
                acc += (J * s[v] * s[d.col[e]]) < 0;
            }
        }
    }
    // block reduction
    __shared__ unsigned long long red[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0ull;
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
        if (threadIdx.x == 0 && acc)
            atomicAdd((unsigned long long*)(job.dst + rq * job.stride_r + k * job.stride_k), acc);
    }
}

int vb_plain_count(const VbPlainDev& d, const VbCountJob& job, cudaStream_t st) {
    const int nq = job.kind == 1 ? d.R / 2 : d.R;
    if (nq <= 0) return 0;
    const int bs = 256;
    int nb = (d.N + bs - 1) / bs;
    if (nb > 64) nb = 64;
    dim3 grid((unsigned)nb, (unsigned)(nq * d.L));
    k_vb_plain_count<<<grid, bs, 0, st>>>(d, job);
    return 1;
}

}  // namespace sg
