// sg_noalloc.cu -- SK local fields h = J s without any device allocation.
//
// Some callers cannot allocate device memory at the point where they need this computation: a
// host application that hands the library a fixed memory budget and forbids further
// allocations, or a plugin whose process owns every device allocation.  sg_sk_fields_noalloc
// serves them: the caller passes its own input and output buffers, and one launch takes the int8
// operands to the fields through shared and tensor memory only.  The call waits for its own work (it
// synchronises the caller's stream before returning).
#include <cuda.h>

#include <condition_variable>
#include <mutex>
#include <string>

#include "../../include/sg.h"
#include "sg_internal.cuh"
#include "sg_model.h"
#include "sk_internal.cuh"

namespace sg {
namespace {

constexpr int kNoallocMaxN = 2048;      // spins (padded to a multiple of 128)
constexpr int kNoallocMaxR = 128;       // replicas
constexpr int kFieldsThreads = 256;
constexpr int kFieldsMaxSplit = 8;      // CTAs of a cluster, each with its own share of the columns
constexpr uint32_t kFieldsPolls = 1u << 24;

// Where h overlaps J or s (each CTA writes fields while others still read): the fields go here first.
static __device__ __align__(256) int32_t g_noalloc_h[(size_t)kNoallocMaxR * kNoallocMaxN];

// signs of 4 int8 as e4m3: +-1.0 (0x38, 0xB8) or 0
__device__ __forceinline__ uint32_t e4m3_signs(uint32_t v) {
    const uint32_t neg = v & 0x80808080u;
    const uint32_t nz = ((((v & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | v) & 0x80808080u) >> 7;
    return nz * 0x38u | neg;
}

// 16 bytes of a row from p, of which m are the row's (the rest becomes zero).  Words holds what is loaded
// ahead: with A16 the piece itself (p 16-byte aligned, m = 16), else the five 4-byte words around it,
// where all of them lie inside the array [a, end); otherwise finish() reads the bytes one by one.
template <bool A16>
struct Piece {
    uint32_t x[A16 ? 4 : 5];
    const int8_t* p;
    int m;
    __device__ __forceinline__ bool words(const int8_t* a, const int8_t* end) const {
        const int8_t* q = p - ((uintptr_t)p & 3u);
        return q >= a && q + 20 <= end;
    }
    __device__ __forceinline__ void load(const int8_t* a, const int8_t* end) {
        if constexpr (A16) {
            const uint4 v = m > 0 ? __ldg(reinterpret_cast<const uint4*>(p)) : make_uint4(0u, 0u, 0u, 0u);
            x[0] = v.x;
            x[1] = v.y;
            x[2] = v.z;
            x[3] = v.w;
        } else {
            const bool in = m > 0 && words(a, end);
            const uint32_t* q = reinterpret_cast<const uint32_t*>(p - ((uintptr_t)p & 3u));
#pragma unroll
            for (int k = 0; k < 5; ++k) x[k] = in ? __ldg(q + k) : 0u;
        }
    }
    __device__ __forceinline__ uint4 finish(const int8_t* a, const int8_t* end) const {
        if constexpr (A16) return make_uint4(x[0], x[1], x[2], x[3]);
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (m > 0 && !words(a, end)) {
            for (int k = 0; k < m; ++k) w[k >> 2] |= (uint32_t)(uint8_t)__ldg(p + k) << (8 * (k & 3));
        } else if (m > 0) {
            const uint32_t sh = ((uintptr_t)p & 3u) * 8u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                w[k] = __funnelshift_r(x[k], x[k + 1 < 5 ? k + 1 : 4], sh);
                const int left = m - 4 * k;
                if (left < 4) w[k] = left <= 0 ? 0u : w[k] & ((1u << (8 * left)) - 1u);
            }
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// The CTA's operands into shared memory: 16-byte pieces of kt tiles of 128 columns from k0 of the
// coupling rows m0 .. m0 + 127 and of the R spin rows; piece c of row r goes to c ^ (r & 7) of that row.
// Several pieces of a thread are on their way at once.
template <bool A16>
__device__ __forceinline__ void load_operands(const int8_t* __restrict__ J, const int8_t* __restrict__ s,
                                              int n, int R, int kt, int m0, int k0, uint8_t* sA,
                                              uint8_t* sB, int tid) {
    constexpr int U = A16 ? 8 : 4;
    const int pieces = kt * 8, lp = kt == 2 ? 4 : 3;  // kt is 1 or 2
    const int total = (128 + R) * pieces;
    const int8_t *end_j = J + (int64_t)n * n, *end_s = s + (int64_t)R * n;
    for (int i0 = tid; i0 < total; i0 += kFieldsThreads * U) {
        Piece<A16> pc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * kFieldsThreads, row = i >> lp, o = k0 + (i & (pieces - 1)) * 16;
            const bool j = row < 128;
            const int left = n - o;
            pc[u].m = i < total && (!j || m0 + row < n) ? (left < 16 ? left : 16) : 0;
            pc[u].p = j ? J + (int64_t)(m0 + row) * n + o : s + (int64_t)(row - 128) * n + o;
            pc[u].load(j ? J : s, j ? end_j : end_s);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * kFieldsThreads, row = i >> lp, c = i & (pieces - 1);
            if (i >= total) break;
            const bool j = row < 128;
            const int r = j ? row : row - 128;
            uint4 v = pc[u].finish(j ? J : s, j ? end_j : end_s);
            v.x = e4m3_signs(v.x);
            v.y = e4m3_signs(v.y);
            v.z = e4m3_signs(v.z);
            v.w = e4m3_signs(v.w);
            uint8_t* tile = j ? sA + (size_t)(c >> 3) * 128 * 128 : sB + (size_t)(c >> 3) * R * 128;
            *reinterpret_cast<uint4*>(tile + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = v;
        }
    }
}

__device__ __forceinline__ uint32_t fields_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

size_t fields_smem(int kt, int R) { return 1024 + (size_t)kt * (128 + R) * 128 + (size_t)R * 128 * 4; }

}  // namespace

// h[r][i] = sum_j J[i][j] s[r][j]: a cluster per 128 rows, its CTAs sharing the columns (kt tiles of 128
// each).  A CTA turns its int8 operands into e4m3 in shared memory (the 128-byte swizzle the tensor
// cores read), multiplies (kind::f8f6f4, FP32 accumulators: exact, |h| <= 2048) and leaves its part
// in shared memory; the CTAs of the cluster then add the parts up, each for its own replicas.
// At n = 2000 with 128 replicas the work is 4 MB of couplings and a launch: what bounds it is latency,
// so all 128 CTAs load at once and nothing goes through memory twice: 32 to 36 us for the whole call,
// against 154 for a staging launch, 16 dependent GEMM launches of 128 columns and a copy.
__global__ void __launch_bounds__(kFieldsThreads)
    k_noalloc_fields(const int8_t* __restrict__ J, const int8_t* __restrict__ s, int n, int R, int kt,
                     int split, int32_t* __restrict__ h, volatile int* status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    uint8_t* sA = smem;                                   // kt x [128 rows][128 columns]
    uint8_t* sB = smem + (size_t)kt * 128 * 128;          // kt x [R][128]
    int32_t* part = reinterpret_cast<int32_t*>(sB + (size_t)kt * R * 128);  // [R][128 rows]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)fields_rank();
    const int m0 = ((int)blockIdx.x / split) * 128, k0 = rank * kt * 128;
    const uint32_t ncols = R <= 32 ? 32u : R <= 64 ? 64u : 128u;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&tslot)), "r"(ncols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if ((((uintptr_t)J | (uintptr_t)s | (uintptr_t)n) & 15u) == 0)
        load_operands<true>(J, s, n, R, kt, m0, k0, sA, sB, tid);
    else
        load_operands<false>(J, s, n, R, kt, m0, k0, sA, sB, tid);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tslot;
    if (tid == 0) {
        const uint32_t idesc = (1u << 4) | ((uint32_t)(R >> 3) << 17) | ((128u >> 4) << 24);
        for (int t = 0; t < kt; ++t)
            for (int ks = 0; ks < 4; ++ks) {
                const uint64_t ad = smem_desc(smem_addr(sA + (size_t)t * 128 * 128) + ks * 32, 128);
                const uint64_t bd = smem_desc(smem_addr(sB + (size_t)t * R * 128) + ks * 32, 128);
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "setp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"((uint32_t)(t | ks))
                    : "memory");
            }
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(&bar))
            : "memory");
    }
    bool ok = mbar_wait(&bar, 0, kFieldsPolls);
    if (!ok) {
        *status = 1;
        mbar_wait(&bar, 0, kFieldsPolls);  // the products end before their tensor memory is freed
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp < 4 && ok) {
        for (int c = 0; c < R; c += 16) {
            uint32_t v[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                  "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
                  "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                : "r"(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) part[(c + j) * 128 + 32 * warp + lane] = __float2int_rn(__uint_as_float(v[j]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    cluster_sync_all();  // every part of the cluster is written; orders this CTA's threads too
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols)
                     : "memory");
    // replicas rank, rank + split, ... of this CTA, one per warp: four rows per thread
    for (int r = rank + split * warp; r < R; r += split * (kFieldsThreads / 32)) {
        const uint32_t a = smem_addr(part + r * 128 + 4 * lane);
        int4 v[kFieldsMaxSplit];
#pragma unroll
        for (int k = 0; k < kFieldsMaxSplit; ++k) {
            v[k] = make_int4(0, 0, 0, 0);
            if (k < split) {
                uint32_t ra;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(k));
                asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(v[k].x), "=r"(v[k].y), "=r"(v[k].z), "=r"(v[k].w) : "r"(ra));
            }
        }
        int sum[4] = {0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < kFieldsMaxSplit; ++k) {
            sum[0] += v[k].x;
            sum[1] += v[k].y;
            sum[2] += v[k].z;
            sum[3] += v[k].w;
        }
        int32_t* out = h + (int64_t)r * n + m0 + 4 * lane;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (m0 + 4 * lane + j < n) out[j] = sum[j];
    }
    cluster_sync_all();  // no CTA leaves while another may read its part
}

namespace {

// Status words in page-locked host memory that the kernel writes directly (only when a wait expires), so that
// a call reads its own after the synchronisation without a copy.  One word per call in flight; a
// call waits while all are taken.
constexpr int kStatusWords = 256;
std::mutex g_status_mutex;
std::condition_variable g_status_free;
int* g_status = nullptr;      // kept until the process exits
int* g_status_dev = nullptr;  // the same words to the GPUs (one address space)
bool g_status_used[kStatusWords] = {};

class StatusWord {
public:
    StatusWord() {
        std::unique_lock<std::mutex> lock(g_status_mutex);
        if (!g_status) {
            void* p = nullptr;
            check_cuda(cudaHostAlloc(&p, kStatusWords * sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped),
                       "cudaHostAlloc");
            void* q = nullptr;
            check_cuda(cudaHostGetDevicePointer(&q, p, 0), "cudaHostGetDevicePointer");
            g_status_dev = static_cast<int*>(q);
            g_status = static_cast<int*>(p);
        }
        for (;;) {
            for (k_ = 0; k_ < kStatusWords && g_status_used[k_]; ++k_) {}
            if (k_ < kStatusWords) break;
            g_status_free.wait(lock);
        }
        g_status_used[k_] = true;
        *word() = 0;
    }
    ~StatusWord() {
        {
            std::lock_guard<std::mutex> lock(g_status_mutex);
            g_status_used[k_] = false;
        }
        g_status_free.notify_one();
    }
    volatile int* word() const { return g_status + k_; }
    int* device() const { return g_status_dev + k_; }

private:
    int k_ = 0;
};

// The device that owns p: its ordinal for device memory, -2 for managed memory (usable from
// any device), -1 for anything else (host memory, or no CUDA device at all).  A buffer on
// another GPU would be dereferenced as a peer address, which faults when peer access is not
// enabled, so the caller compares the ordinal with the current device.
int pointer_device(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    if (a.type == cudaMemoryTypeManaged) return -2;
    return a.type == cudaMemoryTypeDevice ? a.device : -1;
}

// the kernel's shared memory limit, raised once on each device
void prepare_kernel(int dev) {
    static std::mutex m;
    static bool done[64] = {};
    std::lock_guard<std::mutex> lock(m);
    if (dev >= 0 && dev < 64 && done[dev]) return;
    check_cuda(cudaFuncSetAttribute(k_noalloc_fields, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)fields_smem(2, kNoallocMaxR)),
               "cudaFuncSetAttribute");
    if (dev >= 0 && dev < 64) done[dev] = true;
}

bool overlap(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + nb && y < x + na;
}

}  // namespace
}  // namespace sg

extern "C" int sg_sk_fields_noalloc(const int8_t* J, const int8_t* s, int32_t n, int32_t n_replicas,
                                    int32_t* h, void* cuda_stream) {
    using namespace sg;
    try {
        if (!J || !s || !h) fail(SG_EINVAL, "null pointer");
        if (n < 2 || n > kNoallocMaxN)
            fail(SG_EINVAL, "n must be in [2, " + std::to_string(kNoallocMaxN) + "]");
        if (n_replicas < 16 || n_replicas > kNoallocMaxR || n_replicas % 16)
            fail(SG_EINVAL, "n_replicas must be a multiple of 16 in [16, " +
                                std::to_string(kNoallocMaxR) + "]");
        const int owner[3] = {pointer_device(J), pointer_device(s), pointer_device(h)};
        for (int o : owner)
            if (o == -1) fail(SG_EINVAL, "J, s and h must be device memory");
        int dev = 0;
        check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
        for (int o : owner)
            if (o >= 0 && o != dev) fail(SG_EINVAL, "J, s and h must be memory of the current device");
        cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
        const int R = n_replicas;
        const int tiles = (n + 127) / 128;
        // up to 8 CTAs share the columns of a row tile: the largest instance then has 128 CTAs
        int split = 1;
        while (split < kFieldsMaxSplit && split < tiles) split *= 2;
        const int kt = (tiles + split - 1) / split;
        const size_t bytes_h = (size_t)R * n * 4;
        const bool via = overlap(h, bytes_h, J, (size_t)n * n) || overlap(h, bytes_h, s, (size_t)R * n);
        int32_t* out = h;
        if (via) {
            void* p = nullptr;
            check_cuda(cudaGetSymbolAddress(&p, g_noalloc_h), "cudaGetSymbolAddress");
            out = static_cast<int32_t*>(p);
        }
        StatusWord status;
        const size_t smem = fields_smem(kt, R);
        prepare_kernel(dev);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(tiles * split));
        cfg.blockDim = dim3(kFieldsThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)split;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        check_cuda(cudaLaunchKernelEx(&cfg, k_noalloc_fields, J, s, (int)n, R, kt, split, out,
                                      (volatile int*)status.device()),
                   "field launch");
        if (via)
            check_cuda(cudaMemcpyAsync(h, out, bytes_h, cudaMemcpyDeviceToDevice, st), "field copy");
        check_cuda(cudaStreamSynchronize(st), "cudaStreamSynchronize");
        if (*status.word()) fail(SG_ETIMEOUT, "a device-side wait expired in the field kernel");
        record_error("");
        return SG_OK;
    } catch (const sg::Error& e) {
        record_error(e.msg);
        return e.code;
    } catch (...) {
        record_error("unknown error");
        return SG_EINVAL;
    }
}
