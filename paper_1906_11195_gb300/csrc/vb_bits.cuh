// vb_bits.cuh -- spin words of one vertex (R replicas of 64 lanes), their loads and stores, and
// bit-sliced counting: one 64-bit word holds one binary digit of 64 lanes' counts.
#pragma once

#include "sg_internal.cuh"

namespace sg {

template <int R>
struct SpinWords { uint64_t v[R]; };

template <int R>
__device__ __forceinline__ SpinWords<R> load_words(const uint64_t* p) {
    SpinWords<R> s;
    if constexpr (R == 1) {
        s.v[0] = p[0];
    } else if constexpr (R == 2) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p);
        s.v[0] = a.x; s.v[1] = a.y;
    } else {
        const ulonglong2 a = reinterpret_cast<const ulonglong2*>(p)[0];
        const ulonglong2 b = reinterpret_cast<const ulonglong2*>(p)[1];
        s.v[0] = a.x; s.v[1] = a.y; s.v[2] = b.x; s.v[3] = b.y;
    }
    return s;
}

template <int R>
__device__ __forceinline__ SpinWords<R> gather_words(const uint64_t* p) {
    SpinWords<R> s;
    if constexpr (R == 1) {
        s.v[0] = __ldg(p);
    } else if constexpr (R == 2) {
        const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2*>(p));
        s.v[0] = a.x; s.v[1] = a.y;
    } else {
        const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2*>(p));
        const ulonglong2 b = __ldcg(reinterpret_cast<const ulonglong2*>(p) + 1);
        s.v[0] = a.x; s.v[1] = a.y; s.v[2] = b.x; s.v[3] = b.y;
    }
    return s;
}

template <int R>
__device__ __forceinline__ void store_words_keep(uint64_t* p, const SpinWords<R>& s, uint64_t pol) {
    if constexpr (R == 1) {
        asm volatile("st.global.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(p), "l"(s.v[0]), "l"(pol)
                     : "memory");
    } else {
#pragma unroll
        for (int h = 0; h < R / 2; ++h)
            asm volatile("st.global.L2::cache_hint.v2.u64 [%0], {%1, %2}, %3;" ::"l"(p + 2 * h),
                         "l"(s.v[2 * h]), "l"(s.v[2 * h + 1]), "l"(pol)
                         : "memory");
    }
}

// add one 64-lane word into a P-plane bit-sliced counter (the count never exceeds 2^P - 1)
template <int P>
__device__ __forceinline__ void bitslice_add(uint64_t (&p)[P], uint64_t x) {
#pragma unroll
    for (int b = 0; b < P; ++b) {
        const uint64_t c = p[b] & x;
        p[b] ^= x;
        x = c;
    }
}

// full adder on 64 lanes at once (lowers to 3-input logic operations)
__device__ __forceinline__ void full_add(uint64_t a, uint64_t b, uint64_t c, uint64_t& s,
                                         uint64_t& cy) {
    s = a ^ b ^ c;
    cy = (a & b) | (c & (a ^ b));
}

// p += x0 + x1 + x2 + x3, lane by lane (the sum fits P planes)
template <int P>
__device__ __forceinline__ void bitslice_add4(uint64_t (&p)[P], uint64_t x0, uint64_t x1, uint64_t x2,
                                              uint64_t x3) {
    uint64_t c1, c2, c;
    full_add(p[0], x0, x1, p[0], c1);
    full_add(p[0], x2, x3, p[0], c2);
    full_add(p[1], c1, c2, p[1], c);
#pragma unroll
    for (int b = 2; b < P; ++b) {
        const uint64_t s = p[b] ^ c;
        c = p[b] & c;
        p[b] = s;
    }
}

// lanes whose P-plane count u is >= k (0 <= k <= 2^P - 1): the carry out of u + (2^P - k)
template <int P>
__device__ __forceinline__ uint64_t at_least(const uint64_t (&p)[P], int k) {
    const uint32_t c = (1u << P) - (uint32_t)k;
    uint64_t carry = 0ull;
#pragma unroll
    for (int b = 0; b < P; ++b) {
        const uint64_t cb = ((c >> b) & 1u) ? ~0ull : 0ull;
        carry = (p[b] & carry) | (cb & (p[b] | carry));
    }
    return k == 0 ? ~0ull : carry;
}

}  // namespace sg
