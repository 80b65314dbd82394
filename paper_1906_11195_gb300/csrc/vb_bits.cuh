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

// lanes whose counter value is >= k (k a per-thread scalar, 0 <= k <= 2^P - 1)
template <int P>
__device__ __forceinline__ uint64_t bitslice_ge(const uint64_t (&p)[P], int k) {
    uint64_t gt = 0ull, eq = ~0ull;
#pragma unroll
    for (int b = P - 1; b >= 0; --b) {
        const uint64_t kb = ((k >> b) & 1) ? ~0ull : 0ull;
        gt |= eq & p[b] & ~kb;
        eq &= ~(p[b] ^ kb);
    }
    return gt | eq;
}

// full adder and half adder on 64 lanes at once (each lowers to 3-input logic operations)
__device__ __forceinline__ void full_add(uint64_t a, uint64_t b, uint64_t c, uint64_t& s,
                                         uint64_t& cy) {
    s = a ^ b ^ c;
    cy = (a & b) | (c & (a ^ b));
}

__device__ __forceinline__ void half_add(uint64_t a, uint64_t b, uint64_t& s, uint64_t& cy) {
    s = a ^ b;
    cy = a & b;
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

// planes needed to count W one-bit inputs
template <int W>
struct CountBits { static constexpr int P = W <= 1 ? 1 : W <= 3 ? 2 : W <= 7 ? 3 : 4; };

// p = bit-sliced number of set inputs among x[0..W-1], per lane (carry-save adder trees)
template <int W>
__device__ __forceinline__ void count_bits(const uint64_t (&x)[W], uint64_t (&p)[CountBits<W>::P]) {
    if constexpr (W == 1) {
        p[0] = x[0];
    } else if constexpr (W == 2) {
        half_add(x[0], x[1], p[0], p[1]);
    } else if constexpr (W == 3) {
        full_add(x[0], x[1], x[2], p[0], p[1]);
    } else if constexpr (W == 4 || W == 5) {
        uint64_t s1, c1, c2;
        full_add(x[0], x[1], x[2], s1, c1);
        if constexpr (W == 4) half_add(s1, x[3], p[0], c2);
        else full_add(s1, x[3], x[4], p[0], c2);
        half_add(c1, c2, p[1], p[2]);
    } else if constexpr (W == 6 || W == 7) {
        uint64_t s1, c1, s2, c2, c3;
        full_add(x[0], x[1], x[2], s1, c1);
        full_add(x[3], x[4], x[5], s2, c2);
        if constexpr (W == 6) half_add(s1, s2, p[0], c3);
        else full_add(s1, s2, x[6], p[0], c3);
        full_add(c1, c2, c3, p[1], p[2]);
    } else {
        static_assert(W == 8, "narrow path covers widths 1..8");
        uint64_t s1, c1, s2, c2, s3, c3, c4;
        full_add(x[0], x[1], x[2], s1, c1);
        full_add(x[3], x[4], x[5], s2, c2);
        full_add(s1, s2, x[6], s3, c3);
        half_add(s3, x[7], p[0], c4);
        // the four weight-2 carries
        uint64_t t1, d1, d2;
        full_add(c1, c2, c3, t1, d1);
        half_add(t1, c4, p[1], d2);
        half_add(d1, d2, p[2], p[3]);
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
