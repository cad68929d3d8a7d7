// rank_select.cuh -- warp-wide selection and sorting of (score, id) entries,
// shared by the ranking kernels.
#pragma once

#include "search.cuh"

namespace sieve {

// selection: monotone map of fp32 to uint32 (larger float -> larger key); -0
// is mapped as +0 so that equal scores have equal keys
__device__ __forceinline__ uint32_t order_key(float s) {
    const uint32_t u = __float_as_uint(s + 0.f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// the inverse of order_key
__device__ __forceinline__ float key_score(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

constexpr int kSelectMaxR = 8;   // lane order statistics used for the lower bracket

// warp-wide reductions in one instruction (redux.sync), not a chain of shuffles
__device__ __forceinline__ int warp_sum(int x) { return __reduce_add_sync(0xffffffffu, x); }

template <int KPL>
__device__ __forceinline__ int count_ge(const uint32_t (&key)[KPL], uint32_t t) {
    int c = 0;
#pragma unroll
    for (int j = 0; j < KPL; ++j) c += key[j] >= t;
    return warp_sum(c);
}

// A bracket L <= T* <= U of the want-th largest of the warp's keys (keys of
// padding are 0, below every score): U = the largest key, L = the smallest over
// lanes of each lane's ceil(want / 32)-th largest key, so at least want keys
// are >= L.  L = 0 when that rank is past kSelectMaxR.
template <int KPL>
__device__ __forceinline__ void warp_bracket(const uint32_t (&key)[KPL], int want, uint32_t &L,
                                             uint32_t &U) {
    const int r = (want + 31) / 32;
    uint32_t m[kSelectMaxR] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (r <= 2) {
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
            m[1] = max(m[1], min(m[0], key[j]));
            m[0] = max(m[0], key[j]);
        }
    } else if (r <= 4) {
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
            uint32_t x = key[j];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t hi = max(m[i], x);
                x = min(m[i], x);
                m[i] = hi;
            }
        }
    } else if (r <= kSelectMaxR) {
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
            uint32_t x = key[j];
#pragma unroll
            for (int i = 0; i < kSelectMaxR; ++i) {
                const uint32_t hi = max(m[i], x);
                x = min(m[i], x);
                m[i] = hi;
            }
        }
    } else {   // no lower bracket, but U is still the largest key
#pragma unroll
        for (int j = 0; j < KPL; ++j) m[0] = max(m[0], key[j]);
    }
    L = 0u;
#pragma unroll
    for (int i = 0; i < kSelectMaxR; ++i) L = r == i + 1 ? m[i] : L;
    U = __reduce_max_sync(0xffffffffu, m[0]);
    L = __reduce_min_sync(0xffffffffu, L);
}

// A threshold T <= T* (T* = the want-th largest of the warp's keys) with C =
// #{keys >= T} >= want, refined bit by bit (the largest T with at least want
// keys >= T) until C <= cap or T == T*.  The search starts from the common
// high bits of the bracket L, U.
template <int KPL>
__device__ __forceinline__ void warp_threshold(const uint32_t (&key)[KPL], int want, int cap,
                                               uint32_t &T, int &C) {
    uint32_t L, U;
    warp_bracket(key, want, L, U);
    int b;
    if (L == U) {
        b = -1;
        T = L;
    } else {
        b = 31 - __clz(L ^ U);                                // highest bit where they differ
        T = b == 31 ? 0u : (L & ~((2u << b) - 1u));           // their common high bits
    }
    C = count_ge(key, T);
    for (; b >= 0 && C > cap; --b) {
        const uint32_t t = T | (1u << b);
        const int c = count_ge(key, t);
        if (c >= want) {
            T = t;
            C = c;
        }
    }
}

// Bitonic sort of the warp's R * 32 entries (entry i = r * 32 + lane in
// register r), first-ranked first by (score desc, id asc).  Partners within a
// register are exchanged by shuffles, partners across registers in place.
// Entries are distinct except identical padding, so both sides of a pair
// take the same decision.
template <int R>
__device__ __forceinline__ void warp_sort_regs(float (&s)[R], int (&c)[R]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
                const int jr = j >> 5;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r & jr) continue;
                    const int r2 = r | jr;
                    const bool up = ((r * 32) & k) == 0;   // this block sorts first-ranked first
                    // the lower entry keeps the better one when up, else the worse
                    const bool swap = up ? ranks_before(s[r2], c[r2], s[r], c[r])
                                         : ranks_before(s[r], c[r], s[r2], c[r2]);
                    if (swap) {
                        const float ts = s[r];
                        const int tc = c[r];
                        s[r] = s[r2];
                        c[r] = c[r2];
                        s[r2] = ts;
                        c[r2] = tc;
                    }
                }
            } else {
                const bool lower = (lane & j) == 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float ps = __shfl_xor_sync(0xffffffffu, s[r], j);
                    const int pc = __shfl_xor_sync(0xffffffffu, c[r], j);
                    const bool up = (((r * 32) + lane) & k) == 0;
                    const bool take = (lower == up) ? ranks_before(ps, pc, s[r], c[r])
                                                    : ranks_before(s[r], c[r], ps, pc);
                    if (take) {
                        s[r] = ps;
                        c[r] = pc;
                    }
                }
            }
        }
    }
}

}  // namespace sieve
