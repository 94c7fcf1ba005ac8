// Device-side building blocks of the Falcon kernels (sm_103a).
//
// Work decomposition: one warp per chunk of B <= 1025 values.  Lane l owns the 32
// consecutive delta columns 32l .. 32l+31 (column c holds z_{c+2}, Eq. 5), so a 32x32
// bit transpose in registers turns each bit plane into one 32-bit word whose
// little-endian bytes are row bytes 4l .. 4l+3 of that plane (Sec. 3.3, Fig. 8).
#pragma once
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "falcon_internal.h"

#define FALCON_TABLE_QUAL static __constant__ const
#include "falcon_tables.h"

namespace falcon {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Value kinds of the kernels: D = 0 FP64, 1 FP32, 2 FP16 (binary16, R18).  U holds a value's
// bit pattern and every integer derived from it (G, Z) modulo 2^W.
constexpr int kD64 = 0, kD32 = 1, kD16 = 2;
template <int D> struct Traits;
template <> struct Traits<kD64> {
    using U = uint64_t;
    static constexpr int W = 64;            // bits per value
    static constexpr int S = 8;             // bytes per value
    static constexpr int Z1B = 8;           // bytes of z_1 in a record
    static constexpr int A_MAX = 22;        // Case 1: alpha_max <= 22 (Thm 3)
    static constexpr int B_MAX = 15;        // Case 1: beta_hat_max <= 15 (Thm 2)
    static constexpr int A_SENT = 23;       // Case-2 header sentinels
    static constexpr int B_SENT = 16;
    static constexpr int UNITS = 16;        // 16-byte units per lane (32 values)
};
template <> struct Traits<kD32> {
    using U = uint32_t;
    static constexpr int W = 32;
    static constexpr int S = 4;
    static constexpr int Z1B = 4;
    static constexpr int A_MAX = 10;        // 5^10 < 2^24: 10^alpha exact in FP32
    static constexpr int B_MAX = 7;         // 10^7 < 2^24
    static constexpr int A_SENT = 11;
    static constexpr int B_SENT = 8;
    static constexpr int UNITS = 8;
};
template <> struct Traits<kD16> {
    using U = uint16_t;
    static constexpr int W = 16;
    static constexpr int S = 2;
    static constexpr int Z1B = 2;
    static constexpr int A_MAX = 4;         // 5^4 < 2^11: 10^alpha exact in binary16
    static constexpr int B_MAX = 3;         // 10^3 < 2^11
    static constexpr int A_SENT = 5;
    static constexpr int B_SENT = 4;
    static constexpr int UNITS = 4;
};

// --------------------------------------------------------------------------------------
// small helpers
// --------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_none() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Programmatic dependent launch: a kernel launched with launch_after (falcon_internal.h) may start once
// every CTA of the kernel before it has called pdl_trigger or ended; after pdl_wait that kernel, and
// with it all before it, has completed and its writes are visible.  Nothing global is touched earlier.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bulk (TMA) copy of `bytes` from shared to global memory, both 16-byte aligned, bytes a
// multiple of 16, tracked in the issuing thread's bulk groups.  The writers of the shared
// bytes must have executed fence_proxy_async() first.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void bulk_store(void *gdst, const void *ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_addr(ssrc)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the shared source of every committed bulk copy has been read
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// every committed bulk copy has completed
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ uint64_t zigzag(uint64_t x) { return (x << 1) ^ (uint64_t)((int64_t)x >> 63); }
__device__ __forceinline__ uint32_t zigzag(uint32_t x) { return (x << 1) ^ (uint32_t)((int32_t)x >> 31); }
// in 32-bit words: left to the 64-bit forms, 2^26 FP64 segments decompress in 278 us against 273
__device__ __forceinline__ uint64_t unzigzag(uint64_t z) {
    const uint32_t lo = (uint32_t)z, hi = (uint32_t)(z >> 32), s = (uint32_t)((int32_t)(lo << 31) >> 31);
    return ((uint64_t)((hi >> 1) ^ s) << 32) | (__funnelshift_r(lo, hi, 1) ^ s);
}
__device__ __forceinline__ uint32_t unzigzag(uint32_t z) { return (z >> 1) ^ (0u - (z & 1u)); }
__device__ __forceinline__ uint16_t zigzag(uint16_t x) {
    return (uint16_t)(((uint32_t)x << 1) ^ (uint32_t)((int32_t)(int16_t)x >> 15));
}
__device__ __forceinline__ uint16_t unzigzag(uint16_t z) { return (uint16_t)((z >> 1) ^ (0u - (z & 1u))); }

__device__ __forceinline__ uint64_t shfl_u64(uint64_t v, int src) {
    return ((uint64_t)__shfl_sync(kFull, (uint32_t)(v >> 32), src) << 32) |
           __shfl_sync(kFull, (uint32_t)v, src);
}
__device__ __forceinline__ uint64_t shfl_down_u64(uint64_t v, int d) {
    return ((uint64_t)__shfl_down_sync(kFull, (uint32_t)(v >> 32), d) << 32) |
           __shfl_down_sync(kFull, (uint32_t)v, d);
}
__device__ __forceinline__ uint64_t shfl_up_u64(uint64_t v, int d) {
    return ((uint64_t)__shfl_up_sync(kFull, (uint32_t)(v >> 32), d) << 32) |
           __shfl_up_sync(kFull, (uint32_t)v, d);
}
__device__ __forceinline__ uint32_t shfl_x(uint32_t v, int src) { return __shfl_sync(kFull, v, src); }
__device__ __forceinline__ uint64_t shfl_x(uint64_t v, int src) { return shfl_u64(v, src); }
__device__ __forceinline__ uint32_t shfl_down_x(uint32_t v, int d) { return __shfl_down_sync(kFull, v, d); }
__device__ __forceinline__ uint64_t shfl_down_x(uint64_t v, int d) { return shfl_down_u64(v, d); }
__device__ __forceinline__ uint16_t shfl_x(uint16_t v, int src) { return (uint16_t)__shfl_sync(kFull, (uint32_t)v, src); }
__device__ __forceinline__ uint16_t shfl_down_x(uint16_t v, int d) {
    return (uint16_t)__shfl_down_sync(kFull, (uint32_t)v, d);
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
    uint32_t hi = __reduce_max_sync(kFull, (uint32_t)(v >> 32));
    uint32_t lo = __reduce_max_sync(kFull, ((uint32_t)(v >> 32) == hi) ? (uint32_t)v : 0u);
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ uint32_t warp_max_x(uint32_t v) { return __reduce_max_sync(kFull, v); }
__device__ __forceinline__ uint64_t warp_max_x(uint64_t v) { return warp_max_u64(v); }
__device__ __forceinline__ uint32_t warp_or_x(uint32_t v) { return __reduce_or_sync(kFull, v); }
__device__ __forceinline__ uint16_t warp_max_x(uint16_t v) { return (uint16_t)__reduce_max_sync(kFull, (uint32_t)v); }
__device__ __forceinline__ uint16_t warp_or_x(uint16_t v) { return (uint16_t)__reduce_or_sync(kFull, (uint32_t)v); }
__device__ __forceinline__ uint64_t warp_or_x(uint64_t v) {
    return ((uint64_t)__reduce_or_sync(kFull, (uint32_t)(v >> 32)) << 32) | __reduce_or_sync(kFull, (uint32_t)v);
}
// exclusive prefix sum of a 64-bit lane value over the warp
__device__ __forceinline__ uint64_t warp_exclusive_u64(uint64_t v, int lane) {
    uint64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint64_t t = shfl_up_u64(incl, o);
        if (lane >= o) incl += t;
    }
    return incl - v;
}

// the same for a 32-bit lane value
__device__ __forceinline__ uint32_t warp_exclusive_u32(uint32_t v, int lane) {
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    return incl - v;
}

// x where the mask's bits are set, y elsewhere
__device__ __forceinline__ uint32_t bit_select(uint32_t mask, uint32_t x, uint32_t y) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xCA;" : "=r"(r) : "r"(mask), "r"(x), "r"(y));
    return r;
}

// --------------------------------------------------------------------------------------
// 32x32 bit transpose in registers: afterwards bit j of a[i] = old bit i of a[j].
// Recursive exchange of the off-diagonal blocks (Hacker's Delight, Sec. 7-3).
// --------------------------------------------------------------------------------------
__device__ __forceinline__ void transpose32(uint32_t (&a)[32]) {
    // 16- and 8-bit block exchanges are byte permutations (one PRMT per output word)
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t x = a[k], y = a[k + 16];
        a[k] = __byte_perm(x, y, 0x5410);
        a[k + 16] = __byte_perm(x, y, 0x7632);
    }
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if ((k & 8) == 0) {
            const uint32_t x = a[k], y = a[k + 8];
            a[k] = __byte_perm(x, y, 0x6240);
            a[k + 8] = __byte_perm(x, y, 0x7351);
        }
    }
    // the others are a shift and a select each way: four operations per pair of words, where the
    // exchange by masked exclusive ors takes five, four of them on the integer pipe that bounds these
    // kernels (2^26 FP64: compression 373 -> 365 us, decompression 284 -> 278; FP32 144 -> 138)
#define FALCON_TSTEP(h, mask)                                                       \
    _Pragma("unroll") for (int k = 0; k < 32; ++k) {                               \
        if ((k & (h)) == 0) {                                                       \
            const uint32_t x = a[k], y = a[k + (h)];                                \
            a[k] = bit_select(mask, x, y << (h));                                   \
            a[k + (h)] = bit_select(mask, x >> (h), y);                             \
        }                                                                           \
    }
    FALCON_TSTEP(4, 0x0F0F0F0Fu)
    FALCON_TSTEP(2, 0x33333333u)
    FALCON_TSTEP(1, 0x55555555u)
#undef FALCON_TSTEP
}

// 32x32 bit transpose across the warp: afterwards bit l of lane p's word = old bit p of lane l's.
// The 16- and 8-lane exchanges are one byte permute each, the others a rotate and a bitwise select.
struct LaneTranspose {
    uint32_t sel16, sel8;                         // byte-permute selectors
    uint32_t r4, r2, r1, m4, m2, m1;              // rotations and the bits kept
};
__device__ __forceinline__ LaneTranspose lane_transpose_of(int lane) {
    LaneTranspose t;
    t.sel16 = (lane & 16) ? 0x3276u : 0x5410u;
    t.sel8 = (lane & 8) ? 0x3715u : 0x6240u;
    t.r4 = (lane & 4) ? 28u : 4u;
    t.r2 = (lane & 2) ? 30u : 2u;
    t.r1 = (lane & 1) ? 31u : 1u;
    t.m4 = (lane & 4) ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
    t.m2 = (lane & 2) ? 0xCCCCCCCCu : 0x33333333u;
    t.m1 = (lane & 1) ? 0xAAAAAAAAu : 0x55555555u;
    return t;
}
__device__ __forceinline__ uint32_t lane_transpose(uint32_t a, const LaneTranspose &t) {
    uint32_t b;
    a = __byte_perm(a, __shfl_xor_sync(kFull, a, 16), t.sel16);
    a = __byte_perm(a, __shfl_xor_sync(kFull, a, 8), t.sel8);
    b = __shfl_xor_sync(kFull, a, 4);
    a = (a & t.m4) | (__funnelshift_l(b, b, t.r4) & ~t.m4);
    b = __shfl_xor_sync(kFull, a, 2);
    a = (a & t.m2) | (__funnelshift_l(b, b, t.r2) & ~t.m2);
    b = __shfl_xor_sync(kFull, a, 1);
    return (a & t.m1) | (__funnelshift_l(b, b, t.r1) & ~t.m1);
}

// --------------------------------------------------------------------------------------
// Shared-memory staging of a chunk's values, swizzled so that lane l's 16-byte units
// (values 32l .. 32l+31) are read conflict-free: unit u of lane L sits at L*UNITS + (u^(L&7)).
// --------------------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ uint32_t unit_swizzle(uint32_t L, uint32_t u) {
    // lane L's unit u: every 8 consecutive lanes reading their unit u hit 8 distinct 16-byte
    // bank groups (FP16 has 4 units per lane, so lanes L and L + 4 differ by the XOR)
    constexpr int UN = Traits<D>::UNITS;
    return u ^ (UN >= 8 ? (L & 7u) : ((L >> 1) & 3u));
}
template <int D>
__device__ __forceinline__ uint32_t phys_unit(uint32_t q) {
    constexpr int UN = Traits<D>::UNITS;
    uint32_t L = q / UN, u = q % UN;
    return L * UN + unit_swizzle<D>(L, u);
}
template <int D>
__device__ __forceinline__ uint32_t phys_elem_byte(uint32_t e) {
    constexpr int S = Traits<D>::S;
    constexpr int PER = 16 / S;       // values per unit
    return phys_unit<D>(e / PER) * 16u + (e % PER) * S;
}

// Starts loading m values (m <= 1025) from global src into a warp staging buffer
// (cp.async; the caller commits and waits).
template <int D>
__device__ __forceinline__ void stage_values_async(const uint8_t *src, uint32_t m, uint8_t *wsm, int lane) {
    constexpr int S = Traits<D>::S;
    const uint32_t base = smem_addr(wsm);
    const uint32_t nbytes = m * S;
    uint32_t done = 0;
    if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
        const uint32_t nunits = nbytes >> 4;
        constexpr uint32_t FULL_UNITS = 1024u * S / 16u;    // a whole 1024-value chunk
        if (nunits >= FULL_UNITS) {
            // unit q = lane + 32 i belongs to lane L = q / UNITS, slot u = q % UNITS
#pragma unroll
            for (uint32_t i = 0; i < FULL_UNITS / 32u; ++i) {
                const uint32_t q = lane + 32u * i;
                cp_async16(base + phys_unit<D>(q) * 16u, src + 16u * q);
            }
            for (uint32_t q = FULL_UNITS + lane; q < nunits; q += 32) cp_async16(base + phys_unit<D>(q) * 16u, src + 16u * q);
        } else {
            for (uint32_t q = lane; q < nunits; q += 32) cp_async16(base + phys_unit<D>(q) * 16u, src + 16u * q);
        }
        done = (nunits * 16u) / S;
    }
    for (uint32_t e = done + lane; e < m; e += 32) {
        if constexpr (D == kD64) cp_async8(base + phys_elem_byte<D>(e), src + (size_t)e * S);
        else if constexpr (D == kD32) cp_async4(base + phys_elem_byte<D>(e), src + (size_t)e * S);
        else                                     // no 2-byte cp.async: a plain copy (visible at the next __syncwarp)
            *reinterpret_cast<uint16_t *>(wsm + phys_elem_byte<D>(e)) = *reinterpret_cast<const uint16_t *>(src + (size_t)e * S);
    }
}

template <int D>
__device__ __forceinline__ typename Traits<D>::U read_elem(const uint8_t *wsm, uint32_t e) {
    using U = typename Traits<D>::U;
    return *reinterpret_cast<const U *>(wsm + phys_elem_byte<D>(e));
}

// --------------------------------------------------------------------------------------
// Classification (R1: -0, NaN, inf, subnormals are exceptions)
// --------------------------------------------------------------------------------------
__device__ __forceinline__ bool is_special(uint64_t u) {
    const uint64_t a = u & 0x7FFFFFFFFFFFFFFFull;
    return (u != 0) && (a - 0x0010000000000000ull >= 0x7FE0000000000000ull);
}
__device__ __forceinline__ bool is_special(uint32_t u) {
    const uint32_t a = u & 0x7FFFFFFFu;
    return (u != 0) && (a - 0x00800000u >= 0x7F000000u);
}
__device__ __forceinline__ bool is_special(uint16_t u) {
    const uint32_t a = u & 0x7FFFu;
    return (u != 0) && (a - 0x0400u >= 0x7800u);
}

// floor(log10 a) as the largest k with a >= fl(10^k), for a normal, positive, with binary
// exponent in the table's reach (checked by the caller).
__device__ __forceinline__ int floor_log10(uint64_t a) {
    const int e2 = (int)(a >> 52) - 1023;
    int k = (e2 * 78913) >> 18;        // floor(e2 * log10 2) up to +-1
    if (a >= FALCON_P10_F64[k + 1 - FALCON_P10_F64_LO]) ++k;
    else if (a < FALCON_P10_F64[k - FALCON_P10_F64_LO]) --k;
    return k;
}
__device__ __forceinline__ int floor_log10(uint32_t a) {
    const int e2 = (int)(a >> 23) - 127;
    int k = (e2 * 78913) >> 18;
    if (a >= FALCON_P10_F32[k + 1 - FALCON_P10_F32_LO]) ++k;
    else if (a < FALCON_P10_F32[k - FALCON_P10_F32_LO]) --k;
    return k;
}
__device__ __forceinline__ int floor_log10(uint16_t a) {
    const int e2 = (int)(a >> 10) - 15;
    int k = (e2 * 78913) >> 18;
    if (k < FALCON_P10_F16_HI && a >= FALCON_P10_F16[k + 1 - FALCON_P10_F16_LO]) ++k;
    else if (a < FALCON_P10_F16[k - FALCON_P10_F16_LO]) --k;
    return k;
}
// binary-exponent window where floor_log10 is defined and Case 1 is reachable
__device__ __forceinline__ bool log10_in_range(uint64_t a) {
    const uint32_t be = (uint32_t)(a >> 52);
    return be >= 1023u - 90u && be < 1023u + 50u;
}
__device__ __forceinline__ bool log10_in_range(uint32_t a) {
    const uint32_t be = a >> 23;
    return be >= 127u - 40u && be < 127u + 24u;
}
__device__ __forceinline__ bool log10_in_range(uint16_t) { return true; }   // every normal binary16

// --------------------------------------------------------------------------------------
// The per-value test of Alg. 2 at decimal place a, in exact integer arithmetic.
//
// Alg. 2 accepts a for v when v (x) 10^a lies within |x| 2^-52 of an integer (eps <= mu)
// and round(x) / 10^a gives back v.  With v = m 2^E, P = m 5^a and F = -(E + a), the exact
// product is X = P / 2^F; for |X| < 2^50 both conditions together are equivalent to
//   fl(N / 10^a) == v   with N = round(X),
// i.e. |N 2^F - P| < 5^a / 2 (5^a / 4 below a power of two), because the rounding interval
// of v scaled by 10^a is exactly that wide.  The same holds for FP32 (exact x, R14).
// Callers only ask for a with |X| < 10^15 (FP32: < 10^7).
// --------------------------------------------------------------------------------------
__device__ __forceinline__ bool q_test(uint64_t u, int a) {
    const uint64_t au = u & 0x7FFFFFFFFFFFFFFFull;
    if (au == 0) return true;
    const int E = (int)(au >> 52) - 1075;
    const uint64_t m = (au & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const int F = -(E + a);
    if (F <= 0) return true;
    if (F >= 128) return false;
    const uint64_t p5 = FALCON_POW5[a];
    if (F <= 64) {
        // the low F bits of P are the low bits of the 64-bit product: no 128-bit arithmetic
        const uint64_t mask = (F == 64) ? ~0ull : ((1ull << F) - 1ull);
        const uint64_t r = (m * p5) & mask;
        const uint64_t lim = p5 >> 1;
        if (r > (mask >> 1)) return (mask - r) + 1ull <= lim;          // r >= 2^(F-1)
        return r <= ((m == 0x0010000000000000ull) ? ((p5 - 1) >> 2) : lim);
    }
    const unsigned __int128 P = (unsigned __int128)m * p5;
    const unsigned __int128 one = 1;
    const unsigned __int128 r = P & ((one << F) - 1);
    const unsigned __int128 half = one << (F - 1);
    const uint64_t lim = p5 >> 1;
    if (r >= half) return ((one << F) - r) <= lim;
    return r <= ((m == 0x0010000000000000ull) ? ((p5 - 1) >> 2) : lim);
}
__device__ __forceinline__ bool alg2_step_f32(uint32_t u, int a, bool &rt);
__device__ __forceinline__ bool q_test(uint32_t u, int a) {
    bool rt;
    (void)alg2_step_f32(u, a, rt);
    return rt;
}

// Alg. 2's first test alone (eps <= mu) for FP32, on the exact product x = v * 10^a (R14):
// the distance of X = P / 2^F to the nearest integer is at most X * 2^-23.
__device__ __forceinline__ bool eps_le_mu(uint32_t u, int a) {
    const uint32_t au = u & 0x7FFFFFFFu;
    if (au == 0) return true;
    const int E = (int)(au >> 23) - 150;
    const uint64_t m = (au & 0x007FFFFFu) | 0x00800000u;
    const int F = -(E + a);
    if (F <= 0) return true;
    if (F >= 64) return false;
    const uint64_t P = m * FALCON_POW5[a];
    const uint64_t r = P & ((1ull << F) - 1);
    const uint64_t rc = (1ull << F) - r;
    const uint64_t dist = r < rc ? r : rc;
    return dist <= (P >> 23);
}

// Both tests of Alg. 2 for FP32 at decimal place a, from one product: eps <= mu (returned)
// and the round trip (rt), as eps_le_mu and q_test compute them.  P = m 5^a < 2^48 comes from
// one 32 x 32 -> 64 multiply; for F < 32 the remainder and both bounds are 32-bit.
__device__ __forceinline__ bool alg2_step_f32(uint32_t u, int a, bool &rt) {
    const uint32_t au = u & 0x7FFFFFFFu;
    const int F = 150 - (int)(au >> 23) - a;
    if (au == 0 || F <= 0) { rt = true; return true; }
    if (F >= 64) { rt = false; return false; }
    const uint32_t m = (au & 0x007FFFFFu) | 0x00800000u;
    const uint32_t p5 = (uint32_t)FALCON_POW5[a];          // 5^a < 2^24 for a <= 10
    const uint64_t P = (uint64_t)m * p5;
    const uint32_t lim = p5 >> 1, lim_low = (m == 0x00800000u) ? ((p5 - 1u) >> 2) : lim;
    const uint32_t mu = (uint32_t)(P >> 23);                // < 2^25
    if (F < 32) {
        const uint32_t mask = (1u << F) - 1u;
        const uint32_t r = (uint32_t)P & mask, rc = mask - r + 1u;
        rt = (r > (mask >> 1)) ? (rc <= lim) : (r <= lim_low);
        return (r < rc ? r : rc) <= mu;
    }
    const uint64_t mask = (1ull << F) - 1ull;
    const uint64_t r = P & mask, rc = mask - r + 1ull;
    rt = (r > (mask >> 1)) ? (rc <= lim) : (r <= lim_low);
    return (r < rc ? r : rc) <= mu;
}

// FP32 decimal place of one value as Alg. 2 finds it, restricted to [0, atop]: the first a
// with eps <= mu, accepted only if the round trip holds there; -1 otherwise (an exception
// or a decimal place beyond atop, both of which make the chunk Case 2).  The 24-bit
// significand leaves no margin for Thm 4 at beta = 7, so early spurious passes are real
// and must be reproduced value by value.
__device__ __forceinline__ int first_pass_f32(uint32_t u, int atop) {
    if ((u & 0x7FFFFFFFu) == 0) return 0;
    for (int a = 0; a <= atop; ++a)
        if (eps_le_mu(u, a)) return q_test(u, a) ? a : -1;
    return -1;
}

// g = round(v (x) 10^a) (Eq. 4, Case 1) for a value that passed q_test at a.  Passing means
// X = v 10^a lies within 5^a / 2^(F+1) <= 1/8 of the integer g (the rounding interval of v,
// scaled), so an approximation of X closer than 3/8 rounds to g: with m and 5^a both
// normalised to 64 bits, mulhi(m 2^11, 5^a 2^(63-d)) = floor(X 2^sh), sh = F + 10 - d >= 13,
// is X within 2^-13, and rounding it at bit sh gives g.  One 64-bit high product per value.
__device__ __forceinline__ uint64_t case1_round(uint64_t m, uint64_t norm, int sh) {
    const uint64_t t = __umul64hi(m << 11, norm);
    return ((t >> (sh - 1)) + 1ull) >> 1;
}
__device__ __forceinline__ uint64_t case1_g(uint64_t u, int a) {
    const uint64_t au = u & 0x7FFFFFFFFFFFFFFFull;
    if (au == 0) return 0;
    const int E = (int)(au >> 52) - 1075;
    const uint64_t m = (au & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const uint64_t N = case1_round(m, FALCON_POW5_NORM[a], -(E + a) + 10 - (int)FALCON_LOG2_POW5[a]);
    return (u >> 63) ? (0ull - N) : N;
}
// The same for values with |g| < 10^8 (beta_hat <= kNarrowBeta): one 32-bit high product.  The top
// words of m and 5^a, both normalised, give t >= 2^30 within three of X 2^sh, and X < 10^8 makes
// sh >= 4, so t 2^-sh is within 3/16 of X, itself within X 2^-53 of g.
constexpr int kNarrowBeta = 8;
struct Case1Narrow {
    uint32_t norm;                                // top word of 5^a normalised
    int c;                                        // sh - 1 = c - exponent field
};
__device__ __forceinline__ Case1Narrow case1_narrow_of(int a) {
    return {(uint32_t)(FALCON_POW5_NORM[a] >> 32), 1075 - a + 10 - (int)FALCON_LOG2_POW5[a] - 32 - 1};
}
// shifts that give 0 past 31 (a value of +0 has the largest)
__device__ __forceinline__ uint32_t shr_clamp(uint32_t x, uint32_t n) {
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
__device__ __forceinline__ uint64_t shr_clamp64(uint64_t x, uint32_t n) {
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
}
__device__ __forceinline__ uint32_t shl_clamp(uint32_t x, uint32_t n) {
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
__device__ __forceinline__ uint32_t case1_n_narrow(uint32_t hi, uint32_t lo, const Case1Narrow &q) {      // |g|
    const uint32_t top = __funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, 11);
    const uint32_t sh = (uint32_t)(q.c - (int)((hi >> 20) & 0x7FFu));
    return (shr_clamp(__umulhi(top, q.norm), sh) + 1u) >> 1;
}
__device__ __forceinline__ uint32_t case1_g_narrow(uint64_t u, const Case1Narrow &q) {
    const uint32_t hi = (uint32_t)(u >> 32), s = (uint32_t)((int32_t)hi >> 31);
    return (case1_n_narrow(hi, (uint32_t)u, q) ^ s) - s;
}
// FP32: m 2^8 times 5^a normalised to 32 bits is the exact product P, normalised; X < 10^7 makes its
// rounding bit lie in the top word, so g = floor(X + 1/2) comes from one 32-bit high product.
struct Case1F32 {
    uint32_t p5, norm;                            // 5^a, 5^a with its top bit at bit 31
    int c, f0;                                    // shift - 1 = c - exponent field, F = f0 - exponent field
};
__device__ __forceinline__ Case1F32 case1_f32_of(int a) {
    const uint32_t p5 = (uint32_t)FALCON_POW5[a];
    const int d = (int)FALCON_LOG2_POW5[a];
    // X = P 2^-F, t = P 2^(8 + 31 - d - 32): shift = F + 7 - d
    return {p5, p5 << (31 - d), 150 - a + 7 - d - 1, 150 - a};
}
__device__ __forceinline__ uint32_t case1_n(uint32_t u, const Case1F32 &q) {            // |g|
    const uint32_t m8 = (u << 8) | 0x80000000u;
    return (shr_clamp(__umulhi(m8, q.norm), (uint32_t)(q.c - (int)((u >> 23) & 0xFFu))) + 1u) >> 1;
}
__device__ __forceinline__ uint32_t case1_g(uint32_t u, const Case1F32 &q) {
    const uint32_t s = (uint32_t)((int32_t)u >> 31);
    return (case1_n(u, q) ^ s) - s;
}
__device__ __forceinline__ uint32_t case1_g(uint32_t u, int a) { return case1_g(u, case1_f32_of(a)); }

// binary16 (R18): both tests of Alg. 2 at decimal place a, in exact FP32 arithmetic (the FMA pipe has
// room where the integer pipe is the limit): X = v 10^a has an 11-bit times a 10-bit significand, its
// nearest integer N comes from adding 1.5 2^23 (callers only ask for |X| < 2^22), X - N is exact.
// eps <= mu is |X - N| <= |X| 2^-10, the round trip |X - N| <= half an ulp of v times 10^a.  (Equality
// cannot occur there: 5^a is odd.  Below a power of two the ulp is half as wide, which changes nothing:
// X 2^F = 2^10 5^a, and its distance to a multiple of 2^F is 0 or at least 2^10 > 5^a / 2.)
struct Scale16 {
    float p, half;                                // 10^a, 10^a 2^-11
};
__device__ __forceinline__ Scale16 scale16_of(int a) {
    const float p = __uint_as_float(FALCON_P10_F32[a - FALCON_P10_F32_LO]);
    return {p, p * 0x1p-11f};
}
constexpr float kRound16 = 12582912.0f;           // 1.5 2^23
__device__ __forceinline__ bool alg2_step_f16(uint16_t u, const Scale16 &q, bool &rt) {
    const float v = __half2float(__ushort_as_half(u)), x = v * q.p;
    const float n = (x + kRound16) - kRound16, eps = fabsf(x - n);
    rt = eps <= __uint_as_float(__float_as_uint(v) & 0x7F800000u) * q.half;
    return eps <= fabsf(x) * 0x1p-10f;
}
__device__ __forceinline__ bool alg2_step_f16(uint16_t u, int a, bool &rt) { return alg2_step_f16(u, scale16_of(a), rt); }
__device__ __forceinline__ bool q_test(uint16_t u, int a) {
    bool rt;
    (void)alg2_step_f16(u, a, rt);
    return rt;
}
// Alg. 2's decimal place of one binary16 value within [0, atop]: the first a with eps <= mu,
// -1 if the round trip fails there (an early stop) or no a passes
__device__ __forceinline__ int first_pass_f16(uint16_t u, int atop) {
    if ((u & 0x7FFFu) == 0) return 0;
    for (int a = 0; a <= atop; ++a) {
        bool rt;
        if (alg2_step_f16(u, a, rt)) return rt ? a : -1;
    }
    return -1;
}
// g of a value that passed: the low bits of X + 1.5 2^23
__device__ __forceinline__ uint16_t case1_g(uint16_t u, const Scale16 &q) {
    return (uint16_t)__float_as_uint(__half2float(__ushort_as_half(u)) * q.p + kRound16);
}
__device__ __forceinline__ uint16_t case1_g(uint16_t u, int a) { return case1_g(u, scale16_of(a)); }

// fl(g / 10^a), correctly rounded (nearest, ties to even), for |g| <= 2^53 and 0 <= a <= 22, in
// integer arithmetic (the inverse of Eq. 4, Case 1).  g / 10^a = (g / 5^a) 2^-a and the
// scaling by 2^-a is exact (no result is subnormal), so the work is one correctly rounded
// division by 5^a: with G = |g| normalised to [2^63, 2^64), d = floor(log2 5^a) and the
// reciprocal R = floor(2^(64+d) / 5^a), T = mulhi(G, R) is floor(Q) or one less, Q = G 2^d / 5^a
// (division by an invariant integer, Granlund and Montgomery, PLDI 1994).  (a = 0: R = 2^64 - 1
// gives T = G - 1.)  Q has 63 or 64 integer bits, of which 10 or 11 lie below the 53-bit result.
// A tie cannot occur (a 54-bit quotient times 5^a exceeds 2^53 or a = 0 and g fits), so Q rounds up
// iff Q's dropped part is at least half: T's next bit decides, except when T's dropped bits are
// one below half, where the remainder G 2^d - T 5^a (below 2 * 5^a, exact modulo 2^64) says
// whether floor(Q) is T + 1.  That happens for one value in 1024 to 2048, so its two products are
// off the common path.
struct Div10 {
    uint64_t R, D;                                // reciprocal, 5^a
    int d, e0;                                    // floor(log2 5^a), exponent of T's unit
};
__device__ __forceinline__ Div10 div10_of(int a) {
    const int d = FALCON_LOG2_POW5[a];
    return {a > 0 ? FALCON_RECIP5[a] : ~0ull, FALCON_POW5[a], d, 11 - d - a + 52 + 1022};
}
// bits of the double T-or-T+1 rounds to; s = the shift that normalised |g|
__device__ __forceinline__ uint64_t div10_round(uint64_t G, uint64_t T, int s, const Div10 &q) {
    const uint32_t lz = (uint32_t)(~T >> 63);     // T has 63 or 64 significant bits
    const uint64_t Tn = T << lz;
    uint32_t up = ((uint32_t)Tn >> 10) & 1u;
    if (((((uint32_t)Tn) & 0x7FFu) | lz) == 0x3FFu) up = (G << q.d) - T * q.D >= q.D;
    // the significand's leading one adds one to the biased exponent field, a carry another
    return ((uint64_t)(uint32_t)(q.e0 - (int)lz - s) << 52) + (Tn >> 11) + up;
}
__device__ __forceinline__ uint64_t div_pow10_exact(int64_t g, const Div10 &q) {
    const uint64_t sign = (uint64_t)g & 0x8000000000000000ull;
    const uint64_t ag = g < 0 ? 0ull - (uint64_t)g : (uint64_t)g;
    const int s = __clzll((long long)ag);
    const uint64_t G = ag << (s & 63);
    const uint64_t v = div10_round(G, __umul64hi(G, q.R), s, q) | sign;
    return ag ? v : 0;
}
// The same for |g| < 2^32 and a <= 17, given as |g| and a sign word (top bit), with a 96-bit
// reciprocal and no remainder: T = floor(Q - e) with e < 2^-32, and Q, a multiple of 1 / 5^a that is
// never a tie, lies at least 2^9 / 5^a > 2^-32 from the point where rounding changes, so T's next
// bit decides.  (Q an integer: T = Q - 1 rounds alike, as above.)
struct Div10Narrow {
    uint32_t r0, r1, r2;                          // 2^(96+d) / 5^a, low word first
    int e0;
};
constexpr int kDiv10NarrowMax = 17;
__device__ __forceinline__ Div10Narrow div10_narrow_of(int a) {
    const uint64_t r = a > 0 ? FALCON_RECIP5[a] : ~0ull;
    return {FALCON_RECIP5_LO[a], (uint32_t)r, (uint32_t)(r >> 32), 11 - (int)FALCON_LOG2_POW5[a] - a + 52 + 1022 - 32};
}
__device__ __forceinline__ uint64_t div_pow10_exact32(uint32_t ag, uint32_t sgn, const Div10Narrow &q) {
    const int s = __clz((int)ag);
    const uint32_t G = ag << (s & 31);
    const uint64_t lo = (uint64_t)G * q.r1 + __umulhi(G, q.r0);
    const uint64_t T = (uint64_t)G * q.r2 + (uint32_t)(lo >> 32);
    // T's top bit is bit 63 or 62: one bit more than the significand, then rounded (40 M decimal
    // values at block 1025: 182.8 us normalised first, 179.2 with this one variable shift)
    const uint32_t hi = (uint32_t)(T >> 32), b = hi >> 31, n = 9u + b;
    const uint64_t M = ((((uint64_t)(hi >> n) << 32) | __funnelshift_r((uint32_t)T, hi, n)) + 1u) >> 1;
    const uint32_t top = ((uint32_t)(q.e0 - 1 - s + (int)b) << 20) + (uint32_t)(M >> 32);
    return ((uint64_t)(ag ? top | (sgn & 0x80000000u) : 0u) << 32) | (uint32_t)M;      // of 0: M = 0
}

__device__ __forceinline__ void set_status(unsigned long long *result, uint32_t code) {
    atomicCAS(&result[1], 0ull, (unsigned long long)code);
}

// block-wide exclusive scan of one u64 per thread (1024 threads); returns the block total
__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t &total, uint64_t *warp_sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t incl = v + warp_exclusive_u64(v, lane);
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint64_t ws = warp_sums[lane];
        const uint64_t wincl = ws + warp_exclusive_u64(ws, lane);
        warp_sums[lane] = wincl - ws;
        if (lane == 31) warp_sums[32] = wincl;
    }
    __syncthreads();
    const uint64_t r = warp_sums[warp] + incl - v;
    total = warp_sums[32];
    __syncthreads();
    return r;
}

// Finds the job that owns global chunk t (jobs sorted by chunk_begin), the whole warp probing 32
// places at a time: two dependent loads for a thousand jobs instead of ten.
__device__ __forceinline__ const Job *find_job(const Job *jobs, int njobs, uint64_t t, int lane) {
    int lo = 0, n = njobs;                        // the owner lies in [lo, lo + n)
    while (n > 1) {
        const int step = (n + 31) / 32, i = lane * step;
        const unsigned le = __ballot_sync(kFull, i < n && jobs[lo + (i < n ? i : 0)].chunk_begin <= t);
        const int k = (31 - __clz((int)le)) * step;       // the last probe that begins at or before t
        lo += k;
        n = min(step, n - k);
    }
    return jobs + lo;
}

// Chunk hand-out (Control).  A warp's first chunk is the one of its own number; tickets, drawn by
// one atomic add each, hand out the rest, so a grid with a warp for every chunk draws none (and nobody
// has to reset its counter).  draw issues lane 0's atomic and returns its raw result (valid in lane 0
// only); chunk broadcasts it.  Issuing the atomic a chunk before its result is read hides its latency
// behind the current chunk; the add is predicated into a register set beforehand, so no instruction
// selects between the two and waits for it.
struct Tickets {
    Control *ctl;
    int which;
    uint64_t total;
    __device__ __forceinline__ uint32_t warps() const { return gridDim.x * (blockDim.x >> 5); }
    __device__ __forceinline__ uint64_t first() const { return blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); }
    __device__ __forceinline__ unsigned long long draw(int lane) const {
        unsigned long long r;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\tmov.b64 %0, %3;\n\t"
            "@p atom.global.add.u64 %0, [%2], 1;\n\t}"
            : "=l"(r)
            : "r"((int)(lane == 0 && warps() < total)), "l"(&ctl->ticket[which]), "l"(total)
            : "memory");
        return r;
    }
    __device__ __forceinline__ uint64_t chunk(unsigned long long raw) const { return warps() + shfl_u64(raw, 0); }
};

__device__ __forceinline__ uint32_t chunk_cols(uint32_t m) { return m <= 1 ? 0u : ((m - 1u + 63u) & ~63u); }

}  // namespace falcon
