// Falcon compression (Sec. 3 of the paper; the work of Alg. 3 CmpKernel) for sm_103a, as
// two or three launches, none of which waits on another warp:
//   1. analyse: each warp takes its chunks by ticket (its one shared-memory value buffer
//      receives the next chunk by cp.async, swizzled, as soon as the current one is in registers)
//      and computes
//      - specials (R1) and the largest magnitude from three-input maxima and minima of the values'
//        magnitudes,
//      - Case 1 / Case 2 of Eq. 4, out of line over the staged values: the smallest decimal place
//        alpha_max at which every value passes Alg. 2's test, in exact integer arithmetic (q_test,
//        test_g); FP32 checks Alg. 2's early stops where they are possible; Case 1 leaves G in the
//        values' place,
//      - the ORs of |Z| (Eq. 5) over 8-column groups, the bit width w, and from those ORs,
//        transposed across the warp, the non-zero bytes of every row (Sec. 3.3 lambda) without
//        forming the bit planes; sparse/dense per row; the record size, which goes
//        into the stream's size array; alpha, beta_hat, w and the dense-row mask, which go into the
//        workspace;
//   2. offsets (decompress.cu; the size synchronisation of Sec. 3.4): every record's position into
//      the workspace.  Streams of at most 1024 chunks skip it, their emit warps add up the sizes;
//   3. emit: the values again (straight from global memory, a whole sector per lane and load, not kept in
//      L1, the next chunk prefetched into L2), G, the deltas' bit planes (32x32 register transposes, one
//      32-bit word per plane: 4 row bytes per lane), zigzagged by one XOR with the sign plane, through
//      128-byte slots into the record, assembled in shared memory at the output's 16-byte phase and
//      sent to its offset with one TMA bulk copy;
//      the warp of each job's first chunk writes the header and the stream length and checks
//      the capacity.
// Both are bound by integer issue (FP64 segments: ALU pipe 75 % and 66 % of active cycles, 1235 and 2741
// warp instructions per chunk, against 1801 and 3590 with ballots and reductions per sparse row,
// per-value zigzags and bit-sliced counts) and, where chunks take different paths, by instruction fetch.
// 2^26 segment values: FP64 520 -> 357 us, FP32 270 -> 206 us; Case-1 FP64 of 40 M values in 1025-value
// chunks 622 -> 317 us.  Slower, and left out (each measured when the rest stood at about 450 us): two
// copies of the row code (FP64 485 us: instruction fetch), a transpose shared by both halves in a loop
// (475 us), dense rows moved in 16-byte units (FP64 461, FP32 238 us), values kept in L1 (483 us).  The
// offsets launch in place of per-tile and per-group sums (two atomics per chunk in the analysis, five loads
// and a reduction per chunk in the emit, a reset of the workspace): FP64 452 -> 441 us, 2^20-value walk 40 -> 37 us.
// The paper resolves offsets inside one launch with a decoupled look-back; with about 1800
// resident warps on a GB300 the waits of that look-back took half of every warp's time, while
// the analysis recomputed by the emit launch costs less.
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "falcon_device.cuh"

namespace falcon {

namespace {

// one chunk of values (1025, swizzled) of a kind
template <int D> constexpr int kAnalyseWarpBytes = 1024 * Traits<D>::S + 32;

// The emit launch's per-warp buffers: the record, assembled at the output's 16-byte phase, and
// 128-byte slots for the rows of 32 planes at a time, top plane first (FP64 runs its two halves one
// after the other through the same slots).  A row takes at most 128 bytes of the record, 16 more in
// an every-row-sparse one (Sec. 5.4.2 ablation, the wide layout).
// A chunk's planes go into the slots while the bulk copy of the warp's previous record may still be
// reading its buffer, so the slots lie past the longest record of any kind the warp meets: the form's
// layout places them, for every kind it runs.  (Placed by the chunk's own kind in the either-dtype form,
// the slots of an FP32 or FP16 chunk were inside the FP64 record before it.)
template <int D, bool kWide> struct EmitLayout {
    static constexpr uint32_t W = Traits<D>::W;
    static constexpr uint32_t kRec = (3u + Traits<D>::Z1B + W / 8u + W * (kWide ? 144u : 128u) + 15u + 15u) / 16u * 16u;
    static constexpr uint32_t kRows = W < 32u ? W : 32u;
    static constexpr uint32_t kBytes = kRec + kRows * 128u + 16u;         // + 16 readable past any slot
    // where kind K's chunks have their slots in this form's buffer
    template <int K> static constexpr uint32_t slots_of() {
        using Own = EmitLayout<K, kWide>;
        static_assert(Own::kRec <= kRec && kRec + Own::kRows * 128u + 16u <= kBytes,
                      "a chunk's slots would overlap a record that is still being copied out, or the next warp's buffer");
        return kRec;
    }
};

// Byte-permute selector that moves a word's non-zero bytes to its front, by nibble n (bit 3 - i: byte
// i is non-zero).  Lane l keeps the selector of nibble l & 15, so one shuffle looks it up.
__device__ __forceinline__ uint32_t compact_sel(uint32_t n) {
    uint32_t sel = 0x4444u, r = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if ((n >> (3 - i)) & 1u) {
            sel = (sel & ~(15u << (4 * r))) | ((uint32_t)i << (4 * r));
            ++r;
        }
    }
    return sel;
}

// 128 times the non-zero nibble of x (bit 3 - i set iff byte i is non-zero): the bytes' high-bit flags
// weighted and added by one four-way dot product (by a high multiply: 2^26 FP64 361 us against 356.5)
__device__ __forceinline__ uint32_t nz_nibble128(uint32_t x) {
    const uint32_t y = (((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u;
    return __dp4a(y, 0x01020408u, 0u);
}

// inclusive prefix sum over the warp (the shuffle's own predicate says which lanes add)
__device__ __forceinline__ uint32_t warp_inclusive(uint32_t v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        asm volatile("{\n\t.reg .b32 t;\n\t.reg .pred p;\n\tshfl.sync.up.b32 t|p, %0, %1, 0, -1;\n\t@p add.u32 %0, %0, t;\n\t}"
                     : "+r"(v)
                     : "r"(o));
    return v;
}

// Copies a run of rows (len bytes, a multiple of 8) from 4-byte aligned src to any byte address
// dst: one aligned word per lane, built from two words and a funnel shift; the unaligned head and tail
// bytes singly.
__device__ __forceinline__ void copy_rows(uint8_t *dst, const uint8_t *src, uint32_t len, int lane) {
    const uint32_t head = (0u - (uint32_t)reinterpret_cast<uintptr_t>(dst)) & 3u;
    const uint32_t tail = (len - head) & 3u;
    if ((uint32_t)lane < head) dst[lane] = src[lane];
    if ((uint32_t)lane < tail) dst[len - tail + lane] = src[len - tail + lane];
    const uint32_t words = (len - head) >> 2, sb = head * 8u;
    const uint32_t *s = reinterpret_cast<const uint32_t *>(src) + lane;
    uint32_t *d = reinterpret_cast<uint32_t *>(dst + head) + lane;
#pragma unroll 4
    for (uint32_t j = (uint32_t)lane; j < words; j += 32u, s += 32, d += 32) *d = __funnelshift_r(s[0], s[1], sb);
}

// The rows of up to 32 planes (Sec. 3.3) from their slots into the record.  `rows`: the planes that
// exist (low bits), `dense` the dense ones among them; `cur`: record position of the top plane's row,
// moved to the end of the last.  Plane p's row is in slot 31 - p.
// Sparse rows go four at a time: their nibbles in the bytes of one word, so one shuffle serves four
// bitmaps, and their byte counts in the bytes of another, so one prefix scan serves four rows (a
// row has at most 128 non-zero bytes); what used to be a chain of ballots and reductions per row
// has four rows' work to overlap.  Then runs of dense rows are copied.  `line` is where plane 0's row
// would lie if every row below the sparse ones met so far were dense: plane q's row is at
// line - row_bytes * q, and a sparse row moves it by its length less row_bytes.
__device__ __forceinline__ void emit_rows(uint8_t *rec, const uint8_t *slots, uint32_t &cur, uint32_t rows,
                                          uint32_t dense, uint32_t row_bytes, uint32_t bm_bytes, uint32_t seltab, int lane) {
    const bool maps = !(lane & 1) && (uint32_t)lane < 2u * bm_bytes;      // this lane stores a bitmap byte
    // through a reduction, so that the mask and the totals are known to be the warp's: the arithmetic on
    // them leaves the integer pipe (2^26 FP32 211.5 -> 208.2 us, 2^24 FP16 83.8 -> 82.6, FP64 -0.3 %; the
    // addresses as well: 1 % slower)
    uint32_t sparse = __reduce_or_sync(kFull, rows & ~dense);
    const uint32_t step = bm_bytes - row_bytes;
    uint32_t line = cur + row_bytes * ((uint32_t)__popc(rows) - 1u), mine = line;       // mine: for this lane's plane
    uint8_t *bm = rec + (lane >> 1);
#pragma unroll 1
    while (sparse) {
        uint32_t p[4], x[4], nibs = 0;
        bool have[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            have[i] = sparse != 0u;
            p[i] = have[i] ? 31u - (uint32_t)__clz((int)sparse) : 0u;
            sparse &= ~(1u << p[i]);
            x[i] = *reinterpret_cast<const uint32_t *>(slots + 128u * (31u - p[i]) + 4u * lane);
            if (i > 0) x[i] = have[i] ? x[i] : 0u;
            const uint32_t n = nz_nibble128(x[i]);
            nibs = i == 0 ? n >> 7 : nibs + (n << (8 * i - 7));
        }
        uint32_t c = nibs - ((nibs >> 1) & 0x05050505u);             // set bits of every nibble
        c = (c & 0x03030303u) + ((c >> 2) & 0x03030303u);
        const uint32_t incl = warp_inclusive(c);
        const uint32_t tot = __reduce_add_sync(kFull, c), excl = incl - c;
        const uint32_t pair = (nibs << 4) | __shfl_down_sync(kFull, nibs, 1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t at = line - row_bytes * p[i];
            if (have[i]) line += step + ((tot >> (8 * i)) & 255u);
            if ((uint32_t)lane < p[i]) mine = line;
            if (have[i] && maps) bm[at] = (uint8_t)(pair >> (8 * i));
            const uint32_t packed = __byte_perm(x[i], 0u, __shfl_sync(kFull, seltab, (int)(nibs >> (8 * i))));
            uint8_t *q = rec + at + bm_bytes + ((excl >> (8 * i)) & 255u);
            const uint32_t n = (c >> (8 * i)) & 7u;
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (n > (uint32_t)t) q[t] = (uint8_t)(packed >> (8 * t));
        }
    }
    cur = line + row_bytes;
    const uint32_t place = mine - row_bytes * (uint32_t)lane;              // of dense plane `lane`
    uint32_t dm = dense;
#pragma unroll 1
    while (dm) {
        // a run of dense rows p, p-1, ..., q: contiguous in the slots when rows are 128 bytes long
        const uint32_t p = 31u - (uint32_t)__clz((int)dm);
        const uint32_t holes = ~dm & ((2u << p) - 1u);
        const uint32_t q = row_bytes == 128u ? 32u - (uint32_t)__clz((int)holes) : p;
        copy_rows(rec + __shfl_sync(kFull, place, (int)p), slots + 128u * (31u - p), (p - q + 1u) * row_bytes, lane);
        dm &= (1u << q) - 1u;
    }
}

// value k of this lane from the swizzled staging buffer
template <int D>
__device__ __forceinline__ typename Traits<D>::U lane_value(const uint8_t *buf, int lane, int k) {
    using U = typename Traits<D>::U;
    constexpr int UN = Traits<D>::UNITS;
    constexpr int PER = 16 / Traits<D>::S;
    return *reinterpret_cast<const U *>(buf + (lane * UN + unit_swizzle<D>(lane, k / PER)) * 16 + (k % PER) * Traits<D>::S);
}

// A tail chunk's staged values past the m-th repeat it: Eq. 5's pad columns (R11) are zero because
// their G are equal, and every test over 1024 values answers as over the m.
template <int D>
__device__ __forceinline__ void pad_values(uint8_t *buf, uint32_t m, int lane) {
    if (m >= 1024u) return;
    using U = typename Traits<D>::U;
    const U last = read_elem<D>(buf, m - 1u);
#pragma unroll 1
    for (uint32_t e = m + (uint32_t)lane; e < 1024u; e += 32) *reinterpret_cast<U *>(buf + phys_elem_byte<D>(e)) = last;
    __syncwarp();
}

// Every value of the chunk passes Alg. 2's test at a; the values are re-read from the staging
// buffer (index >= m: not a value).  A failing decimal place usually fails on every lane's
// first value already, so those 32 are tested first.
template <int D>
__device__ __forceinline__ bool all_pass(const uint8_t *buf, int lane, uint32_t m, typename Traits<D>::U vx,
                                         int a) {
    const bool has0 = 32u * lane < m;
    if (!__all_sync(kFull, !has0 || q_test(lane_value<D>(buf, lane, 0), a))) return false;
    bool ok = q_test(vx, a);
#pragma unroll 4
    for (int k = 1; k < 32; ++k)
        if (32u * lane + k < m) ok &= q_test(lane_value<D>(buf, lane, k), a);
    return __all_sync(kFull, ok);
}

// Test and g of one value at decimal place a together (Eq. 4, Case 1): g = round(v 10^a) from one
// 64-bit high product, then the exact distance |m 5^a - g 2^F| against 5^a / 2, modulo 2^64 (exact
// while F <= 62, since g lies within one of v 10^a).  Below a power of two the interval is half as
// wide, which changes nothing: there m 5^a = 2^52 5^a, and its distance to a multiple of 2^F is 0 or
// at least 2^52 > 5^a / 2.  Other values but +0 (which passes, and whose g is 0 as the shift says) set
// `slow` and are left to q_test, which stays out of the loop over the values.
struct Case1At {                                  // constants of a decimal place
    uint64_t p5, norm;                            // 5^a, 5^a with its top bit at bit 63
    int f0, sh0;                                  // F = f0 - exponent field, shift = F + sh0
};
__device__ __forceinline__ Case1At case1_at(int a) {
    return {FALCON_POW5[a], FALCON_POW5_NORM[a], 1075 - a, 10 - (int)FALCON_LOG2_POW5[a]};
}
__device__ __forceinline__ uint64_t test_g(uint64_t u, const Case1At &c, bool &ok, uint32_t &slow) {
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const int F = c.f0 - (int)((hi >> 20) & 0x7FFu);
    const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
    const uint64_t N = (shr_clamp64(__umul64hi(m << 11, c.norm), (uint32_t)(F + c.sh0 - 1)) + 1ull) >> 1;
    if (F > 62 || F <= 0) {
        slow |= (hi << 1) | lo;
    } else {
        const uint64_t lim = c.p5 >> 1;
        ok &= (m * c.p5 - (N << F)) + lim <= 2u * lim;
    }
    return (hi >> 31) ? 0ull - N : N;
}
// The same for |g| < 10^8 and 5^a < 2^31.  The product is scaled by 2^t so that F + t >= 32 (X < 10^8
// and m >= 2^52 give F >= 26 + 2.3 a), which leaves g 2^F out of its low word; modulo 2^64 it is exact
// while F + t <= 64: g then is the only multiple in reach.  (With q_test out of line, 40 M decimal values
// at block 1025 compress in 367 us against 389 with both tests per value in 64-bit shifts; q_test in
// line again: 379.)
struct TestNarrow {
    Case1Narrow g;
    uint32_t p5, lim;                             // 2^t 5^a, 2^t floor(5^a / 2)
    int c;                                        // F + t - 32 = c - exponent field
};
__device__ __forceinline__ TestNarrow test_narrow_of(int a) {
    const int t = a < 3 ? 6 : 0;
    const uint32_t p5 = (uint32_t)FALCON_POW5[a];
    return {case1_narrow_of(a), p5 << t, (p5 >> 1) << t, 1075 - a + t - 32};
}
__device__ __forceinline__ uint64_t test_g(uint64_t u, const TestNarrow &q, bool &ok, uint32_t &slow) {
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const uint32_t N = case1_n_narrow(hi, lo, q.g);
    const uint32_t f = (uint32_t)(q.c - (int)((hi >> 20) & 0x7FFu));
    const uint64_t P = (uint64_t)lo * q.p5 + ((uint64_t)(((hi & 0xFFFFFu) | 0x100000u) * q.p5 - shl_clamp(N, f)) << 32);
    if (f > 32u) slow |= (hi << 1) | lo;
    else ok &= P + q.lim <= 2u * q.lim;
    // a negative value with g = 0 has failed
    const uint32_t s = (uint32_t)((int32_t)hi >> 31);
    return ((uint64_t)s << 32) | ((N ^ s) - s);
}
// FP32: the round trip |m 5^a - g 2^F| <= 5^a / 2 as in q_test, on the normalised product m 2^8 5^a
// 2^(31-d) that g comes from (g 2^F scaled alike is a multiple of 2^32, and exact modulo 2^64 up to
// 2^64: past that, |v 10^a| < 1/2 and only +0 passes).
struct TestF32 {
    Case1F32 g;
    uint64_t lim;                                 // floor(5^a / 2) scaled alike
};
__device__ __forceinline__ TestF32 test_f32_of(int a) {
    const Case1F32 g = case1_f32_of(a);
    return {g, (uint64_t)(g.p5 >> 1) << (39 - (int)FALCON_LOG2_POW5[a])};
}
__device__ __forceinline__ uint32_t test_g(uint32_t u, const TestF32 &q, bool &ok) {
    const uint64_t P = (uint64_t)((u << 8) | 0x80000000u) * q.g.norm;
    const uint32_t sh = (uint32_t)(q.g.c - (int)((u >> 23) & 0xFFu));        // the shift - 1, as in case1_n
    const uint32_t N = (shr_clamp((uint32_t)(P >> 32), sh) + 1u) >> 1;
    const bool near = P - ((uint64_t)shl_clamp(N, sh + 1u) << 32) + q.lim <= 2u * q.lim;
    ok &= (near && sh < 32u) || (u << 1) == 0u;
    const uint32_t s = (uint32_t)((int32_t)u >> 31);
    return (N ^ s) - s;
}
__device__ __forceinline__ uint16_t test_g(uint16_t u, const Scale16 &q, bool &ok) {
    bool rt;
    (void)alg2_step_f16(u, q, rt);
    ok &= rt;
    return case1_g(u, q);
}

// FP32 chunks at beta_hat = 7 (R14) and FP16 chunks at beta_hat = 3 (R18): Alg. 2, value by
// value, stops at the first decimal place where eps <= mu passes, and if the round trip fails
// there the value is an exception.  That can happen below a value's own decimal place k only if
// |v| 10^k >= 2^(p-1) / 1.5 (p = 24 or 11 significand bits): with d / 10^k its shortest decimal,
// v 10^a (a < k) lies at least 10^-(k-a) - |v| 10^a 2^-p from every integer, more than
// mu = |v 10^a| 2^-(p-1) below that bound (checked exhaustively over every decimal below it).
// k <= alpha, so a value can stop early only if |v| 10^alpha reaches the bound.  FP32 tests
// 3 |v| 10^alpha >= 2^23 (half the bound, as a margin: the bound was checked exhaustively only
// up to that point); FP16 tests the bound itself, 3 |v| 10^alpha >= 2^11, checked over all
// 65,536 patterns.  Only those values go through Alg. 2, and none when v_max is below.
__device__ __forceinline__ bool may_stop_early(uint32_t u, int a) {
    const uint32_t au = u & 0x7FFFFFFFu;
    if (au == 0) return false;
    if (au < 0x00800000u) return true;          // subnormal: take the full test
    const int E = (int)(au >> 23) - 150;
    const uint64_t p = 3ull * ((au & 0x007FFFFFu) | 0x00800000u) * FALCON_POW5[a];   // < 2^50
    const int s = 23 - E - a;                    // 3 m 5^a 2^(E+a) >= 2^23  <=>  p >= 2^s
    return s <= 0 || (s < 50 && p >= (1ull << s));
}
__device__ __forceinline__ bool may_stop_early(uint16_t u, int a) {
    const uint32_t au = u & 0x7FFFu;
    if (au == 0) return false;
    if (au < 0x0400u) return true;
    const int E = (int)(au >> 10) - 25;
    const uint32_t p = 3u * ((au & 0x3FFu) | 0x400u) * (uint32_t)FALCON_POW5[a];     // < 2^22
    const int s = 11 - E - a;                    // 3 m 5^a 2^(E+a) >= 2^11  <=>  p >= 2^s
    return s <= 0 || (s < 32 && p >= (1u << s));
}
// A magnitude no larger than the smallest that may stop early at a (chunks here hold no subnormals), so
// that a unit's largest magnitude tells whether any of its values is to be looked at: the bound over
// 3 10^a, rounded down.  (may_stop_early of every value instead: 2^24 FP16 segments 83.0 us against 78.7,
// 2^25 FP32 decimals 212.6 against 206.6, 2^25 FP32 walk 144.6 against 142.8.)
template <int D> __device__ __forceinline__ uint32_t early_floor(int a) {
    const float p10 = (float)(FALCON_POW5[a] << a);             // exact: a <= 10
    if constexpr (D == kD32) return __float_as_uint(__fdiv_rd(2796202.5f, p10));          // below 2^23 / 3
    else return __half_as_ushort(__float2half_rd(__fdiv_rd(682.5f, p10)));                // below 2^11 / 3
}
__device__ __forceinline__ int first_pass(uint32_t u, int atop) { return first_pass_f32(u, atop); }
__device__ __forceinline__ int first_pass(uint16_t u, int atop) { return first_pass_f16(u, atop); }

// Classification of a chunk's magnitudes: FP64 by a key that keeps the top 25 bits of the high word
// and carries the value's index below, FP32 and FP16 by the magnitude itself.
template <int D> struct Mag {
    using U = typename Traits<D>::U;
    static constexpr U ABS = (U)((U)~(U)0 >> 1);                 // every bit but the sign
    static constexpr uint32_t kExpAll = D == kD64 ? 0x7FF00000u : (D == kD32 ? 0x7F800000u : 0x7C00u);
    static constexpr uint32_t kExpOne = D == kD64 ? 0x00100000u : (D == kD32 ? 0x00800000u : 0x0400u);
    static __device__ __forceinline__ uint32_t key(U u, uint32_t k) {
        if constexpr (D == kD64) return ((uint32_t)(u >> 32) & 0x7FFFFFC0u) | k;
        else return (uint32_t)(u & ABS);
    }
};

// q_test of a 16-byte unit's values, out of the loop over them (instruction fetch)
__device__ __noinline__ bool unit_pass(uint64_t x, uint64_t y, int a) { return q_test(x, a) && q_test(y, a); }

// whether Alg. 2 stops early on one of the first `count` values of a 16-byte unit (those from floor_bits
// on can)
template <int D> __device__ __noinline__ bool unit_stops(uint4 w, int a, uint32_t floor_bits, uint32_t count) {
    union { uint4 w; typename Traits<D>::U e[16 / Traits<D>::S]; } x;
    x.w = w;
    bool early = false;
#pragma unroll
    for (int k = 0; k < 16 / Traits<D>::S; ++k)
        if ((uint32_t)k < count && (uint32_t)(x.e[k] & Mag<D>::ABS) >= floor_bits) early |= first_pass(x.e[k], a) < 0;
    return early;
}

// all_pass that leaves every value's g in the staging buffer in its place (rolled: small code).
// kNarrow (FP64): |v 10^a| < 10^8 for every value.  With `watch` (FP32, FP16 at the largest beta_hat) no
// value may stop early either; that test reads the chunk's own values, not a tail's
// padding (one FP32 value of seven digits and its 1023 copies: 37 us for the call, 14 so).
template <int D, bool kNarrow = false>
__device__ __forceinline__ bool pass_to_g(uint8_t *buf, int lane, uint32_t m, int a, bool watch) {
    using U = typename Traits<D>::U;
    constexpr int UN = Traits<D>::UNITS, PER = 32 / UN;
    bool ok = true;
    uint32_t slow = 0;
    Case1At c{};
    if constexpr (D == kD64 && !kNarrow) c = case1_at(a);
    TestNarrow cn{};
    if constexpr (kNarrow) cn = test_narrow_of(a);
    TestF32 cf{};
    if constexpr (D == kD32) cf = test_f32_of(a);
    Scale16 ch{};
    if constexpr (D == kD16) ch = scale16_of(a);
    uint32_t floor_bits = 0;
    if constexpr (D != kD64) floor_bits = early_floor<D>(a);
    auto one = [&](U u) {
        if constexpr (kNarrow) return test_g(u, cn, ok, slow);
        else if constexpr (D == kD64) return test_g(u, c, ok, slow);
        else if constexpr (D == kD32) return test_g(u, cf, ok);
        else return test_g(u, ch, ok);
    };
    if (m > 1024u && lane == 31) {
        U *e = reinterpret_cast<U *>(buf + phys_elem_byte<D>(1024));
        const U x = *e;
        *e = one(x);
        if constexpr (D == kD64) {
            if (slow) ok &= unit_pass(x, x, a);
        } else {
            if (watch && (uint32_t)(x & Mag<D>::ABS) >= floor_bits) ok &= first_pass(x, a) >= 0;
        }
    }
#pragma unroll 1
    for (int u = 0; u < UN; ++u) {
        uint4 *q = reinterpret_cast<uint4 *>(buf + (lane * UN + unit_swizzle<D>(lane, u)) * 16);
        union { uint4 w; U e[PER]; } x, g;
        x.w = *q;
        slow = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) g.e[k] = one(x.e[k]);
        *q = g.w;
        const uint32_t first = 32u * (uint32_t)lane + (uint32_t)(u * PER);        // the unit's first value
        if constexpr (D == kD64) {
            if (slow) ok &= unit_pass(x.e[0], x.e[1], a);
        } else if (watch && first < m) {
            uint32_t top = 0;
#pragma unroll
            for (int k = 0; k < PER; ++k) top = max(top, (uint32_t)(x.e[k] & Mag<D>::ABS));
            if (top >= floor_bits) ok &= !unit_stops<D>(x.w, a, floor_bits, m - first);
        }
        if (!__all_sync(kFull, ok)) return false;
    }
    return true;
}

// alpha_max is the smallest a in [0, atop] at which every value passes the round-trip test (none: Case
// 2).  For chunks of valid values the predicate is monotone in a (Thm 4 with Thm 3), and its smallest
// true point is the largest decimal place of the values; a failure at atop means some value is an
// exception or needs alpha > atop.  A lower bound: each lane's first value is tested at atop (a failure
// settles Case 2: -1), then its own decimal place is found, and the warp's maximum is returned.  For most
// chunks it is the answer, which the caller's test of every value confirms; otherwise alpha_above goes on.
template <int D>
__device__ __forceinline__ int alpha_bound(const uint8_t *buf, int lane, uint32_t m, int atop) {
    using U = typename Traits<D>::U;
    const U v0 = 32u * lane < m ? lane_value<D>(buf, lane, 0) : (U)0;
    if (!__all_sync(kFull, q_test(v0, atop))) return -1;
    int a0 = 0;
#pragma unroll 1
    while (a0 < atop && !q_test(v0, a0)) ++a0;
    return (int)__reduce_max_sync(kFull, (uint32_t)a0);
}
// the answer above a lower bound that failed (test atop, then bisect), or -1
template <int D>
__device__ __forceinline__ int alpha_above(const uint8_t *buf, int lane, uint32_t m, typename Traits<D>::U vx,
                                           int lb, int atop) {
    if (lb >= atop) return -1;
    int lo = lb + 1, hi = atop;                 // the answer, if any, lies in [lo, hi]
    bool hi_ok = false;                         // all_pass(hi) is known to hold
    int a = atop;
#pragma unroll 1
    for (;;) {
        const bool ok = all_pass<D>(buf, lane, m, vx, a);
        if (ok) {
            hi = a;
            hi_ok = true;
        } else {
            if (a == atop) return -1;
            lo = a + 1;
        }
        if (hi_ok && lo >= hi) return hi;
        a = (lo + hi) >> 1;                     // lo <= a < hi once atop has passed
    }
}

// Fal._Elf's decimal place of one value (Sec. 1's trial and error, ablation of Sec. 5.4.2):
// the first a with v (x) 10^a integral, a <= 22 and a + floor(log10|v|) + 1 <= 15 (FP32: 10
// and 7), else -1 (exception).  The products are IEEE multiplies, as the method defines.
__device__ __forceinline__ int elf_dp(uint64_t u) {
    const uint64_t au = u & 0x7FFFFFFFFFFFFFFFull;
    if (au == 0) return 0;
    if (is_special(u) || !log10_in_range(au)) return -1;
    const int atop = min(22, 14 - floor_log10(au));
    const double v = __longlong_as_double((long long)u);
    for (int a = 0; a <= atop; ++a) {
        const double x = __dmul_rn(v, __longlong_as_double((long long)FALCON_P10_F64[a - FALCON_P10_F64_LO]));
        if (x == floor(x)) return a;
    }
    return -1;
}
__device__ __forceinline__ int elf_dp(uint32_t u) {
    const uint32_t au = u & 0x7FFFFFFFu;
    if (au == 0) return 0;
    if (is_special(u) || !log10_in_range(au)) return -1;
    const int atop = min(10, 6 - floor_log10(au));
    const float v = __uint_as_float(u);
    for (int a = 0; a <= atop; ++a) {
        const float x = __fmul_rn(v, __uint_as_float(FALCON_P10_F32[a - FALCON_P10_F32_LO]));
        if (x == floorf(x)) return a;
    }
    return -1;
}
__device__ __forceinline__ int elf_dp(uint16_t u) {      // binary16: products rounded to binary16
    const uint32_t au = u & 0x7FFFu;
    if (au == 0) return 0;
    if (is_special(u)) return -1;
    const int atop = min(4, 2 - floor_log10((uint16_t)au));
    const float v = __half2float(__ushort_as_half(u));
    for (int a = 0; a <= atop; ++a) {
        // the product of two binary16 values is exact in FP32, so one rounding gives fl16
        const float x = __half2float(__float2half_rn(v * (float)(FALCON_POW5[a] << a)));
        if (x == floorf(x)) return a;
    }
    return -1;
}

// Fal._Elf: alpha_max = the largest of the values' Elf decimal places, then Eq. 4's bounds and
// the R6 round trip at alpha_max, as for Falcon; -1 means Case 2.  Out of line (an ablation).
template <int D>
__device__ __noinline__ int alpha_elf(const uint8_t *buf, int lane, uint32_t m, typename Traits<D>::U vx,
                                      bool has_vx, int e_max) {
    using T = Traits<D>;
    int amax = has_vx ? elf_dp(vx) : 0;
    bool bad = amax < 0;
#pragma unroll 1
    for (int k = 0; k < 32; ++k) {
        if (32u * lane + k < m) {
            const int a = elf_dp(lane_value<D>(buf, lane, k));
            bad |= a < 0;
            amax = a > amax ? a : amax;
        }
    }
    if (__any_sync(kFull, bad)) return -1;
    amax = (int)__reduce_max_sync(kFull, (uint32_t)amax);
    if (amax > T::A_MAX || amax + e_max + 1 > T::B_MAX) return -1;
    return all_pass<D>(buf, lane, m, vx, amax) ? amax : -1;
}

// Case 1's alpha_max of a chunk that may be Case 1 (no special value, the test value passes at
// atop), or -1.  On success the staging buffer holds G (Eq. 4) in place of the values, otherwise
// the values.  Out of line, over the staged values: many workloads' chunks never get here, and its code
// stays out of the others' instruction stream.
// vmax: the chunk's largest magnitude; own: this lane's (FP32 and FP16 only).
template <int D>
__device__ __noinline__ int case1_alpha(const uint8_t *src, uint8_t *buf, int lane, uint32_t m, int e_max, int atop,
                                           typename Traits<D>::U vmax, uint32_t own, bool elf) {
    using T = Traits<D>;
    using U = typename T::U;
    const bool has_vx = m > 1024u && lane == 31;
    const U vx = has_vx ? read_elem<D>(buf, 1024) : (U)0;
    auto restage = [&]() {                        // the values again
        __syncwarp();
        stage_values_async<D>(src, m, buf, lane);
        cp_async_commit();
        cp_async_wait_none();
        __syncwarp();
        pad_values<D>(buf, m, lane);
    };
    // FP32 (R14), FP16 (R18): below beta_hat = B_MAX no value can stop early, so Alg. 2 value by value
    // gives the same alpha_max.  At B_MAX (a = atop) a chunk with an early stop is Case 2, as one with a
    // failing value is; in data full of them every lane's largest value tells most chunks (1023 FP32
    // decimals of seven digits: 43 us for the call, 12 so).  FP64: no value can stop (Thm 4).
    auto pass = [&](int a) {
        bool watch = false;
        if constexpr (D != kD64) {
            watch = !elf && a + e_max + 1 == T::B_MAX && may_stop_early(vmax, a);
            if (watch && __any_sync(kFull, first_pass((U)own, a) < 0)) return false;
        }
        if constexpr (D == kD64) {
            if (a + e_max + 1 <= kNarrowBeta && a <= 13) return pass_to_g<D, true>(buf, lane, m, a, false);
        }
        return pass_to_g<D>(buf, lane, m, a, watch);
    };
    int alpha = elf ? alpha_elf<D>(buf, lane, m, vx, has_vx, e_max) : alpha_bound<D>(buf, lane, m, atop);
    if (alpha < 0) return -1;
    bool ok = pass(alpha);
    if (!ok) {
        restage();
        alpha = alpha_above<D>(buf, lane, m, vx, alpha, atop);
        if (alpha < 0) return -1;
        ok = pass(alpha);
    }
    if (D != kD64 && !ok) {                       // every value passes, but some value stops early
        restage();
        return -1;
    }
    return alpha;
}

// Case decision (Eq. 4) of a chunk whose keys have maximum `top` (kmax: this lane's) and, if
// `low`, some value with a zero exponent field.  Returns alpha_max | beta_hat << 8, alpha_max = 31
// in Case 2; the staging buffer holds G on a Case 1 return, the values otherwise.
constexpr int kCase2 = 31;
// the value a lane's FP64 key stands for
template <int D>
__device__ __forceinline__ typename Traits<D>::U lane_max(const uint8_t *buf, int lane, uint32_t key) {
    return read_elem<D>(buf, 32u * (uint32_t)lane + (key & 63u)) & Mag<D>::ABS;
}
template <int D>
__device__ __forceinline__ int case_decision(const uint8_t *src, uint8_t *buf, int lane, uint32_t m, uint32_t kmax,
                                             uint32_t top, bool low, bool elf) {
    using T = Traits<D>;
    using U = typename T::U;
    constexpr U ABS = Mag<D>::ABS;
    constexpr int kNone = kCase2 | (T::B_SENT << 8);
    if (low) {                                    // +0 or a special value (-0, subnormal)
        constexpr int PER = 16 / T::S;
        bool s = m > 1024u && lane == 31 && is_special(read_elem<D>(buf, 1024));
#pragma unroll 2
        for (int u = 0; u < T::UNITS; ++u) {
            union { uint4 w; U e[PER]; } x;
            x.w = *reinterpret_cast<const uint4 *>(buf + (lane * T::UNITS + unit_swizzle<D>(lane, u)) * 16);
#pragma unroll
            for (int k = 0; k < PER; ++k) s |= Mag<D>::key(x.e[k], 0) < Mag<D>::kExpOne && x.e[k] != 0;
        }
        if (__any_sync(kFull, s)) return kNone;
    }
    // the largest magnitude (FP64: one that shares its key's top bits)
    U vmax;
    if constexpr (D == kD64) {
        const uint32_t owner = __ffs(__ballot_sync(kFull, kmax == top)) - 1u;
        vmax = top < 64u ? 0 : read_elem<D>(buf, 32u * owner + (top & 63u)) & ABS;
    } else {
        vmax = (U)top;
    }
    if (vmax == 0) return 0;                      // every value is +0, and its G
    if (!log10_in_range(vmax)) return kNone;
    int e_max = floor_log10(vmax);
    if constexpr (D == kD64) {
        // a power of ten between vmax and a larger value with the same key bits?
        const uint32_t p = (uint32_t)(FALCON_P10_F64[e_max + 1 - FALCON_P10_F64_LO] >> 32);
        if (((p ^ top) & 0x7FFFFFC0u) == 0) {
            U x = m > 1024u ? read_elem<D>(buf, 1024) & ABS : (U)0;
#pragma unroll 4
            for (int k = 0; k < 32; ++k) x = max(x, (U)(lane_value<D>(buf, lane, k) & ABS));
            e_max = floor_log10(warp_max_x(x));
        }
    }
    const int atop = min(T::A_MAX, T::B_MAX - 1 - e_max);
    // quick rejection: Alg. 2's round trip on every lane's largest magnitude first (the test reads only
    // |v|).  One outlier that happens to pass does not send its chunk through the search: a few such
    // chunks, each worth a hundred others, made a launch's tail (2^24 values: 55 us of analysis against 33).
    if (!elf) {
        U own;
        if constexpr (D == kD64) own = lane_max<D>(buf, lane, kmax);
        else own = (U)kmax;
        if (atop < 0 || !__all_sync(kFull, q_test(own, atop))) return kNone;
    }
    const int alpha = case1_alpha<D>(src, buf, lane, m, e_max, atop, vmax, D == kD64 ? 0u : kmax, elf);
    return alpha < 0 ? kNone : alpha | ((alpha + e_max + 1) << 8);
}

__device__ __forceinline__ uint32_t values_in(const Job &job, uint64_t c) {
    const uint64_t left = job.n - c * (uint64_t)job.block;
    return (uint32_t)(left < job.block ? left : job.block);
}

// Starts the copy of chunk c's values; kD: the kind, or -1 for the job's own.
template <int kD>
__device__ __forceinline__ void issue_chunk(const Job &job, uint64_t c, uint8_t *buf, int lane) {
    const uint64_t first = c * (uint64_t)job.block;
    const uint32_t m = values_in(job, c);
    if (kD == kD64 || (kD < 0 && job.dtype == 0)) stage_values_async<kD64>(job.in + first * 8u, m, buf, lane);
    else if (kD == kD32 || (kD < 0 && job.dtype == 1)) stage_values_async<kD32>(job.in + first * 4u, m, buf, lane);
    else stage_values_async<kD16>(job.in + first * 2u, m, buf, lane);
}

// Workspace words of a job (job.flags), written by the analysis launch:
//   flags[c]            alpha byte (5 bits) | beta_hat (5) | w (7), in bits 47..63; the offsets launch
//                       adds the record's position (from the first record) below;
//   flags[nchunks + c]  the dense-row mask (bit p: plane p is stored dense).
constexpr int kMetaShift = 47;
static_assert(kMetaShift == kOffsetBits, "the offsets launch fills the bits below");

__device__ __forceinline__ unsigned long long pack_meta(int alpha_byte, int beta_hat, int w) {
    return (unsigned long long)(((uint32_t)alpha_byte << 12) | ((uint32_t)beta_hat << 7) | (uint32_t)w) << kMetaShift;
}

// the sign of a delta, as a mask
__device__ __forceinline__ uint64_t sign_mask(uint64_t x) { return (uint64_t)((int64_t)x >> 63); }
__device__ __forceinline__ uint32_t sign_mask(uint32_t x) { return (uint32_t)((int32_t)x >> 31); }
__device__ __forceinline__ uint16_t sign_mask(uint16_t x) { return (uint16_t)((int32_t)(int16_t)x >> 15); }

// Launch 1, one chunk: everything up to the record size (see the file comment).  `next`
// starts the copy of the warp's next chunk into buf; it is called once, as soon as the
// staged values are no longer read (after the Case decision).
template <int D, class Next>
__device__ __forceinline__ void analyse_chunk(const Job &job, uint64_t c, uint8_t *buf, int lane, Next &&next) {
    using T = Traits<D>;
    using U = typename T::U;
    const uint32_t B = job.block;
    const uint64_t first = c * (uint64_t)B;
    const uint32_t m = (uint32_t)((job.n - first) < B ? (job.n - first) : B);

    // ---- 1. Case decision (Eq. 4) -----------------------------------------------------------
    // Three-input maxima and minima over the keys settle the special values: exponent all ones iff
    // the maximum says so; a zero exponent field (rare but for zeros) is looked at again.
    pad_values<D>(buf, m, lane);
    constexpr int UN = T::UNITS, PER = 32 / UN, GU = UN / 4;         // 16-byte units; of 8 values
    // unit GU i + u of this lane: the swizzle splits into a part for i and one for u
    const uint32_t key_bits = D == kD16 ? ((uint32_t)lane >> 1) & 3u : (uint32_t)lane & 7u;
    const uint8_t *own = buf + lane * (UN * 16);
    auto group = [&](int i) { return ((GU * (uint32_t)i) ^ (key_bits & ~(GU - 1u))) * 16u; };
    uint32_t low_unit[GU];
#pragma unroll
    for (int u = 0; u < GU; ++u) low_unit[u] = ((uint32_t)u ^ (key_bits & (GU - 1u))) * 16u;
    uint32_t kmax = 0, kmin = ~0u;
#pragma unroll 2
    for (int i = 0; i < 4; ++i) {
        const uint8_t *at = own + group(i);
#pragma unroll
        for (int u = 0; u < GU; ++u) {
            union { uint4 w; U e[PER]; } x;
            x.w = *reinterpret_cast<const uint4 *>(at + low_unit[u]);
#pragma unroll
            for (int k = 0; k < PER; k += 2) {
                const uint32_t n = (uint32_t)(8 * i + u * PER + k);
                const uint32_t a = Mag<D>::key(x.e[k], n), b = Mag<D>::key(x.e[k + 1], n + 1);
                kmax = __vimax3_u32(kmax, a, b);
                kmin = __vimin3_u32(kmin, a, b);
            }
        }
    }
    if (m > 1024u && lane == 31) {
        const uint32_t a = Mag<D>::key(read_elem<D>(buf, 1024), 32);
        kmax = max(kmax, a);
        kmin = min(kmin, a);
    }
    const uint32_t top = __reduce_max_sync(kFull, kmax);
    const bool low = __any_sync(kFull, kmin < Mag<D>::kExpOne);
    int alpha = kCase2, beta_hat = T::B_SENT;
    if (top < Mag<D>::kExpAll) {
        const int r = case_decision<D>(job.in + first * T::S, buf, lane, m, kmax, top, low, job.variant == kVariantElf);
        alpha = r & 31;
        beta_hat = r >> 8;
        __syncwarp();
    }
    const bool case1 = alpha != kCase2;

    // ---- 2. G and |Z| by 8-column groups, w ----------------------------------------------------
    // o[i]: OR of the Z of columns 8 i .. 8 i + 7; Z = (x ^ s) << 1 | (s & 1) for the delta x with
    // sign s.  One group at a time (nine values in registers, not 32).
    // From the last group to the first, so that each hands its first value's G to the one before.
    U o[4] = {0, 0, 0, 0};
    // the value after lane 31's last group: past the chunk's last value there is no further delta
    U after = (lane == 31 && m <= 1024u) ? read_elem<D>(buf, 1023) : read_elem<D>(buf, 32u * lane + 32u);
    if (!case1) after = zigzag(after);
#pragma unroll 1
    for (int i = 3; i >= 0; --i) {
        const uint8_t *at = own + group(i);
        U g[9];
#pragma unroll
        for (int u = 0; u < GU; ++u) {
            union { uint4 w; U e[PER]; } x;
            x.w = *reinterpret_cast<const uint4 *>(at + low_unit[u]);
#pragma unroll
            for (int k = 0; k < PER; ++k) g[u * PER + k] = x.e[k];
        }
        if (!case1) {
#pragma unroll
            for (int k = 0; k < 8; ++k) g[k] = zigzag(g[k]);
        }
        g[8] = after;
        after = g[0];
        uint32_t neg = 0;
        o[3] = o[2];                             // the loop is rolled: the groups move up
        o[2] = o[1];
        o[1] = o[0];
        if constexpr (D == kD64) {
            uint32_t lo = 0, hi = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint64_t x = g[k + 1] - g[k];
                const uint32_t xh = (uint32_t)(x >> 32), sg = (uint32_t)((int32_t)xh >> 31);
                lo |= (uint32_t)x ^ sg;
                hi |= xh ^ sg;
                neg |= sg;
            }
            o[0] = ((uint64_t)__funnelshift_l(lo, hi, 1) << 32) | ((lo << 1) | (neg & 1u));
        } else {
            U mag = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const U x = (U)(g[k + 1] - g[k]);
                const U sg = sign_mask(x);
                mag |= x ^ sg;
                neg |= sg;
            }
            o[0] = (U)((U)(mag << 1) | (neg & 1u));
        }
    }
    __syncwarp();
    next();                                     // the staged values have been read
    const U zor = warp_or_x((U)(o[0] | o[1] | o[2] | o[3]));
    const int w = zor ? ((D == 0) ? 64 - __clzll((long long)zor) : 32 - __clz((int)zor)) : 0;

    // ---- 4. non-zero bytes per row, without forming the bit planes ----------------------------
    // This lane's four bytes of row p cover its columns 8i .. 8i + 7 (i = 0..3); byte i is
    // non-zero iff bit p is set in o[i].  Transposed across the warp, lane p holds which lanes'
    // byte i of row p is non-zero, and four population counts give the row's total.
    const uint32_t cols = chunk_cols(m);
    const uint32_t row_bytes = cols / 8u;
    const LaneTranspose lt = lane_transpose_of(lane);
    uint32_t nz[2] = {0, 0};                    // of planes `lane` and `lane + 32`
#pragma unroll
    for (int h = 0; h < (D == kD64 ? 2 : 1); ++h) {
        if (h == 1 && w <= 32) break;
#pragma unroll
        for (int i = 0; i < 4; ++i) nz[h] += __popc(lane_transpose((uint32_t)((uint64_t)o[i] >> (32 * h)), lt));
    }

    // ---- 5. storage choice (Sec. 3.3) and record size ------------------------------------------
    // the ablations of Sec. 5.4.2 force one scheme for every row
    const bool all_sparse = job.variant == kVariantSparse, all_dense = job.variant == kVariantDense;
    uint32_t cost = 0;
    bool dense_lo = false, dense_hi = false;
    if (lane < w) {                              // plane `lane`
        const bool sparse = all_sparse || (!all_dense && (row_bytes - nz[0]) > cols / 64u);   // tie -> dense (R10)
        cost += sparse ? cols / 64u + nz[0] : row_bytes;
        dense_lo = !sparse;
    }
    if (D == 0 && lane + 32 < w) {                  // plane `lane + 32`
        const bool sparse = all_sparse || (!all_dense && (row_bytes - nz[1]) > cols / 64u);
        cost += sparse ? cols / 64u + nz[1] : row_bytes;
        dense_hi = !sparse;
    }
    const uint32_t body = __reduce_add_sync(kFull, cost);
    const uint64_t dense_mask = (uint64_t)__ballot_sync(kFull, dense_lo) |
                                ((uint64_t)__ballot_sync(kFull, dense_hi) << 32);
    const uint32_t size = 3u + T::Z1B + ((uint32_t)w + 7u) / 8u + body;
    if (lane == 0) {
        reinterpret_cast<uint32_t *>(job.out + 32)[c] = size;
        job.flags[c] = pack_meta(case1 ? alpha : T::A_SENT, beta_hat, w);
        job.flags[job.nchunks + c] = dense_mask;
    }
}

// 32 bytes (one sector) from global memory with one load, 32-byte aligned.
__device__ __forceinline__ void load32(const void *p, uint64_t (&x)[4]) {
    asm volatile("ld.global.nc.L1::no_allocate.v4.b64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(x[0]), "=l"(x[1]), "=l"(x[2]), "=l"(x[3])
                 : "l"(p));
}

// Lane reads its 32 values (indices 32 lane + k; indices >= m read as the last value) from global
// memory: 16 bytes at a time when the chunk is whole and 16-byte aligned.  A whole FP64 chunk at 8
// modulo 16 (`window`: the 16-byte units around it lie inside the input) reads the lane's 17 aligned
// units and takes the values one half later, instead of 32 loads of 8 bytes.
template <int D>
__device__ __forceinline__ void load_own(const uint8_t *src, bool window, int lane, uint32_t m,
                                         typename Traits<D>::U (&v)[32]) {
    using U = typename Traits<D>::U;
    constexpr int UN = Traits<D>::UNITS;
    constexpr int PER = 32 / UN;
    const bool al16 = (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
    if (D != kD16 && m >= 1024u && (reinterpret_cast<uintptr_t>(src) & 31u) == 0) {
        const uint8_t *mine = src + lane * (32 * Traits<D>::S);
#pragma unroll
        for (int u = 0; u < Traits<D>::S; ++u) {
            uint64_t x[4];
            load32(mine + 32 * u, x);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                if constexpr (D == kD64) {
                    v[4 * u + h] = x[h];
                } else if constexpr (D == kD32) {
                    v[8 * u + 2 * h] = (U)x[h];
                    v[8 * u + 2 * h + 1] = (U)(x[h] >> 32);
                }
            }
        }
        return;
    }
    if (m >= 1024u && al16) {
        const uint4 *q4 = reinterpret_cast<const uint4 *>(src) + lane * UN;
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            const uint4 q = __ldg(q4 + u);
            if constexpr (D == kD64) {
                v[PER * u + 0] = ((U)q.y << 32) | q.x;
                v[PER * u + 1] = ((U)q.w << 32) | q.z;
            } else if constexpr (D == kD16) {
                const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    v[PER * u + 2 * h] = (U)(w4[h] & 0xFFFFu);
                    v[PER * u + 2 * h + 1] = (U)(w4[h] >> 16);
                }
            } else {
                v[PER * u + 0] = q.x;
                v[PER * u + 1] = q.y;
                v[PER * u + 2] = q.z;
                v[PER * u + 3] = q.w;
            }
        }
    } else if (D == kD64 && window) {
        const uint4 *q4 = reinterpret_cast<const uint4 *>(src - 8) + lane * UN;
#pragma unroll
        for (int u = 0; u < UN + 1; ++u) {
            const uint4 q = __ldg(q4 + u);
            if (u > 0) v[u > 0 ? 2 * u - 1 : 0] = (U)(((uint64_t)q.y << 32) | q.x);
            if (u < UN) v[u < UN ? 2 * u : 0] = (U)(((uint64_t)q.w << 32) | q.z);
        }
    } else {
        const U *e = reinterpret_cast<const U *>(src) + 32 * lane;
        const U last = __ldg(reinterpret_cast<const U *>(src) + (m - 1u));
        const int have = (int)m - 32 * lane;
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = k < have ? __ldg(e + k) : last;
    }
}

// Asks for a chunk's values to be brought into L2 (one prefetch per 128-byte line).
__device__ __forceinline__ void prefetch_chunk(const Job &job, uint64_t c, int lane) {
    const uint64_t first = c * (uint64_t)job.block;
    const uint32_t m = (uint32_t)((job.n - first) < job.block ? (job.n - first) : job.block);
    const uint32_t s = job.dtype == 0 ? 8u : (job.dtype == 1 ? 4u : 2u);
    const uint8_t *src = job.in + first * s;
    const uint8_t *end = src + (size_t)m * s;
    for (const uint8_t *q = src + 128u * (uint32_t)lane; q < end; q += 128u * 32u)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
}

// Chunk c's values into v (the lane's 32) and vx (value 1024 of a 1025-value chunk, lane 31).
template <int D>
__device__ __forceinline__ void load_chunk(const Job &job, uint64_t c, int lane, typename Traits<D>::U (&v)[32],
                                           typename Traits<D>::U &vx) {
    using U = typename Traits<D>::U;
    const uint64_t first = c * (uint64_t)job.block;
    const uint32_t m = (uint32_t)((job.n - first) < job.block ? (job.n - first) : job.block);
    const uint8_t *src = job.in + first * Traits<D>::S;
    const bool window = D == kD64 && m >= 1024u && src - 8 >= job.in &&
                        src + (m + 1u) * 8u <= job.in + job.n * 8u && (reinterpret_cast<uintptr_t>(src) & 15u) == 8u;
    load_own<D>(src, window, lane, m, v);
    vx = (m > 1024u && lane == 31) ? __ldg(reinterpret_cast<const U *>(src) + 1024) : v[31];
}

// v[k] = f(v[k]), kStep values at a time in a rolled loop: the values rotate through the first kStep
// places.  Twice the moves and an eighth of the code; see emit_chunk.
template <int kStep, class U, class F>
__device__ __forceinline__ void map_rolled(U (&v)[32], F &&f) {
#pragma unroll 1
    for (int i = 0; i < 32; i += kStep) {
        U e[kStep];
#pragma unroll
        for (int k = 0; k < kStep; ++k) e[k] = f(v[k]);
#pragma unroll
        for (int k = 0; k < 32 - kStep; ++k) v[k] = v[k + kStep];
#pragma unroll
        for (int k = 0; k < kStep; ++k) v[32 - kStep + k] = e[k];
    }
}

// Emit, one chunk: G and its deltas again (alpha and w from the analysis), their planes, and the record at
// its offset.  word / dense: the chunk's workspace words; size: its record size; rel: its record offset
// relative to the first record.
// L: the form's buffer layout.
template <int D, class L>
__device__ __forceinline__ void emit_chunk(const Job &job, uint64_t c, uint8_t *buf, uint32_t seltab, int lane,
                                           uint64_t word, uint64_t dense, uint32_t size, uint64_t rel) {
    using T = Traits<D>;
    using U = typename T::U;
    const uint32_t B = job.block;
    const uint64_t first = c * (uint64_t)B;
    const uint32_t m = (uint32_t)((job.n - first) < B ? (job.n - first) : B);
    const uint64_t data_start = 32ull + 4ull * job.nchunks;
    const uint32_t mb = (uint32_t)(word >> kMetaShift);
    const int alpha_byte = (int)(mb >> 12), beta_hat = (int)((mb >> 7) & 31u), w = (int)(mb & 127u);
    const uint64_t rec_off = data_start + rel;
    if (rec_off + size > job.out_cap) return;    // the job's first chunk reports the capacity error

    // ---- planes (Sec. 3.3) and record -----------------------------------------------------------
    // The zigzag is done on the planes: plane p of Z is plane p - 1 of the deltas XOR their sign
    // plane, plane 0 is the sign plane (one XOR per plane instead of five operations per value).
    // Half h of the deltas holds planes 32 h .. 32 h + 31; with w <= 32 every delta fits 32 bits and
    // its sign is bit 31, otherwise it is bit 63.
    const uint32_t cols = chunk_cols(m);
    const uint32_t row_bytes = cols / 8u, bm_bytes = cols / 64u;
    uint8_t *gdst = job.out + rec_off;
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(gdst) & 15u);
    const uint32_t flag_bytes = ((uint32_t)w + 7u) / 8u;
    const uint32_t hdr = 3u + T::Z1B + flag_bytes;
    constexpr int R = T::W < 32 ? T::W : 32;
    uint8_t *slots = buf + L::template slots_of<D>() - (32u - R) * 128u;      // plane p of a half: 128 (31 - p) further
    uint8_t *dst = slots + 31 * 128 + 4 * lane;                      // plane 0; plane p lies 128 p below
    uint32_t pos = sh + hdr;                      // next record byte in the buffer
    U z1;
    auto header = [&]() {
        // record header: byte `lane` (branch-free: every lane computes its byte, lanes < hdr store it)
        const int i = lane;
        const uint32_t zb = (uint32_t)((uint64_t)z1 >> ((8 * (i - 2)) & 63)) & 0xFFu;
        const uint32_t fb = (uint32_t)(dense >> ((8u * (flag_bytes - 1u - (uint32_t)(i - 3 - T::Z1B))) & 63u)) & 0xFFu;
        uint32_t byte = i < 2 + T::Z1B ? zb : ((i == 2 + T::Z1B) ? (uint32_t)w : fb);
        byte = i == 0 ? (uint32_t)alpha_byte : (i == 1 ? (uint32_t)beta_hat : byte);
        if ((uint32_t)lane < hdr) buf[sh + i] = (uint8_t)byte;
    };
    uint32_t sgn = 0;
    const bool two = D == kD64 && w > 32;
    uint32_t a[32];                               // the deltas' low words, transposed below
    // G (Eq. 4) and its deltas (Eq. 5).  FP64's two Case 1 conversions are rolled: unrolled over the 32
    // values they are 7 and 18 KB of code, and warps on chunks of both kinds waited for instructions
    // two thirds of the time (40 M decimal values at block 1025: 364 us unrolled, 320 so; the wide one alone 335).
    U v[32], vx;
    load_chunk<D>(job, c, lane, v, vx);
    if (D == kD64 && alpha_byte != T::A_SENT && beta_hat <= kNarrowBeta) {
        // Case 1 with |g| < 10^8: 32-bit arithmetic throughout (and w <= 32)
        const Case1Narrow q = case1_narrow_of(alpha_byte);
        uint32_t g[32];
        map_rolled<8>(v, [&](U u) { return (U)case1_g_narrow((uint64_t)u, q); });
#pragma unroll
        for (int k = 0; k < 32; ++k) g[k] = (uint32_t)v[k];
        const uint32_t gx = case1_g_narrow((uint64_t)vx, q);
        z1 = (U)(int64_t)(int32_t)__shfl_sync(kFull, g[0], 0);
        uint32_t nxt = __shfl_down_sync(kFull, g[0], 1);
        if (lane == 31) nxt = gx;
#pragma unroll
        for (int j = 0; j < 32; ++j) a[j] = ((j ^ 7) < 31 ? g[(j ^ 7) < 31 ? (j ^ 7) + 1 : 0] : nxt) - g[j ^ 7];
    } else {
        if (alpha_byte != T::A_SENT) {
            if constexpr (D == kD64) {
                map_rolled<4>(v, [&](U u) { return case1_g(u, alpha_byte); });
            } else {
#pragma unroll
                for (int k = 0; k < 32; ++k) v[k] = case1_g(v[k], alpha_byte);
            }
            vx = case1_g(vx, alpha_byte);
        } else {
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] = zigzag(v[k]);
            vx = zigzag(vx);
        }
        z1 = shfl_x(v[0], 0);
        U nxt = shfl_down_x(v[0], 1);
        if (lane == 31) nxt = vx;
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = (U)((k < 31 ? v[k + 1] : nxt) - v[k]);
        if constexpr (D == kD64) {
            if (two) {
#pragma unroll
                for (int j = 0; j < 32; ++j) a[j] = (uint32_t)(v[j ^ 7] >> 32);
                transpose32(a);
                sgn = a[31];
#pragma unroll
                for (int p = 0; p < 31; ++p) *reinterpret_cast<uint32_t *>(dst - (p + 1) * 128) = a[p] ^ sgn;
            }
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) a[j] = (uint32_t)v[j ^ 7];
    }
    transpose32(a);
    if (!two) sgn = a[R - 1];
    if (two) *reinterpret_cast<uint32_t *>(dst) = a[31] ^ sgn;
    auto low_planes = [&]() {
        *reinterpret_cast<uint32_t *>(dst) = sgn;
#pragma unroll
        for (int p = 0; p < R - 1; ++p) *reinterpret_cast<uint32_t *>(dst - (p + 1) * 128) = a[p] ^ sgn;
    };
    auto half_rows = [&](int h) {
        const int wh = w - 32 * h;
        emit_rows(buf, slots, pos, wh >= 32 ? ~0u : (1u << wh) - 1u, (uint32_t)(dense >> (32 * h)), row_bytes,
                  bm_bytes, seltab, lane);
        __syncwarp();
    };
    if constexpr (D == kD64) {
        if (lane == 0) bulk_wait_read();          // the previous record has left the buffer
        __syncwarp();
        header();
        // one copy of the row code for both halves (the low half's planes wait in registers): with
        // two, instruction fetch made every phase of the kernel slower (485 -> 452 us)
#pragma unroll 1
        for (int h = two ? 1 : 0; h >= 0; --h) {
            if (h == 0) low_planes();
            __syncwarp();
            half_rows(h);
        }
    } else {
        low_planes();
        if (lane == 0) bulk_wait_read();
        __syncwarp();
        header();
        half_rows(0);
    }

    // to global memory: the 16-byte units entirely inside the record with one bulk copy
    // (lane 0), the partial units at its ends (shared with the neighbouring records) bytewise
    uint8_t *gbase = gdst - sh;
    const uint32_t total = sh + size;
    const uint32_t u0 = (sh + 15u) / 16u, u1 = total / 16u;
    if (u0 >= u1) {
        for (uint32_t b = sh + (uint32_t)lane; b < total; b += 32) gbase[b] = buf[b];
    } else {
        const uint32_t head = 16u * u0 - sh, tail = total - 16u * u1;
        if ((uint32_t)lane < head) gbase[sh + lane] = buf[sh + lane];
        if ((uint32_t)lane < tail) gbase[16u * u1 + lane] = buf[16u * u1 + lane];
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
            bulk_store(gbase + 16u * u0, buf + 16u * u0, 16u * (u1 - u0));
            bulk_commit();
        }
    }
    __syncwarp();
}

// The hot kernels come in four forms by dtype: kDt = 0 (every job FP64), 1 (every job FP32),
// 3 (every job FP16) or 2 (any, per job: batches and the server).  A single-dtype form carries
// a third of the code, which the instruction caches notice, and serves a single stream, whose job
// it reads from shared memory.
constexpr int kDtF64 = 0, kDtF32 = 1, kDtMixed = 2, kDtF16 = 3;

// Single streams of at most this many chunks need no offsets launch: their emit warps read at most
// 4 KB of sizes each, one round trip, where the launch costs about 3 us.
constexpr uint64_t kDirectChunks = 1024;

}  // namespace

// Launch 1: analysis of every chunk (chunks by ticket; the next chunk is copied into
// the warp's one value buffer while the current one is finished).
template <int kDt>
__device__ __forceinline__ void analyse_loop(const Job *__restrict__ jobs, int njobs, Job single,
                                             uint64_t total_chunks, Control *ctl) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    uint8_t *wbase = smem + warp * kAnalyseWarpBytes<kDt == kDtF32 ? kD32 : (kDt == kDtF16 ? kD16 : kD64)>;
    __shared__ Job s_single;                      // the single job, read from shared memory
    if (threadIdx.x == 0) s_single = single;
    pdl_trigger();
    __syncthreads();
    constexpr bool kTable = kDt == kDtMixed;
    constexpr int kD = kTable ? -1 : (kDt == kDtF32 ? kD32 : (kDt == kDtF16 ? kD16 : kD64));
    const Tickets tickets{ctl, kTicketAnalyse, total_chunks};
    uint64_t t = tickets.first();
    if (t >= total_chunks) return;
    const Job *job = kTable ? find_job(jobs, njobs, t, lane) : &s_single;
    issue_chunk<kD>(*job, kTable ? t - job->chunk_begin : t, wbase, lane);
    cp_async_commit();
    for (;;) {
        const unsigned long long raw = tickets.draw(lane);       // the chunk after t
        uint64_t tn = total_chunks;
        const Job *jn = job;
        cp_async_wait_none();                    // the current chunk has landed
        __syncwarp();
        auto next = [&]() {
            tn = tickets.chunk(raw);
            if (tn < total_chunks) {
                if (kTable) jn = find_job(jobs, njobs, tn, lane);
                issue_chunk<kD>(kTable ? *jn : s_single, kTable ? tn - jn->chunk_begin : tn, wbase, lane);
            }
            cp_async_commit();
        };
        if constexpr (!kTable) {
            analyse_chunk<kD>(s_single, t, wbase, lane, next);
        } else {
            const uint64_t c = t - job->chunk_begin;
            if (job->dtype == 0) analyse_chunk<kD64>(*job, c, wbase, lane, next);
            else if (job->dtype == 1) analyse_chunk<kD32>(*job, c, wbase, lane, next);
            else analyse_chunk<kD16>(*job, c, wbase, lane, next);
        }
        __syncwarp();
        if (tn >= total_chunks) break;
        t = tn;
        job = jn;
    }
    cp_async_wait_none();
}

// FP32 and FP16 in 80 registers, 24 warps per SM; FP64 and the either-dtype form in 96 and 20 warps (FP64
// in 80 spills 16 bytes: 2^24 walk 104.8 us against 102.3, 40 M decimal values 367.0 against 364.8; the
// either-dtype form spills 12 bytes in 96).
template <int kDt>
__global__ void __maxnreg__(kDt == kDtF32 || kDt == kDtF16 ? 80 : 96)
analyse_kernel(const Job *__restrict__ jobs, int njobs, Job single, uint64_t total_chunks, Control *ctl) {
    analyse_loop<kDt>(jobs, njobs, single, total_chunks, ctl);
}

// Where a chunk's record starts, relative to the first record, is in its workspace word (the offsets
// launch, Sec. 3.4's size synchronisation), or, for a single stream of at most kDirectChunks chunks
// (`direct`), the sum of the sizes before it, added up here.
__device__ __forceinline__ uint64_t sizes_before(const Job &job, uint64_t c, int lane) {
    const uint32_t *sizes = reinterpret_cast<const uint32_t *>(job.out + 32);
    uint32_t part = 0;                            // at most 1024 records of 9235 bytes
#pragma unroll 4
    for (uint32_t i = 4u * (uint32_t)lane; i + 4u <= (uint32_t)c; i += 128u) {
        const uint4 q = *reinterpret_cast<const uint4 *>(sizes + i);
        part += q.x + q.y + q.z + q.w;
    }
    if ((uint32_t)lane < ((uint32_t)c & 3u)) part += sizes[((uint32_t)c & ~3u) + (uint32_t)lane];
    return __reduce_add_sync(kFull, part);
}
constexpr uint64_t kOffsetMask = (1ull << kOffsetBits) - 1ull;

// Stream header, stream length and status of one job (one warp): the length is the header, the size
// array and the records.
__device__ void finish_job(const Job &job, bool direct, int lane) {
    const uint64_t nc = job.nchunks;
    uint64_t total = 0;
    if (nc > 0) {
        total = direct ? sizes_before(job, nc - 1u, lane) : (job.flags[nc - 1u] & kOffsetMask);
        total += reinterpret_cast<const uint32_t *>(job.out + 32)[nc - 1u];
    }
    if (lane == 0) {
        const uint64_t bytes = 32ull + 4ull * nc + total;
        job.result[0] = bytes;
        job.result[1] = bytes > job.out_cap ? kErrCapacity : kOk;
        uint4 *dst = reinterpret_cast<uint4 *>(job.out);
        dst[0] = make_uint4(0x4E434C46u, 1u | (job.dtype << 8), job.block, 0u);
        dst[1] = make_uint4((uint32_t)job.n, (uint32_t)(job.n >> 32), (uint32_t)nc, (uint32_t)(nc >> 32));
    }
}

// A chunk to emit: its workspace words and record size, loaded a chunk ahead (unconditionally: a
// ticket past the last chunk reads the last chunk's, so nothing waits for the loads).
template <bool kTable, class Mask> struct EmitInfo {
    const Job *job;
    uint64_t c;                                   // chunk of the job
    unsigned long long word;
    Mask dense;                                   // 32 bits in the narrow kinds' forms
    uint32_t size;
};
template <bool kTable, class Mask>
__device__ __forceinline__ EmitInfo<kTable, Mask> load_info(const Job *jobs, int njobs, const Job &single, uint64_t t, uint64_t total_chunks,
                                                            int lane) {
    EmitInfo<kTable, Mask> e;
    t = t < total_chunks ? t : total_chunks - 1u;
    e.job = kTable ? find_job(jobs, njobs, t, lane) : &single;
    e.c = kTable ? t - e.job->chunk_begin : t;
    e.word = e.job->flags[e.c];
    e.dense = *reinterpret_cast<const Mask *>(e.job->flags + e.job->nchunks + e.c);
    e.size = reinterpret_cast<const uint32_t *>(e.job->out + 32)[e.c];
    return e;
}

// The records (chunks by ticket; the next chunk's values are prefetched into L2: FP32 loading them into
// registers during the current record left 20 warps per SM instead of 24 and took 234 us against 225).
template <bool kWide, int kDt>
__device__ __forceinline__ void emit_loop(const Job *__restrict__ jobs, int njobs, const Job &s_single,
                                          uint64_t total_chunks, bool direct, Control *ctl, uint8_t *smem) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    constexpr bool kTable = kDt == kDtMixed;
    constexpr int DL = kDt == kDtF32 ? kD32 : (kDt == kDtF16 ? kD16 : kD64);
    using L = EmitLayout<DL, kWide>;
    uint8_t *wbase = smem + warp * L::kBytes;
    const uint32_t seltab = compact_sel((uint32_t)lane & 15u);
    if (blockIdx.x == 0 && warp == 0) {          // jobs without chunks: header and length only
        if constexpr (!kTable) {
            if (s_single.nchunks == 0) finish_job(s_single, false, lane);
        } else {
            for (int j0 = 0; j0 < njobs; j0 += 32) {
                unsigned empty = __ballot_sync(kFull, j0 + lane < njobs && jobs[j0 + lane].nchunks == 0);
                while (empty) {
                    const int j = j0 + __ffs(empty) - 1;
                    empty &= empty - 1;
                    finish_job(jobs[j], false, lane);
                }
            }
        }
    }
    const Tickets tickets{ctl, kTicketEmit, total_chunks};
    uint64_t t = tickets.first();
    if (t >= total_chunks) return;
    using Mask = typename std::conditional<DL == kD64, unsigned long long, uint32_t>::type;
    auto info = load_info<kTable, Mask>(jobs, njobs, s_single, t, total_chunks, lane);
    t = tickets.chunk(tickets.draw(lane));       // the next chunk
    for (;;) {
        // the ticket after t, read at the next iteration; t's workspace words are fetched now
        const unsigned long long raw = tickets.draw(lane);
        const auto next = load_info<kTable, Mask>(jobs, njobs, s_single, t, total_chunks, lane);
        if (t < total_chunks) prefetch_chunk(*next.job, next.c, lane);
        const Job &job = *info.job;
        const bool dir = !kTable && direct;
        const uint64_t rel = dir ? sizes_before(job, info.c, lane) : (info.word & kOffsetMask);
        if (info.c == 0) finish_job(job, dir, lane);
        auto emit = [&](auto kind) {
            emit_chunk<decltype(kind)::value, L>(job, info.c, wbase, seltab, lane, info.word, info.dense, info.size, rel);
        };
        if constexpr (!kTable) emit(std::integral_constant<int, DL>{});
        else if (job.dtype == 0) emit(std::integral_constant<int, kD64>{});
        else if (job.dtype == 1) emit(std::integral_constant<int, kD32>{});
        else emit(std::integral_constant<int, kD16>{});
        __syncwarp();
        if (t >= total_chunks) break;
        t = tickets.chunk(raw);
        info = next;
    }
    if (lane == 0) bulk_wait();
}

// FP64 and either-dtype forms: 128 registers, 16 warps per SM; FP32 and FP16: 80 and 24.
template <bool kWide, int kDt>
__global__ void __maxnreg__(kDt == kDtF32 || kDt == kDtF16 ? 80 : 128)
emit_kernel(const Job *__restrict__ jobs, int njobs, Job single, uint64_t total_chunks, bool direct, Control *ctl) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ Job s_single;
    if (threadIdx.x == 0) s_single = single;
    __syncthreads();
    pdl_wait();
    emit_loop<kWide, kDt>(jobs, njobs, s_single, total_chunks, direct, ctl, smem);
}

namespace {
int persistent_grid_of(const void *kernel, int warps, int smem_bytes, int lim, uint64_t total_chunks);

template <int kDt> constexpr int kind_of() { return kDt == kDtF32 ? kD32 : (kDt == kDtF16 ? kD16 : kD64); }

// A kernel of a form with its launch shape: pointer, threads, dynamic shared memory, grid.
template <class K> struct Shape {
    K kernel;
    int threads, smem, grid;
};
template <int kDt> auto analyse_shape(uint64_t total_chunks) {
    const int w = g_cta_warps[0], smem = w * kAnalyseWarpBytes<kind_of<kDt>()>;
    auto *k = analyse_kernel<kDt>;
    return Shape<decltype(k)>{k, 32 * w, smem,
                              persistent_grid_of(reinterpret_cast<const void *>(k), w, smem, g_ctas_per_sm[0], total_chunks)};
}
template <bool kWide, int kDt> auto emit_shape(uint64_t total_chunks) {
    const int w = g_cta_warps[0], smem = w * (int)EmitLayout<kind_of<kDt>(), kWide>::kBytes;
    auto *k = emit_kernel<kWide, kDt>;
    return Shape<decltype(k)>{k, 32 * w, smem,
                              persistent_grid_of(reinterpret_cast<const void *>(k), w, smem, g_ctas_per_sm[0], total_chunks)};
}

template <bool kWide, int kDt>
cudaError_t launch_form(const Job *d_jobs, int njobs, const Job &single, uint64_t total_chunks, Control *ctl,
                        cudaStream_t stream) {
    const auto an = analyse_shape<kDt>(total_chunks);
    const auto em = emit_shape<kWide, kDt>(total_chunks);
    // the chunk tickets, unless both grids have a warp for every chunk
    if (((uint64_t)an.grid * an.threads / 32u < total_chunks || (uint64_t)em.grid * em.threads / 32u < total_chunks) &&
        cudaMemsetAsync(ctl, 0, sizeof(Control), stream) != cudaSuccess)
        return cudaGetLastError();
    if (total_chunks > 0) an.kernel<<<an.grid, an.threads, an.smem, stream>>>(d_jobs, njobs, single, total_chunks, ctl);
    // a stream of a few chunks: each emit warp adds up the sizes before its record itself
    const bool direct = d_jobs == nullptr && single.nchunks <= kDirectChunks;
    if (!direct) launch_offsets(d_jobs, njobs, single, kOffsetsOfOutput, ctl, stream);
    // the emit launch also writes the header and length of every job, chunks or none
    (void)launch_after(g_ctas_per_sm[0] == 0, em.kernel, em.grid, em.threads, em.smem, stream, d_jobs, njobs, single, total_chunks, direct, ctl);
    return cudaGetLastError();
}

// Resident CTAs per SM of a persistent kernel at one CTA shape, looked up once per (kernel,
// device, shape) under a lock (the server and the pipeline launch from several host threads).
std::mutex g_occ_mu;
std::map<std::tuple<const void *, int, int, int>, std::pair<int, int>> g_occ;   // -> (CTAs per SM, SMs)

int persistent_grid_of(const void *kernel, int warps, int smem_bytes, int lim, uint64_t total_chunks) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::pair<int, int> oc;
    {
        std::lock_guard<std::mutex> lk(g_occ_mu);
        const auto key = std::make_tuple(kernel, dev, warps, smem_bytes);
        auto it = g_occ.find(key);
        if (it == g_occ.end()) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
            int sms = 0, occ = 0;
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 32 * warps, smem_bytes);
            it = g_occ.emplace(key, std::make_pair(occ > 0 ? occ : 1, sms > 0 ? sms : 1)).first;
        } else {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
        }
        oc = it->second;
    }
    const int cached = oc.second * ((lim > 0 && lim < oc.first) ? lim : oc.first);
    const uint64_t need = (total_chunks + (uint64_t)warps - 1) / (uint64_t)warps;
    return (int)(need < (uint64_t)cached ? (need > 0 ? need : 1) : (uint64_t)cached);
}
}  // namespace

int persistent_grid_size(const void *kernel, int warps, int smem_bytes, int lim, uint64_t total_chunks) {
    return persistent_grid_of(kernel, warps, smem_bytes, lim, total_chunks);
}

cudaError_t launch_compress(const Job *d_jobs, int njobs, const Job &single, uint64_t total_chunks,
                            Control *ctl, cudaStream_t stream) {
    if (d_jobs != nullptr) return launch_form<false, kDtMixed>(d_jobs, njobs, single, total_chunks, ctl, stream);
    // the every-row-sparse ablation writes records larger than the plane slots hold
    if (single.variant == kVariantSparse) {
        if (single.dtype == 0) return launch_form<true, kDtF64>(d_jobs, njobs, single, total_chunks, ctl, stream);
        if (single.dtype == 1) return launch_form<true, kDtF32>(d_jobs, njobs, single, total_chunks, ctl, stream);
        return launch_form<true, kDtF16>(d_jobs, njobs, single, total_chunks, ctl, stream);
    }
    if (single.dtype == 0) return launch_form<false, kDtF64>(d_jobs, njobs, single, total_chunks, ctl, stream);
    if (single.dtype == 1) return launch_form<false, kDtF32>(d_jobs, njobs, single, total_chunks, ctl, stream);
    return launch_form<false, kDtF16>(d_jobs, njobs, single, total_chunks, ctl, stream);
}

}  // namespace falcon
