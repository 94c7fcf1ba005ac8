// Falcon decompression (Sec. 4 of the paper) for sm_103a: two launches per call.
//
// 1. offsets_kernel (a table's: table_offsets_kernel): the chunk-size array is read and its exclusive prefix (the chunk
//    offset array) is written to the workspace - the step Sec. 4 performs first.
// 2. decompress_kernel: persistent; each warp takes its chunks by ticket (one atomic add each; no
//    ordering constraint remains).  Each warp has one record buffer: the cp.async of its
//    next record starts as soon as the current one has been read; offsets are loaded one step
//    earlier still.  Decoding a record:
//      a. header and flags; a walk over the sparse rows' bitmaps gives every row's
//         position; sparse rows are expanded into 128-byte slots,
//      b. every plane's row is read where it lies (dense: unaligned in the record; sparse: its
//         slot), 32 planes at a time; the planes, shifted down one and XORed with plane 0, go
//         through 32x32 transposes, which gives the unzigzagged deltas at once; a warp scan gives
//         G (inverse Eq. 5), Case 1 divides by 10^alpha (correctly rounded) and Case 2 undoes the
//         zigzag of the IEEE bits (inverse Eq. 4),
//      c. whole 32-byte sectors per lane (aligned FP64) or staged, coalesced stores.
// What bounds it: integer issue and latency together (FP64 Case-1 values: ALU pipe 66 %, issue 64 % of cycles
// at 16 warps per SM; HBM 37 % on FP64 segments), and the instruction stream's length: code is kept short
// (both FP64 halves run one copy, Case 1 divides in rolled loops on the way out), which took FP64 segments
// from 310 to 288 us and Case-1 values from 304 to 191 us (40 M in 1025-value chunks).
// Reading the dense rows in place instead of copying them to a plane buffer took the kernel from 4302 to
// 2709 warp instructions per FP64 chunk and its shared memory from 17.6 to 13.7 KB per warp (12 to 16
// warps per SM).  Both launches, 2^26 segment values: FP64 419 -> 270 us, FP32 216 -> 137 us; the Case-1
// values 549 -> 170 us.  Slower, and left out: a TMA bulk copy of the record on an mbarrier (-1 %), tickets
// for groups of 4 to 8 chunks (-7 to -15 %: the window of memory in use grows with the group), more
// registers with fewer warps (144: -6 %).
// Every read of a record is bounds-checked against its size; a malformed record sets
// FALCON_ERR_CORRUPT and writes no value.
#include <algorithm>

#include "falcon.h"
#include "falcon_device.cuh"

namespace falcon {

namespace {

// Shared memory: a 144-byte row of zeros per CTA (what planes >= w read), then per warp
//   - one record at a 0..15 byte phase + 16 readable bytes (an FP64 record is at most
//     19 + 64 * 144 = 9235 bytes, an FP32 one 11 + 32 * 144 = 4619, an FP16 one 7 + 16 * 144 = 2311:
//     every row sparse without a zero byte, bitmap + 128 bytes),
//   - 128-byte slots for the expanded sparse rows of 32 planes at a time (FP64 runs its two
//     halves one after the other through the same slots), later the staging of a chunk whose
//     output is not 32-byte aligned,
//   - where each of those 32 planes' rows lies: (word address, bit shift) pairs,
//   - what the chunk's last steps need again (ChunkNote).
// Dense rows are read where they lie in the record, so no plane buffer is kept: 13.6 KB per FP64
// warp instead of 17.6 KB, 16 resident warps per SM instead of 12.
constexpr uint32_t kZeroBytes = 144;
template <int D> struct DecLayout {
    static constexpr uint32_t kBuf = D == kD64 ? 9280 : (D == kD32 ? 4672 : 2368);
    static constexpr uint32_t kRows = Traits<D>::W < 32 ? Traits<D>::W : 32;
    static constexpr uint32_t kSlots = kRows * 128;
    static constexpr uint32_t kTab = 32 * 8;
    static constexpr uint32_t kNote = kBuf + kSlots + kTab;
    static constexpr uint32_t kWarpBytes = kNote + 32;
};

// Header fields and place of the chunk being decoded, written down while its planes take the registers
// (kept in registers they were spilled, and with them the ticket in flight, which is then waited for).
struct ChunkNote {
    uint64_t c, z1;
    const Job *job;
    uint32_t alpha, beta_hat;
};
static_assert(sizeof(ChunkNote) == 32, "ChunkNote is 32 bytes of each warp's shared memory");

// The 32-bit word at any byte offset of the CTA's dynamic shared memory.
__device__ __forceinline__ uint32_t lds_any(const uint8_t *smem, uint32_t off) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(smem + (off & ~3u));
    return __funnelshift_r(w[0], w[1], off * 8u);           // the shift counts modulo 32
}
__device__ __forceinline__ uint32_t bswap(uint32_t x) { return __byte_perm(x, 0u, 0x0123); }

// Byte-permute selector that spreads a lane's compacted non-zero bytes over its four row
// bytes, by bitmap nibble n: row byte i (nibble bit 3 - i) takes the next compacted byte if
// the bit is set, else a zero byte (selector 4, the zero operand).  Lane l keeps the selector of
// nibble l & 15, so one shuffle looks it up.
__device__ __forceinline__ uint32_t expand_sel(uint32_t n) {
    uint32_t sel = 0, r = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if ((n >> (3 - i)) & 1u) sel |= (r++) << (4 * i);
        else sel |= 4u << (4 * i);
    }
    return sel;
}

// fl(fl(g) / 10^a) with IEEE FP64 operations, as the decoder defines it for any g; the hot
// path takes div_pow10_exact for |g| < 2^53 (every g an encoder writes: |g| < 10^15).
__device__ __forceinline__ double div_pow10(int64_t g, int a) {
    return __ddiv_rn(__ll2double_rn(g), __longlong_as_double((long long)FALCON_P10_F64[a - FALCON_P10_F64_LO]));
}
// fl32(fl32(g) / 10^a) by multiplication with r = fl32(10^-a) and one exact residual (Markstein, IBM
// J. Res. Dev. 34, 1990): q = fl(x r), then fl(q + (x - q 10^a) r) is the correctly rounded quotient.  No
// result is subnormal (|g| >= 1, a <= 10); checked against division for every 24-bit significand and a.
struct Div10F32 {
    float p, r;
};
__device__ __forceinline__ Div10F32 div10_f32_of(int a) {
    const float p = __uint_as_float(FALCON_P10_F32[a - FALCON_P10_F32_LO]);
    return {p, __frcp_rn(p)};
}
__device__ __forceinline__ float div_pow10(float x, const Div10F32 &d) {
    const float q = __fmul_rn(x, d.r);
    return __fmaf_rn(__fmaf_rn(-q, d.p, x), d.r, q);
}

// A chunk to decode and where its record lies.  The loads are unconditional (a ticket past the
// last chunk reads the last chunk's words), so nothing waits for them before the record is fetched.
struct Loc {
    const Job *job;
    uint64_t c;                                   // chunk of the job
    uint64_t off;                                 // record position from the stream's first record
    uint32_t size;
};

// Forms for one job (a single stream) read it from shared memory; the either-dtype form finds
// the ticket's job in the table.
template <bool kTable>
__device__ __forceinline__ Loc locate(const Job *jobs, int njobs, const Job &single, uint64_t t, uint64_t total_chunks,
                                      int lane) {
    Loc l;
    t = t < total_chunks ? t : total_chunks - 1u;
    l.job = kTable ? find_job(jobs, njobs, t, lane) : &single;
    l.c = kTable ? t - l.job->chunk_begin : t;
    l.off = l.job->flags[l.c];
    l.size = reinterpret_cast<const uint32_t *>(l.job->in + 32)[l.c];
    return l;
}

// Largest valid record of a chunk of m values: header, flags, and w = W rows of at most
// cols/64 + cols/8 bytes (a sparse row with no zero byte).
__device__ __forceinline__ uint32_t max_record(uint32_t m, uint32_t dtype) {
    const uint32_t W = dtype == 0 ? 64u : (dtype == 1 ? 32u : 16u);
    return 3u + W / 8u + W / 8u + W * (chunk_cols(m) / 8u + chunk_cols(m) / 64u);
}

// A record in (or on its way to) the warp's buffer: its chunk, size and 16-byte phase there.
struct Rec {
    const Job *job;
    uint64_t c;
    uint32_t size;
    uint32_t phase;                               // kBadRecord: its location is invalid
};
constexpr uint32_t kBadRecord = 16u;

// Starts the cp.async of a located record into rbuf.
__device__ __forceinline__ Rec issue_record(const Loc &l, uint8_t *rbuf, int lane) {
    const Job &job = *l.job;
    const uint64_t rec_off = 32ull + 4ull * job.nchunks + l.off;
    const uint64_t first = l.c * (uint64_t)job.block;
    const uint32_t size = l.size;
    const uint32_t m = (uint32_t)((job.n - first) < job.block ? (job.n - first) : job.block);
    const uint32_t z1b = job.dtype == 0 ? 8u : (job.dtype == 1 ? 4u : 2u);
    if (size < 3u + z1b || size > max_record(m, job.dtype) || rec_off + size > job.in_bytes)
        return {l.job, l.c, size, kBadRecord};
    const uint8_t *gsrc = job.in + rec_off;
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(gsrc) & 15u);
    const uint8_t *gbase = gsrc - sh;                       // >= job.in (16-byte aligned)
    const uint8_t *gend = job.in + job.in_bytes;
    const uint32_t units = (sh + size + 15u) / 16u;
    const uint32_t base = smem_addr(rbuf);
    // only the stream's last unit may reach past its end
    const uint32_t whole = gbase + 16u * units <= gend ? units : units - 1u;
#pragma unroll 4
    for (uint32_t u = lane; u < whole; u += 32) cp_async16(base + 16u * u, gbase + 16u * u);
    if (whole < units) {
        const uint32_t b = 16u * whole + (uint32_t)lane;
        if (lane < 16 && gbase + b < gend) rbuf[b] = gbase[b];
    }
    return {l.job, l.c, size, sh};
}

// Where the rows of up to 32 planes lie (Sec. 3.3).  `rows`: the planes that exist (low bits),
// `dense` the dense ones among them; `cur`: shared-memory offset of the top plane's row, moved to
// the end of the last row.  Sparse rows are walked top to bottom (each one's length is known only
// from its bitmap) and expanded into their 128-byte slots; then lane p writes plane p's place.
// Per sparse row the lane reads the 32 bitmap bits of its 8-lane group: the groups' counts meet in
// one byte-packed OR reduction, whose prefix is one multiply, and the lane's non-zero bytes are
// one unaligned word, spread by one byte permute.  No position is checked: a row takes at most
// 16 + 128 bytes, so every read stays in the record buffer whatever the bytes say, and the caller's
// size check rejects a malformed record before anything is stored.
// `line` is where plane 0's row would lie if every row below the sparse ones met so far were dense, so
// plane q's row is at line - row_bytes * q and a sparse row moves it by its length less row_bytes.
struct RowLane {                                  // per-lane constants of a chunk's row walk
    uint32_t keep;                                // bits of this lane's bitmap word that exist
    uint32_t before;                              // those of the lanes before this one
    uint32_t seltab;                              // expand_sel(lane & 15)
};
__device__ __forceinline__ void place_rows(uint8_t *smem, uint32_t slots, uint32_t tab, uint32_t &cur, uint32_t rows,
                                           uint32_t dense, uint32_t row_bytes, uint32_t bm_bytes, const RowLane &rl,
                                           int lane) {
    // bitmap word of 8 lanes as it lies in memory: byte k covers lanes 2 k (high nibble) and 2 k + 1
    const uint32_t group = (uint32_t)lane >> 3, gshift = 8u * group;
    const uint32_t nshift = 8u * (((uint32_t)lane & 7u) >> 1) + ((lane & 1) ? 0u : 4u);
    const uint32_t presel = group ? 0x443Fu + group : 0x4444u;
    const uint32_t step = bm_bytes - row_bytes;
    uint32_t sparse = rows & ~dense;
    uint32_t line = cur + row_bytes * ((uint32_t)__popc(rows) - 1u), mine = line;       // mine: for this lane's plane
    uint8_t *own = smem + slots + 4u * lane;
    // the row before: its two words, shift, selector and slot (its store waits for none of this
    // row's loads; the first iteration stores zeros where the second puts the first row)
    uint32_t w0 = 0, w1 = 0, wsh = 0, sel = 0x4444u;
    uint8_t *slot = own + 128u * (31u - (uint32_t)__clz((int)sparse));
    const bool any = sparse != 0u;
#pragma unroll 1
    while (sparse) {
        const uint32_t p = 31u - (uint32_t)__clz((int)sparse);
        sparse ^= 1u << p;
        const uint32_t at = line - row_bytes * p, b = at + 4u * group;
        const uint32_t *bw = reinterpret_cast<const uint32_t *>(smem + (b & ~3u));
        const uint32_t b0 = bw[0], b1 = bw[1];
        *reinterpret_cast<uint32_t *>(slot) = __byte_perm(__funnelshift_r(w0, w1, wsh), 0u, sel);
        const uint32_t W = __funnelshift_r(b0, b1, b * 8u) & rl.keep;
        const uint32_t incl = __reduce_or_sync(kFull, (uint32_t)__popc(W) << gshift) * 0x01010101u;
        line += step + (incl >> 24);              // at most 128
        const uint32_t q = at + bm_bytes + __byte_perm(incl, 0u, presel) + (uint32_t)__popc(W & rl.before);
        sel = __shfl_sync(kFull, rl.seltab, (int)(W >> nshift));
        const uint32_t *aw = reinterpret_cast<const uint32_t *>(smem + (q & ~3u));
        w0 = aw[0];
        w1 = aw[1];
        wsh = q * 8u;
        slot = own + 128u * p;
        if ((uint32_t)lane < p) mine = line;
    }
    if (any) *reinterpret_cast<uint32_t *>(slot) = __byte_perm(__funnelshift_r(w0, w1, wsh), 0u, sel);
    cur = line + row_bytes;
    const bool mine_dense = (dense >> lane) & 1u, exists = (rows >> lane) & 1u;
    uint32_t a = mine - row_bytes * (uint32_t)lane;
    a = mine_dense ? a : (exists ? slots + 128u * (uint32_t)lane : 0u);
    *reinterpret_cast<uint2 *>(smem + tab + 8u * lane) = make_uint2(a & ~3u, a * 8u);
}

// This lane's word (row bytes 4 lane .. 4 lane + 3) of kN planes placed by place_rows.
template <int kN>
__device__ __forceinline__ void gather_rows(const uint8_t *smem, uint32_t tab, int lane, uint32_t (&r)[kN]) {
    const uint8_t *mine = smem + 4 * lane;
#pragma unroll
    for (int i = 0; i < kN / 2; ++i) {
        const uint4 e = *reinterpret_cast<const uint4 *>(smem + tab + 16 * i);
        const uint32_t *x = reinterpret_cast<const uint32_t *>(mine + e.x), *y = reinterpret_cast<const uint32_t *>(mine + e.z);
        r[2 * i] = __funnelshift_r(x[0], x[1], e.y);
        r[2 * i + 1] = __funnelshift_r(y[0], y[1], e.w);
    }
}

// 32 bytes to global memory with one store (32-byte aligned): a whole sector per lane.
__device__ __forceinline__ void store32(void *dst, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

// Values (four 16-byte words at a time) of a lane as 64-bit words.
__device__ __forceinline__ uint64_t pair64(uint64_t const (&d)[32], int i) { return d[i]; }
__device__ __forceinline__ uint64_t pair64(uint32_t const (&d)[32], int i) { return ((uint64_t)d[2 * i + 1] << 32) | d[2 * i]; }
__device__ __forceinline__ uint64_t pair64(uint16_t const (&d)[32], int i) {
    const uint32_t lo = (uint32_t)d[4 * i] | ((uint32_t)d[4 * i + 1] << 16);
    const uint32_t hi = (uint32_t)d[4 * i + 2] | ((uint32_t)d[4 * i + 3] << 16);
    return ((uint64_t)hi << 32) | lo;
}

// The chunk's m values (lane l holds 32 l .. 32 l + 31 in d, lane 31 value 1024 in vx) to dst, whole
// sectors per lane: a whole FP64 chunk at a 32-byte aligned address.
template <class U>
__device__ __forceinline__ void store_sectors(uint8_t *dst, uint32_t m, const U (&d)[32], U vx, int lane) {
    constexpr int S = sizeof(U);
    if (m > 1024u && lane == 31) *reinterpret_cast<U *>(dst + 1024 * S) = vx;
    uint8_t *mine = dst + lane * (32 * S);
#pragma unroll
    for (int i = 0; i < S; ++i)
        store32(mine + 32 * i, pair64(d, 4 * i), pair64(d, 4 * i + 1), pair64(d, 4 * i + 2), pair64(d, 4 * i + 3));
}

// The same at any alignment: the values pass through the slots (swizzled; FP64 half the lanes at a time)
// and leave as coalesced 16-byte units, or single values where dst is not 16-byte aligned.  `conv`
// maps what is staged to values in place, on the way out (kRolled: it is long, so the loops are rolled);
// the whole warp calls it.  (Whole sectors against staging: FP64 segments 325 / 332 us, FP32
// 170 / 162 us, so FP32 and FP16, whose values pass the slots once, always stage.)
template <int D, bool kRolled, class Conv>
__device__ __forceinline__ void store_staged(uint8_t *dst, uint32_t m, uint8_t *slots,
                                             const typename Traits<D>::U (&d)[32], typename Traits<D>::U vx, int lane,
                                             Conv &&conv) {
    using T = Traits<D>;
    using U = typename T::U;
    constexpr int S = T::S, UN = T::UNITS, PER = 16 / S;
    if (m > 1024u) {
        U e[1] = {vx};
        conv(e);
        if (lane == 31) *reinterpret_cast<U *>(dst + 1024 * S) = e[0];
    }
    constexpr int kPasses = D == kD64 ? 2 : 1, kLanes = 32 / kPasses;
    const bool al16 = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0;
#pragma unroll 1
    for (int pass = 0; pass < kPasses; ++pass) {
        const uint32_t v0 = (uint32_t)(pass * kLanes * 32);
        if (v0 >= m) break;
        const uint32_t cnt = min(m - v0, (uint32_t)(kLanes * 32));
        if (lane / kLanes == pass) {
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                const uint64_t lo = pair64(d, 2 * u), hi = pair64(d, 2 * u + 1);
                *reinterpret_cast<uint4 *>(slots + ((lane % kLanes) * UN + unit_swizzle<D>(lane % kLanes, u)) * 16) =
                    make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
            }
        }
        __syncwarp();
        uint8_t *out = dst + v0 * S;
        auto unit = [&](uint32_t q, bool store) {
            union { uint4 w; U e[PER]; } x;
            x.w = *reinterpret_cast<const uint4 *>(slots + phys_unit<D>(q) * 16u);
            conv(x.e);
            if (store) *reinterpret_cast<uint4 *>(out + 16u * q) = x.w;
        };
        auto one = [&](uint32_t i) {
            U e[1] = {*reinterpret_cast<const U *>(slots + phys_elem_byte<D>(i))};
            conv(e);
            *reinterpret_cast<U *>(out + i * S) = e[0];
        };
        if (!kRolled && cnt == (uint32_t)(kLanes * 32)) {        // whole pass: fixed trip counts
            if (al16) {
#pragma unroll
                for (int i = 0; i < kLanes * UN / 32; ++i) unit(32u * i + lane, true);
            } else {
#pragma unroll
                for (int i = 0; i < kLanes; ++i) one(32u * i + lane);
            }
        } else {
            uint32_t done = 0;
            if (al16) {
                done = cnt * S >> 4;
#pragma unroll 1
                for (uint32_t q = 0; q < done; q += 32) unit(min(q + lane, done - 1u), q + lane < done);
                done *= PER;
            }
            // two values at a time, whose divisions overlap (b = 1025: 179.2 -> 172.6 us; four: 182.1)
#pragma unroll 1
            for (uint32_t i = done + lane; i - lane < cnt; i += 64) {
                const uint32_t j = i + 32u;
                auto at = [&](uint32_t k) { return *reinterpret_cast<const U *>(slots + phys_elem_byte<D>(min(k, cnt - 1u))); };
                U e[2] = {at(i), at(j)};
                conv(e);
                if (i < cnt) *reinterpret_cast<U *>(out + i * S) = e[0];
                if (j < cnt) *reinterpret_cast<U *>(out + j * S) = e[1];
            }
        }
        __syncwarp();
    }
}

// FP64 Case 1: g to fl(g / 10^alpha).  Values of a warp that all fit 32 bits (the common case) take the
// 96-bit reciprocal, others the exact division, |g| > 2^53 (only in streams no encoder writes) the
// FP64 divide.
struct ConvF64 {
    Div10Narrow qn;
    int alpha;
    __device__ __forceinline__ explicit ConvF64(int a) : qn(div10_narrow_of(a < kDiv10NarrowMax ? a : kDiv10NarrowMax)), alpha(a) {}
    template <int N> __device__ __forceinline__ void operator()(uint64_t (&g)[N]) const {
        uint32_t wide = alpha > kDiv10NarrowMax ? 1u : 0u;
#pragma unroll
        for (int i = 0; i < N; ++i) wide |= (uint32_t)(g[i] >> 32) ^ (uint32_t)((int32_t)(uint32_t)g[i] >> 31);
        if (!__any_sync(kFull, wide)) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint32_t s = (uint32_t)((int32_t)(uint32_t)g[i] >> 31);
                g[i] = div_pow10_exact32(((uint32_t)g[i] ^ s) - s, s, qn);
            }
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint32_t hi = (uint32_t)(g[i] >> 32), mag = hi ^ (uint32_t)((int32_t)hi >> 31);
                g[i] = mag >= (1u << 21) ? (uint64_t)__double_as_longlong(div_pow10((int64_t)g[i], alpha))
                                         : div_pow10_exact((int64_t)g[i], div10_of(alpha));
            }
        }
    }
};

// A value's exact FP64 value, and its key in IEEE 754 totalOrder (for min / max of non-NaN values).
__device__ __forceinline__ double value_f64(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ double value_f64(uint32_t b) { return (double)__uint_as_float(b); }
__device__ __forceinline__ double value_f64(uint16_t b) { return (double)__half2float(__ushort_as_half(b)); }
__device__ __forceinline__ uint64_t order_key(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// One chunk's record (in the warp's buffer at shared-memory offset wofs) to its values.  `next`
// starts the copy of the warp's next record into the buffer; it is called exactly once, as soon as
// this record has been read completely.
// kAgg (analytics on compressed data): instead of storing the values, the warp adds them up
// (NaN count, totalOrder min / max, their sum: each lane its 32 values in index order, then a
// butterfly over the lanes, identical in every lane since FP addition commutes); the chunk's
// sum goes to sums[c], the rest into the control block by atomics.
template <int D, class L, bool kAgg, bool kTable, class Next>
__device__ __forceinline__ void decode_chunk(const Rec &r0, const Job &single, uint8_t *smem, uint32_t wofs, uint32_t seltab, int lane,
                                             Next &&next, Control *ctl) {
    using T = Traits<D>;
    using U = typename T::U;
    const uint32_t slots = wofs + L::kBuf, tab = slots + L::kSlots;
    ChunkNote &note = *reinterpret_cast<ChunkNote *>(smem + wofs + L::kNote);
    auto values_in = [](const Job &job, uint64_t c) {
        const uint64_t left = job.n - c * (uint64_t)job.block;
        return (uint32_t)(left < job.block ? left : job.block);
    };
    const uint32_t cols = chunk_cols(values_in(kTable ? *r0.job : single, r0.c));
    const uint32_t row_bytes = cols / 8u, bm_bytes = cols / 64u;
    const uint32_t rec = wofs + (r0.phase & 15u);

    // ---- a. header and flags ------------------------------------------------------------------
    bool bad = r0.phase == kBadRecord;
    // a malformed record: its chunk adds nothing to the aggregate, whose finish reads every chunk's sum
    auto reject = [&]() {
        if (lane != 0) return;
        const Job &job = kTable ? *note.job : single;
        set_status(job.result, kErrCorrupt);
        if constexpr (kAgg) reinterpret_cast<double *>(job.flags + job.nchunks)[note.c] = 0.0;
    };
    if (lane == 0) {
        const uint32_t h0 = lds_any(smem, rec);
        note.c = r0.c;
        if (kTable) note.job = r0.job;
        note.alpha = h0 & 0xFFu;
        note.beta_hat = (h0 >> 8) & 0xFFu;
        if constexpr (D == kD64) note.z1 = ((uint64_t)lds_any(smem, rec + 6) << 32) | lds_any(smem, rec + 2);
        else if constexpr (D == kD32) note.z1 = lds_any(smem, rec + 2);
        else note.z1 = h0 >> 16;
    }
    const uint32_t w = smem[rec + 2 + T::Z1B];
    const uint32_t hdr = 3u + T::Z1B + (w + 7u) / 8u;
    if (w > (uint32_t)T::W || (cols == 0u && w != 0u) || hdr > r0.size) bad = true;
    // the flags' last w bits, big-endian: bit p is plane p's
    const uint32_t rows_lo = w >= 32u ? ~0u : (1u << w) - 1u;
    const uint32_t dense_lo = bswap(lds_any(smem, rec + hdr - 4u)) & rows_lo;
    RowLane rl;
    {
        const uint32_t nact = cols / 32u, g8 = (uint32_t)lane & ~7u;
        const uint32_t have = nact > g8 ? min(nact - g8, 8u) : 0u;          // lanes of this group with row bytes
        const uint32_t k8 = 8u * (((uint32_t)lane & 7u) >> 1);
        rl.keep = have == 8u ? 0xFFFFFFFFu : (1u << (4u * have)) - 1u;       // `have` is even
        rl.before = ((1u << k8) - 1u) | ((lane & 1) ? 0xF0u << k8 : 0u);
        rl.seltab = seltab;
    }
    uint32_t cur = rec + hdr;

    // ---- b. every plane's row: placed, gathered (lane: 4 row bytes per plane), transposed -------
    // The planes are transposed one row up (plane p at row p - 1) and XORed with plane 0, whose
    // bits are the signs: that is the inverse zigzag of all values at once, one XOR per plane.
    // Lanes past the row's bytes (tail chunks) gather stale bytes; their columns lie past the
    // chunk's values, are never stored, and only feed the scan of later lanes.
    U d[32];
    if constexpr (D == kD64) {
        // both halves run one copy of this code (a third of the kernel's instructions otherwise)
        uint32_t hi[32], a[32], top = 0, sgn = 0;         // top: plane 32's word, the low half's last row
#pragma unroll
        for (int k = 0; k < 32; ++k) hi[k] = 0;
        if (!bad) {
#pragma unroll 1
            for (int h = w > 32u ? 1 : 0; h >= 0; --h) {
                const uint32_t wh = w - 32u * (uint32_t)h, rows = wh >= 32u ? ~0u : (1u << wh) - 1u;
                const uint32_t dense = bswap(lds_any(smem, rec + hdr - 4u - 4u * (uint32_t)h)) & rows;
                place_rows(smem, slots, tab, cur, rows, dense, row_bytes, bm_bytes, rl, lane);
                __syncwarp();
                uint32_t r[32];
                gather_rows<32>(smem, tab, lane, r);
                sgn = h ? 0u : r[0];
#pragma unroll
                for (int i = 0; i < 31; ++i) a[i] = r[i + 1] ^ sgn;
                a[31] = top ^ sgn;
                top = r[0];
                __syncwarp();
                if (h == 0) next();               // the record has been read
                transpose32(a);
                if (h) {
#pragma unroll
                    for (int k = 0; k < 32; ++k) hi[k] = a[k ^ 7];
                }
            }
            bad = cur - rec != r0.size;
            if (bad) {
                reject();
                return;
            }
        } else {
            reject();
            __syncwarp();
            next();
            return;
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const uint32_t s = (uint32_t)((int32_t)(sgn << (31 - (k ^ 7))) >> 31);
            d[k] = (U)(((uint64_t)(hi[k] ^ s) << 32) | a[k ^ 7]);
        }
    } else {
        if (!bad) {
            place_rows(smem, slots, tab, cur, rows_lo, dense_lo, row_bytes, bm_bytes, rl, lane);
            bad = cur - rec != r0.size;
        }
        __syncwarp();
        if (bad) {
            reject();
            next();
            return;
        }
        constexpr int R = T::W < 32 ? T::W : 32;
        uint32_t a[32], r[R];
        gather_rows<R>(smem, tab, lane, r);
#pragma unroll
        for (int i = 0; i < 32; ++i) a[i] = i + 1 < R ? r[i + 1 < R ? i + 1 : 0] ^ r[0] : (i + 1 == R ? r[0] : 0u);
        __syncwarp();
        next();                                   // the record has been read
        transpose32(a);
#pragma unroll
        for (int k = 0; k < 32; ++k) d[k] = (U)a[k ^ 7];
    }
    // ---- c. G (inverse Eq. 5): lane l's values 32 l .. 32 l + 31 -------------------------------
    const U z1 = (U)note.z1;
    U run = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) run += d[k];
    if constexpr (D == kD64) run = z1 + warp_exclusive_u64(run, lane);
    else run = (U)(z1 + warp_exclusive_u32((uint32_t)run, lane));
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const U t = d[k];
        d[k] = run;
        run += t;
    }
    U vx = run;                                   // lane 31: value 1024
    const Job &job = kTable ? *note.job : single;
    const uint64_t c = note.c;
    const uint32_t m = values_in(job, c), alpha = note.alpha, beta_hat = note.beta_hat;
    uint8_t *dst = job.out + c * (uint64_t)job.block * T::S;
    // ---- d. values (inverse Eq. 4) ---------------------------------------------------------------
    if (alpha <= (uint32_t)T::A_MAX && beta_hat <= (uint32_t)T::B_MAX) {
        if constexpr (D == kD64) {
            const ConvF64 conv((int)alpha);
            if constexpr (kAgg) {                 // the values are wanted in registers
#pragma unroll 1
                for (int i = 0; i < 32; i += 2) {       // rolled (small code): the values rotate through d[0], d[1]
                    U e[2] = {d[0], d[1]};
                    conv(e);
#pragma unroll
                    for (int k = 0; k < 30; ++k) d[k] = d[k + 2];
                    d[30] = e[0];
                    d[31] = e[1];
                }
                U e[1] = {vx};
                conv(e);
                vx = e[0];
            } else {
                // divided on the way out, in rolled loops: unrolled over the 32 registers, the
                // division cost every chunk spills and instruction fetch (2^26 segments 309 -> 296 us
                // without, 2^25 decimal values 206 -> 160 us)
                store_staged<D, true>(dst, m, smem + slots, d, vx, lane, conv);
                return;
            }
        } else {
            // FP16: fl16(g / 10^a) as fl16(fl32(g / 10^a)): exact for every 16-bit g and a <= 4 (the
            // second rounding never lands on a different value; checked for all 327,680 inputs)
            const Div10F32 q = div10_f32_of((int)alpha);
            auto conv = [&](U g) {
                if constexpr (D == kD32) return __float_as_uint(div_pow10(__int2float_rn((int32_t)g), q));
                else return __half_as_ushort(__float2half_rn(div_pow10((float)(int16_t)g, q)));
            };
#pragma unroll
            for (int k = 0; k < 32; ++k) d[k] = conv(d[k]);
            vx = conv(vx);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) d[k] = unzigzag(d[k]);
        vx = unzigzag(vx);
    }

    if constexpr (kAgg) {
        // keys in the values' own width (IEEE order = unsigned order of the keys), widened to
        // FP64 keys once per chunk
        constexpr U SIGN = (U)((U)1 << (T::W - 1));
        constexpr U ABSM = (U)(SIGN - 1u);
        constexpr U INF = (U)(D == kD64 ? 0x7FF0000000000000ull : (D == kD32 ? 0x7F800000ull : 0x7C00ull));
        uint32_t nan = 0;
        U kmin = (U)~(U)0, kmax = 0;
        double sum = -0.0;                        // -0 + x == x for every x, -0 + -0 == -0
        auto take = [&](U b) {
            if ((U)(b & ABSM) > INF) { ++nan; return; }
            const U key = (b & SIGN) ? (U)~b : (U)(b | SIGN);
            kmin = key < kmin ? key : kmin;
            kmax = key > kmax ? key : kmax;
            sum = __dadd_rn(sum, value_f64(b));
        };
#pragma unroll
        for (int k = 0; k < 32; ++k)
            if (32u * (uint32_t)lane + (uint32_t)k < m) take(d[k]);
        if (m > 1024u && lane == 31) take(vx);
        nan = __reduce_add_sync(kFull, nan);
        if constexpr (D == kD64) {
            kmin = ~warp_max_u64(~kmin);
            kmax = warp_max_u64(kmax);
        } else {
            kmin = (U)__reduce_min_sync(kFull, (uint32_t)kmin);
            kmax = (U)__reduce_max_sync(kFull, (uint32_t)kmax);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum = __dadd_rn(sum, __shfl_xor_sync(kFull, sum, o));
        if (lane == 0) {
            reinterpret_cast<double *>(job.flags + job.nchunks)[c] = sum;
            if (nan) atomicAdd(&ctl->agg[0], (unsigned long long)nan);
            if (kmax) {                           // some value was not a NaN
                auto unkey = [&](U k) { return (k & SIGN) ? (U)(k & ABSM) : (U)~k; };
                atomicMax(&ctl->agg[1], (unsigned long long)~order_key(value_f64(unkey(kmin))));
                atomicMax(&ctl->agg[2], (unsigned long long)order_key(value_f64(unkey(kmax))));
            }
        }
        __syncwarp();
        return;
    }

    if (D == kD64 && m >= 1024u && (reinterpret_cast<uintptr_t>(dst) & 31u) == 0) store_sectors(dst, m, d, vx, lane);
    else store_staged<D, false>(dst, m, smem + slots, d, vx, lane, [](auto &) {});
}

}  // namespace

// The position of every record (exclusive prefix of the u32 size array) of every job into the
// first words of job.flags.  A single stream: `parts` CTAs, each over its own share of the chunks; a CTA
// adds up every size before its share first (at most 152 CTAs reading at most the whole array, from
// L2), then scans its share 1024 chunks at a time, so no CTA waits for another.  A table: `per` jobs per
// CTA, each by a warp of its own when it has at most 32 `per` chunks (a warp scans 32 chunks in about the
// time the CTA takes for a job), the longer ones by the whole CTA in turn.
// 16,000 FP32 series of 10 values, one CTA each: compressed in 366 us, decompressed in 172; so 231 and 52.
__device__ __forceinline__ void put_position(const Job &job, int which, uint64_t c, uint64_t at) {
    if (which == kOffsetsOfInput) job.flags[c] = at;
    else job.flags[c] = ((job.flags[c] >> kOffsetBits) << kOffsetBits) | at;
}
__device__ __forceinline__ const uint32_t *sizes_of(const Job &job, int which) {          // 16-byte aligned
    return reinterpret_cast<const uint32_t *>((which == kOffsetsOfInput ? job.in : job.out) + 32);
}
// chunks [begin, end) by the whole CTA; begin a multiple of 1024
__device__ __forceinline__ void scan_by_cta(const Job &job, int which, uint64_t begin, uint64_t end, uint64_t *warp_sums) {
    const uint32_t *sizes = sizes_of(job, which);
    uint64_t carry = 0;
    if (begin > 0) {
        const uint4 *q = reinterpret_cast<const uint4 *>(sizes);
        uint64_t sum = 0;
        for (uint64_t i = threadIdx.x; i < begin / 4u; i += 1024u) {
            const uint4 x = q[i];
            sum += (uint64_t)x.x + x.y + x.z + x.w;
        }
        (void)block_exclusive_scan(sum, carry, warp_sums);
    }
    for (uint64_t b = begin; b < end; b += 1024u) {
        const uint64_t c = b + threadIdx.x;
        uint64_t total;
        const uint64_t ex = block_exclusive_scan(c < end ? sizes[c] : 0u, total, warp_sums);
        if (c < end) put_position(job, which, c, carry + ex);
        carry += total;
    }
}
// a short job by one warp
__device__ __forceinline__ void scan_by_warp(const Job &job, int which, int lane) {
    const uint32_t *sizes = sizes_of(job, which);
    const uint32_t nc = (uint32_t)job.nchunks;
    uint64_t carry = 0;
    uint32_t size = (uint32_t)lane < nc ? sizes[lane] : 0u;
    for (uint32_t b = 0; b < nc; b += 32u) {
        const uint32_t c = b + (uint32_t)lane, mine = size;
        size = c + 32u < nc ? sizes[c + 32u] : 0u;
        const uint64_t incl = mine + warp_exclusive_u64(mine, lane);
        if (c < nc) put_position(job, which, c, carry + incl - mine);
        carry += shfl_u64(incl, 31);
    }
}
__device__ __forceinline__ void start_decode(const Job &job) {            // the results, ready for the decode
    job.result[0] = job.n;
    job.result[1] = kOk;
}
__global__ void __launch_bounds__(1024, 2)
offsets_kernel(Job single, uint32_t parts, int which, Control *ctl) {
    __shared__ uint64_t warp_sums[33];
    pdl_trigger();
    pdl_wait();                                   // compression: the analysis' sizes
    const uint64_t nc = single.nchunks;
    if (which == kOffsetsOfInput && blockIdx.x == 0 && threadIdx.x == 0) {
        *ctl = Control{};
        start_decode(single);
    }
    const uint64_t share = ((nc + parts - 1) / parts + 1023u) & ~1023ull;
    const uint64_t begin = blockIdx.x * share, end = begin + share < nc ? begin + share : nc;
    if (begin < nc) scan_by_cta(single, which, begin, end, warp_sums);
}
__global__ void __launch_bounds__(1024, 2)
table_offsets_kernel(const Job *__restrict__ jobs, int njobs, uint32_t per, int which, Control *ctl) {
    __shared__ uint64_t warp_sums[33];
    pdl_trigger();
    pdl_wait();
    if (which == kOffsetsOfInput && blockIdx.x == 0 && threadIdx.x == 0) *ctl = Control{};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Job *mine = jobs + (size_t)blockIdx.x * per;
    const int count = min((int)per, njobs - (int)(blockIdx.x * per));
    auto is_short = [&](const Job &job) { return per > 1u && job.nchunks <= 32u * per; };
    if (warp < count) {
        if (which == kOffsetsOfInput && lane == 0) start_decode(mine[warp]);
        if (is_short(mine[warp])) scan_by_warp(mine[warp], which, lane);
    }
    for (int i = 0; i < count; ++i)
        if (!is_short(mine[i])) scan_by_cta(mine[i], which, 0, mine[i].nchunks, warp_sums);
}

// Forms by dtype: kDt = 0 (every job FP64), 1 (every job FP32), 2 (either, per job).
constexpr int kDtF64 = 0, kDtF32 = 1, kDtMixed = 2, kDtF16 = 3;
// the value kind whose buffers a form needs (the either-dtype form: the largest)
template <int kDt> constexpr int layout_kind() { return kDt == kDtF32 ? kD32 : (kDt == kDtF16 ? kD16 : kD64); }

// Registers: 128 (FP64, either-dtype: 16 warps per SM), 80 (FP32, FP16: 24 warps; 96 registers and
// 20 warps: 1.3 % slower).  The aggregate forms keep every value and the FP64 sums in registers: 168
// (FP64: 12 warps) and 128.
template <int kDt, bool kAgg = false>
__global__ void __maxnreg__((kDt == kDtF32 || kDt == kDtF16) && !kAgg ? 80 : (kAgg ? (kDt == kDtF64 ? 168 : 128) : 128))
decompress_kernel(const Job *__restrict__ jobs, int njobs, Job single, uint64_t total_chunks, Control *ctl) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    using L = DecLayout<layout_kind<kDt>()>;
    const uint32_t wofs = kZeroBytes + (uint32_t)warp * L::kWarpBytes;
    uint8_t *wbase = smem + wofs;
    const uint32_t seltab = expand_sel((uint32_t)lane & 15u);
    __shared__ Job s_single;                      // the single job, read from shared memory
    if (threadIdx.x == 0) s_single = single;
    if (threadIdx.x < kZeroBytes / 16u) reinterpret_cast<uint4 *>(smem)[threadIdx.x] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    if constexpr (kAgg) pdl_trigger();            // the finish launch
    pdl_wait();                                   // the offsets, and everything before them
    // chunk tickets two deep: while one chunk is decoded the next one's record is fetched, and the
    // ticket of the one after that is on its way (read, and its position loads issued, when this
    // chunk is done)
    constexpr bool kTable = kDt == kDtMixed;
    const Tickets tickets{ctl, kTicketDecode, total_chunks};
    uint64_t tn = tickets.first();
    if (tn >= total_chunks) return;
    Rec rec = issue_record(locate<kTable>(jobs, njobs, s_single, tn, total_chunks, lane), wbase, lane);
    cp_async_commit();
    tn = tickets.chunk(tickets.draw(lane));
    Loc ln = locate<kTable>(jobs, njobs, s_single, tn, total_chunks, lane);
    for (;;) {
        const unsigned long long raw = tickets.draw(lane);
        cp_async_wait_none();                    // the current record has landed
        __syncwarp();
        // the next record goes into the same buffer once this one has been read
        Rec rn{};
        auto next = [&]() {
            if (tn < total_chunks) rn = issue_record(ln, wbase, lane);
            cp_async_commit();
        };
        if constexpr (kDt == kDtF64) decode_chunk<kD64, L, kAgg, kTable>(rec, s_single, smem, wofs, seltab, lane, next, ctl);
        else if constexpr (kDt == kDtF32) decode_chunk<kD32, L, kAgg, kTable>(rec, s_single, smem, wofs, seltab, lane, next, ctl);
        else if constexpr (kDt == kDtF16) decode_chunk<kD16, L, kAgg, kTable>(rec, s_single, smem, wofs, seltab, lane, next, ctl);
        else if (rec.job->dtype == 0) decode_chunk<kD64, L, kAgg, kTable>(rec, s_single, smem, wofs, seltab, lane, next, ctl);
        else if (rec.job->dtype == 1) decode_chunk<kD32, L, kAgg, kTable>(rec, s_single, smem, wofs, seltab, lane, next, ctl);
        else decode_chunk<kD16, L, kAgg, kTable>(rec, s_single, smem, wofs, seltab, lane, next, ctl);
        if (tn >= total_chunks) break;
        rec = rn;
        tn = tickets.chunk(raw);
        ln = locate<kTable>(jobs, njobs, s_single, tn, total_chunks, lane);
    }
    cp_async_wait_none();
}

// The aggregate's last step (one CTA): thread t adds the chunk sums of its contiguous share in
// chunk order, then a fixed tree over the threads; the NaN count and the min / max keys come
// from the control block, the status from the decode.  Every step has a fixed order, so the
// result does not depend on the schedule.
__global__ void __launch_bounds__(1024)
aggregate_finish_kernel(Job single, Control *ctl, falcon_stats *out) {
    __shared__ double part[1024];
    pdl_wait();
    const uint64_t nc = single.nchunks;
    const double *sums = reinterpret_cast<const double *>(single.flags + nc);
    const uint64_t c0 = nc * threadIdx.x / 1024u, c1 = nc * (threadIdx.x + 1u) / 1024u;
    double s = -0.0;
    for (uint64_t c = c0; c < c1; ++c) s = __dadd_rn(s, sums[c]);
    part[threadIdx.x] = s;
    __syncthreads();
    for (unsigned h = 512; h > 0; h >>= 1) {
        if (threadIdx.x < h) part[threadIdx.x] = __dadd_rn(part[threadIdx.x], part[threadIdx.x + h]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const unsigned long long nan = ctl->agg[0], kmin_c = ctl->agg[1], kmax = ctl->agg[2];
        auto from_key = [](uint64_t k) {
            return __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k));
        };
        out->count = single.n;
        out->nan_count = nan;
        out->min = kmax ? from_key(~kmin_c) : __longlong_as_double(0x7FF8000000000000ll);
        out->max = kmax ? from_key(kmax) : __longlong_as_double(0x7FF8000000000000ll);
        out->sum = kmax ? part[0] : 0.0;          // no non-NaN value: the empty sum
        out->status = single.result[1];
    }
}

namespace {
template <int kDt, bool kAgg = false>
void launch_decode(const Job *d_jobs, int njobs, const Job &single, uint64_t total_chunks, Control *ctl,
                   cudaStream_t stream) {
    const int w = g_cta_warps[1], smem = (int)(kZeroBytes + w * DecLayout<layout_kind<kDt>()>::kWarpBytes);
    const int grid = persistent_grid_size(reinterpret_cast<const void *>(decompress_kernel<kDt, kAgg>), w, smem,
                                          g_ctas_per_sm[1], total_chunks);
    (void)launch_after(g_ctas_per_sm[1] == 0, decompress_kernel<kDt, kAgg>, grid, 32 * w, smem, stream, d_jobs, njobs, single,
                       total_chunks, ctl);
}
}  // namespace

// A single stream: one CTA per 1024 chunks, up to 152.  A table: one CTA per job up to 304 jobs (two
// CTAs of 1024 threads to an SM), beyond that up to 32 jobs share a CTA, so that many short jobs do
// not take their CTAs' launches in turn.
// Compression's follows the analysis; decompression's is the first launch of the call, after whatever
// the caller has enqueued.
void launch_offsets(const Job *d_jobs, int njobs, const Job &single, int which, Control *ctl, cudaStream_t stream) {
    const bool after = which == kOffsetsOfOutput;
    if (d_jobs == nullptr) {
        const uint64_t steps = (single.nchunks + 1023u) / 1024u;
        const uint32_t parts = steps < 1u ? 1u : (steps > 152u ? 152u : (uint32_t)steps);
        if (after) (void)launch_after(true, offsets_kernel, (int)parts, 1024, 0, stream, single, parts, which, ctl);
        else offsets_kernel<<<parts, 1024, 0, stream>>>(single, parts, which, ctl);
        return;
    }
    const uint32_t per = std::min(((uint32_t)njobs + 303u) / 304u, 32u), ctas = ((uint32_t)njobs + per - 1u) / per;
    if (after) (void)launch_after(true, table_offsets_kernel, (int)ctas, 1024, 0, stream, d_jobs, njobs, per, which, ctl);
    else table_offsets_kernel<<<ctas, 1024, 0, stream>>>(d_jobs, njobs, per, which, ctl);
}

cudaError_t launch_aggregate(const Job &single, Control *ctl, void *d_stats, cudaStream_t stream) {
    launch_offsets(nullptr, 1, single, kOffsetsOfInput, ctl, stream);
    if (single.nchunks > 0) {
        if (single.dtype == 0) launch_decode<kDtF64, true>(nullptr, 1, single, single.nchunks, ctl, stream);
        else if (single.dtype == 1) launch_decode<kDtF32, true>(nullptr, 1, single, single.nchunks, ctl, stream);
        else launch_decode<kDtF16, true>(nullptr, 1, single, single.nchunks, ctl, stream);
    }
    (void)launch_after(true, aggregate_finish_kernel, 1, 1024, 0, stream, single, ctl, static_cast<falcon_stats *>(d_stats));
    return cudaGetLastError();
}

cudaError_t launch_decompress(const Job *d_jobs, int njobs, const Job &single, uint64_t total_chunks,
                              Control *ctl, cudaStream_t stream) {
    launch_offsets(d_jobs, njobs, single, kOffsetsOfInput, ctl, stream);
    if (d_jobs != nullptr) launch_decode<kDtMixed>(d_jobs, njobs, single, total_chunks, ctl, stream);
    else if (single.dtype == 0) launch_decode<kDtF64>(d_jobs, njobs, single, total_chunks, ctl, stream);
    else if (single.dtype == 1) launch_decode<kDtF32>(d_jobs, njobs, single, total_chunks, ctl, stream);
    else launch_decode<kDtF16>(d_jobs, njobs, single, total_chunks, ctl, stream);
    return cudaGetLastError();
}

}  // namespace falcon
