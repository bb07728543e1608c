// Streaming kernel for the decode GEMV (PoT and the uniform twin) and the small-batch GEMM on the tiled layout.
//
// Work decomposition.  The matrix is a sequence of units (16 rows x 128 columns, stored contiguously in
// [row block][column block] order, codes and per-group parameters alike).  A CTA -- and every warp in it -- streams a contiguous
// byte range (the even split: a warp two).  Three splits: whole row blocks per CTA; the same number of units for every CTA
// (even split, where the matrix has a row block for each); the same number for every warp of the grid (unit split).
//
// Every warp is its own streaming engine: it owns a private ring of S slots of Q units in shared memory; lane 0 requests
// a slot's codes and scales with 1-D bulk copies (cp.async.bulk + mbarrier transaction bytes), the warp waits for the
// slot, works through its units and, when all lanes are done with it, lane 0 requests the chunk that reuses the slot.
// There is no producer warp, no empty barrier and no synchronisation between warps on the data path; the first S chunks
// are requested before the kernel waits for its predecessor in the stream (the weights are constants).
//
// Arithmetic.  Lane (gid, tig) of a warp owns quarter tig (32 columns) of rows gid and gid + 8 of a unit: exactly its
// share of the A fragments of eight m16n8k16 MMAs.  It decodes its 2 x 32 codes in registers to +-2^E under a constant
// exponent and issues the MMAs against B fragments that hold the activation vector in every column (GEMV) or one token per
// column (small batch); the group's scale multiplies the unit's FP32 sums.  One BF16 token is staged as FP16 numbers relative to the
// largest of each unit where that is exact, and the unit's sums are multiplied by that factor too; the units where it is not are
// decoded to BF16.  (Where a unit's sums mix two groups -- several tokens with G = 64 --, with several BF16 tokens, on small matrices
// with BF16, where x does not fit in shared memory and in the uniform twin the scale goes into the weights: mask, shift and integer add
// into its bit pattern, Sec. 4.2 of the paper.)  The FP32 accumulators stay in registers for as long as the warp stays inside one row block.
//
// Delivery.  A warp that covered a whole row block writes Y.  Otherwise its sums go to slot (row block, position of the
// warp among the row block's contributors) of the workspace; a per-row-block arrival counter tells the last contributor,
// which adds the slots in ascending order -- the result does not depend on timing, and no warp waits for another (even split: see
// stream_even.cuh; there too no CTA waits for another).
#pragma once
#include "common.cuh"
#include "layout.cuh"
#include "sync.cuh"

#include <type_traits>

namespace pot {

enum StreamKind { SK_POT = 0, SK_UINT = 1 };

constexpr int SK_QMAX = 4;  // units per chunk (one ring slot, one set of bulk copies): 4; 2 where 4 would leave one slot; 8 for long ranges

__host__ __device__ constexpr int sk_unit_bytes(int bits) { return 256 * bits; }
// bytes of one ring slot: Q units of codes, then their scales (then their zero-points)
__host__ __device__ constexpr int sk_param_bytes(int group) { return 16 * (128 / group) * 2; }
__host__ __device__ constexpr int sk_unit_total_bytes(int bits, int group, int kind) {
    return sk_unit_bytes(bits) + (kind == SK_UINT ? 2 : 1) * sk_param_bytes(group);
}
__host__ __device__ constexpr int sk_slot_bytes(int bits, int group, int kind, int q) { return q * sk_unit_total_bytes(bits, group, kind); }

// shared-memory header of a CTA: W x 8 full barriers, W x 8 words of per-warp state, W local arrival counters, W x 2 local
// partial-sum slots
__host__ __device__ constexpr int sk_header_bytes(int warps, int tok) {
    return (warps * 64 + warps * 32 + warps * 4 + warps * 2 * 16 * tok * 4 + 127) / 128 * 128;
}

// ---- even split (stream_even.cuh)
// units that are dealt out together (straight-line code; with two of the four in a slot 12288 x 4096 took 8.2 instead of 7.3 us)
__host__ __device__ constexpr int sk_block(int q) { return q == 2 ? 2 : 4; }
// the workspace holds a number and a mark, 8 bytes, for each sum that goes from CTA to CTA (16 rows x tok of each CTA).  These places need not be
// zero before a call, but they must hold no mark, and none is there after it.
constexpr size_t sk_box_bytes(int tok) { return (size_t)kSmCount * 16 * (size_t)tok * 8; }

struct StreamPlan {
    int grid, warps;      // CTAs; consumer warps per CTA
    int ncb;              // column blocks (units per row block)
    uint32_t units;       // U
    uint32_t gw_total;    // GW: warps that own a range (grid * W, or U when there are fewer units than that)
    int q;                // Q: units per slot
    int stages;           // S: slots per warp ring
    int ring_capacity;    // slots per warp that would fit
    int tok;              // B columns in use: 1 (GEMV) or 8 (small batch)
    bool x_in_smem;
    bool unscaled;        // decode without the scale, which multiplies the group's sums instead
    int token_shift;      // log2 of the token slots of the staged activations (0 for the GEMV)
    size_t x_bytes, smem_bytes;
    int max_slots;        // partial-sum slots per row block
    size_t ws_counters, ws_bytes;
    bool aligned;         // whole row blocks per CTA would differ by a fifth at most
    bool even;            // even split: see plan_stream
    uint32_t cta_blocks, cta_more;  // ... of sk_block(q) units: every CTA has cta_blocks of them, the first cta_more CTAs one more
    int nrb;
    bool ok;              // false: the shape cannot run on this kernel (too many units)
};

constexpr int SK_ZERO_BYTES = 256;  // zeros that the unscaled GEMV keeps behind the activations (two groups per unit)
// Whether one BF16 token is decoded without the scale, with x as FP16 numbers.  Every CTA makes all of x such numbers, ncb / 16 units per warp,
// and gets that back on every unit that it decodes, most at 4 bits.  A rest of fewer than four units goes unit by unit and gives nothing
// back, so that two whole slots per warp are worth more than ten units.  Time without the scale / with it at 2 / 3 / 4 bits: 7136 x 4096 (7 units
// per warp) 1.08 / 1.08 / 1.01; 9472 x 4096 (8) 0.95 / 0.93 / 0.95, 18944 x 2048 (8) 0.89 / 0.84 / 0.91, 8192 x 4096 (8, in CTAs of three or four
// row blocks) 1.02 / 0.97 / 0.92; 10656 x 4096 (10) 1.04 / 1.05 / 0.93, with two
// scales per unit 1.05 / 0.96 / 0.93; 13024 x 4096 (12) 0.94 / 0.92 / 0.90.  Where CTAs do not end on row blocks: 2816 x
// 13824 (8) 1.03 / 1.03 / 1.00, 3872 x 13824 (12) 1.02 / 1.00 / 0.97, 4912 x 13824 (15) 0.96 / 0.94 / 0.90; 2032 x 28672 (13) 1.03 / 1.03 / 1.00, 2400 x 28672
// (15) 1.01 / 1.02 / 0.98, 2368 x 28672 (14, CTAs end on row blocks) 0.94 / 0.96 / 0.95, 8192 x 28672 (56) 0.79 / 0.83 / 0.79.
inline bool bf16_as_fp16(const StreamPlan& p, int bits, int group, int64_t rb_min, int64_t rb_max, int64_t per_warp) {
    if (p.aligned && rb_max * p.ncb == 8 * p.warps && p.ncb <= 64 && (bits > 2 || rb_min == rb_max)) return true;
    if (bits == 4) return per_warp >= p.ncb / 16 && per_warp >= (p.aligned ? 8 : 10);
    return per_warp >= p.ncb / (p.aligned ? 16 : 14) && per_warp >= (!p.aligned ? 13 : (bits == 3 && group == 64 && p.ncb >= 24 ? 9 : 11));
}

inline StreamPlan plan_stream(int64_t N, int64_t K, int64_t M, int bits, int group, int kind, int tok, int warps, int occ = 1, int dt = 0) {
    StreamPlan p = {};
    const int64_t nrb = N / 16, ncb = K / 128, U = nrb * ncb;
    p.ok = U > 0 && U < (int64_t(1) << 31) && ncb < (1 << 24);
    if (!p.ok) return p;
    p.warps = warps;
    p.ncb = (int)ncb;
    p.units = (uint32_t)U;
    p.tok = tok;
    // every range must be non-empty (the contributors of a row block are counted as consecutive warps): GW <= U
    int64_t grid = U / warps;
    if (grid < 1) grid = 1;
    p.grid = (int)(grid < kSmCount ? grid : kSmCount);
    p.gw_total = (uint32_t)((int64_t)p.grid * warps < U ? (int64_t)p.grid * warps : U);
    const int64_t GW = (int64_t)p.gw_total;
    // Row-block split: no sums cross CTAs, at the price of CTAs that differ by one row block.  Taken when that costs at
    // most a fifth more than the even split and every warp of a CTA still gets a unit.
    p.nrb = (int)nrb;
    const int64_t rb_min = nrb / p.grid, rb_max = (nrb + p.grid - 1) / p.grid;
    p.aligned = nrb >= p.grid && p.grid == kSmCount && rb_min * ncb >= warps && (double)rb_max * p.grid <= 1.2 * (double)nrb;
    const int64_t per_warp = p.aligned ? (rb_max * ncb + warps - 1) / warps : (U + GW - 1) / GW;
    // shared memory: header, the staged activations, W rings
    const size_t budget = (occ == 2 ? 113 : 224) * 1024;  // two CTAs per SM: 228 KB less 1 KB reserve each
    const size_t hdr = (size_t)sk_header_bytes(warps, tok);
    // multi-token kernel: the staged block has 2, 4 or 8 token slots per 16-byte chunk position (the smallest that holds M)
    p.token_shift = tok > 1 ? (M <= 2 ? 1 : (M <= 4 ? 2 : 3)) : 0;
    p.unscaled = kind == SK_POT && (dt == 0 ? tok == 1 || group == 128 : tok == 1 && bf16_as_fp16(p, bits, group, rb_min, rb_max, per_warp));
    const size_t zeros = p.unscaled && tok == 1 && group == 64 ? SK_ZERO_BYTES : 0;
    const size_t xb = (((size_t)K * 2) << p.token_shift) + (dt == 0 ? zeros : 0);
    // slots of 4 units unless the ring could then hold only one of them next to the staged activations
    int q = SK_QMAX;
    if (hdr + xb + (size_t)warps * 2 * (size_t)sk_slot_bytes(bits, group, kind, q) > budget) q = 2;
    // long ranges (large matrices, one CTA per SM): slots of 8 units halve the per-slot hand-off work, if two of them fit
    else if (occ == 1 && tok == 1 && per_warp >= 32 && hdr + xb + (size_t)warps * 2 * (size_t)sk_slot_bytes(bits, group, kind, 8) <= budget) q = 8;
    p.q = q;
    const size_t slot = (size_t)sk_slot_bytes(bits, group, kind, q);
    const size_t ring2 = (size_t)warps * 2 * slot;  // at least two slots per warp
    p.x_in_smem = hdr + xb + ring2 <= budget;
    p.unscaled = p.unscaled && p.x_in_smem;
    // (BF16: without the scale where zeros and factors fit as well; they decide neither where x goes nor the length of the slots)
    const size_t xf = xb + (dt == 1 ? zeros + (size_t)ncb * 4 : 0);
    if (dt == 1 && hdr + (xf + 127) / 128 * 128 + ring2 > budget) p.unscaled = false;
    p.x_bytes = p.x_in_smem ? ((p.unscaled ? xf : xb) + 127) / 128 * 128 : 0;
    int64_t st = (int64_t)((budget - hdr - p.x_bytes) / ((size_t)warps * slot));
    p.ring_capacity = (int)(st > 8 ? 8 : st);
    const int64_t need = (per_warp + q - 1) / q;
    if (st > need) st = need;
    if (st > 8) st = 8;
    if (st < 1) st = 1;
    // Even split (PoT codes): every CTA takes the same number of blocks of units, wherever row blocks end.  A range is no shorter than a row block, or
    // (the last CTA's, by up to three units) lies inside one, so that a row block has two CTAs at most.  Instead of the unit split always (us: 2480 x 4096
    // 5.7 -> 3.75, 2400 x 8192 6.9 -> 5.95, 7136 x 4096 7.5 -> 5.8, 5120 x 13824 12.4 -> 11.4, eight layers of 2048 / 5504 259 -> 226, of 3200 / 8576
    // 269 -> 240).  Instead of whole row blocks with one CTA per SM, whose launch nothing hides and which gains by the shorter way to the first copies:
    //  * one token always (28672 x 8192 25.0 -> 23.1, 15360 x 8192 17.0 -> 14.7, whole row blocks of 18944 x 8192 17.1 -> 16.7; 4 bits, BF16,
    //    G = 64, 28672 x 8192 28.3 -> 28.0) but at 2 bits in BF16 (17792 x 7552 15.7 -> 16.4), and on long rows, whose activations come in front of all
    //    but the first chunk, only where the longest CTA gets rid of 56 units (7104 x 21760, of none, 18.3 -> 19.3; 4352 x 28672, of 37, 16.2 -> 17.1);
    //  * several tokens, whose sums cost more on their way, where the longest CTA, of three row blocks or more, gets rid of 16 units: two tokens (15360 x
    //    5120 12.8 -> 11.3; 4096 x 11008, of two row blocks, 10.4 -> 12.0), and BF16, which takes longer per unit.  Three and four FP16 tokens: of 40
    //    units (13200 x 9088, 38, 17.3 -> 18.3; 6240 x 6528 at 2 bits, 19, 8.7 -> 10.1), 64 at 2 and 3 bits in three or four row blocks (8096 x
    //    9088, 42, 13.1 -> 14.1); or where x is read through L2 (9200 x 22656 45.2 -> 39.4); or on short rows of 2 or 3 bits in six row blocks and
    //    more (15360 x 5120, 21, 13.4 -> 12.6; in five 10288 x 4096, 21, 8.9 -> 9.25; 14336 x 3456 at 2 bits 8.55 -> 9.45, at
    //    4 bits 15440 x 4352 11.7 -> 12.4).
    // Drawn matrices, of those that the rule takes: one token 0.93 of the time with whole row blocks (250; one above 1.01), two to four 0.94 (400, of
    // which 4 % take 1 - 6 % longer).
    // Two CTAs per SM: alone 12288 x 4096 7.8 -> 7.3, but 11008 x 4096 6.9 -> 7.25, 4096 x 4096 3.5 -> 4.2, and nothing is left where such
    // launches follow one another (eight layers of 4096 / 11008 274 -> 276, 2 bits 245 -> 250).
    const int64_t block = sk_block(q), blocks = (U + block - 1) / block, saved = rb_max * ncb - U / p.grid;
    const bool pays = tok == 1 ? (dt == 0 || bits > 2) && (ncb <= 110 || saved >= 56)
                               : M <= 4 && rb_max >= 3 && saved >= 16 && (M == 2 || dt == 1 || saved >= (rb_max > 4 || bits == 4 ? 40 : 64) || !p.x_in_smem || (bits <= 3 && rb_max >= 6 && saved >= 18 && ncb >= (bits == 2 ? 33 : 24) && ncb <= 60));
    p.even = kind == SK_POT && p.grid == kSmCount && U / 4 / p.grid * 4 >= ncb && ncb > 1 && (!p.aligned || (occ == 1 && pays));
    p.cta_blocks = (uint32_t)(blocks / p.grid);
    p.cta_more = (uint32_t)(blocks % p.grid);
    if (p.even) {  // a warp has a part of the CTA's first row block, if that is shared, and a part of the rest
        const int64_t most = (block * ((p.cta_blocks + 2 + warps) / warps) + q - 1) / q + 1;
        st = (int64_t)((budget - hdr - p.x_bytes) / ((size_t)warps * slot));
        if (st > most) st = most;
        if (st > 8) st = 8;
        if (st < 1) st = 1;
    }
    p.stages = (int)st;
    p.smem_bytes = hdr + p.x_bytes + (size_t)warps * (size_t)p.stages * slot;
    const int64_t m = U / GW;  // shortest warp range
    int64_t slots = m >= 1 ? (ncb + m - 1) / m + 1 : ncb;
    if (slots > ncb) slots = ncb;
    p.max_slots = (int)slots;
    p.ws_counters = ((size_t)nrb * 4 + 255) / 256 * 256;
    // (no smaller than sk_box_bytes(tok) with a row block for every CTA: two slots per row block at least)
    p.ws_bytes = ncb > 1 ? p.ws_counters + (size_t)nrb * (size_t)slots * 16 * (size_t)tok * 4 : 0;
    return p;
}

struct StreamArgs {
    const unsigned char* packed;   // tiled codes
    const unsigned char* scales;   // tiled scales
    const unsigned char* zeros;    // tiled zero-points (uniform twin)
    const uint16_t* X;             // FP16 or BF16 bit patterns
    uint16_t* Y;
    float* partial;
    unsigned* counters;
    int64_t N, K;
    uint32_t units, gw_total;      // U, grid * W
    int ncb, group, stages, x_bytes, max_slots, M;
    int token_shift;               // log2 of the token slots of the staged activations
    int fits32;                    // U * gw_total < 2^32: 32-bit range arithmetic
    int aligned, nrb;              // row-block split (see the kernel), number of row blocks
};
// What only the decode without the scale reads (a type of its own: with twelve more words the parameters of
// stream_kernel_by_value no longer fit in its registers).
struct StreamArgsUnscaled : StreamArgs {
    uint32_t bias;                       // potl::POT_UNIT_BIAS
    uint32_t p2[potl::POT_UNIT_SHIFTS];  // p2[n] = 2^n
    uint32_t zeros_at;                   // shared-memory offset of SK_ZERO_BYTES that are cleared (one group per unit: any that are free)
    uint32_t factors_at;                 // BF16: shared-memory offset of one FP32 factor per unit
};
// ... and only the even split
struct StreamArgsEven : StreamArgsUnscaled {
    uint32_t cta_blocks, cta_more;  // blocks of sk_block(q) units per CTA; the first cta_more CTAs have one more
    uint32_t ncb_mul;               // u / ncb = (u * ncb_mul) >> ncb_shift for u < 2^31
    int ncb_shift;
};
template <bool UNSC>
using StreamKernelArgs = typename std::conditional<UNSC, StreamArgsUnscaled, StreamArgs>::type;

#ifdef __CUDACC__
__device__ __forceinline__ void sk_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void sk_mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                            uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// FP32 sum -> 16-bit output pattern (DT = 0: FP16, 1: BF16), round to nearest even
template <int DT>
__device__ __forceinline__ uint16_t sk_out(float v) {
    if (DT == 0) return __half_as_ushort(__float2half_rn(v));
    return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}
__device__ __forceinline__ uint32_t sk_lds32(const unsigned char* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ uint4 sk_lds128(const unsigned char* p) { return *reinterpret_cast<const uint4*>(p); }
// Eight BF16 numbers -> FP16 numbers relative to the largest one of the half-warp's unit (brought to 2^15 .. 2^16: BF16's largest
// significand stays below FP16's).  Returns the factor that undoes it, negative if one of the unit's numbers might not be exact: not
// zero and a subnormal FP16 number or less, 2^-30 of the largest one; the unit then stays as it is.  All 32 lanes take part; !ok: the lane
// holds nothing.
__device__ __forceinline__ float sk_normalize(uint4& v, bool ok) {
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
    auto bf2 = [](uint32_t b) { return *reinterpret_cast<const __nv_bfloat162*>(&b); };
    __nv_bfloat162 top = __habs2(bf2(w[0]));
#pragma unroll
    for (int i = 1; i < 4; ++i) top = __hmax2(top, __habs2(bf2(w[i])));  // (the maximum of a number and a NaN is the number)
    uint32_t m = *reinterpret_cast<const uint32_t*>(&top);
    m = max(m & 0xFFFFu, m >> 16);
    if (!ok || m > 0x7F80u) m = 0;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const uint32_t up = min(269u - max(m >> 7, 1u), 253u);  // exponent field of the inverse of the factor (253: both are normal numbers)
    const float f = __uint_as_float(up << 23), back = __uint_as_float((254u - up) << 23);
    uint32_t inexact = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 h = __floats2half2_rn(__uint_as_float(w[i] << 16) * f, __uint_as_float(w[i] & 0xFFFF0000u) * f);
        inexact |= __hlt2_mask(__habs2(h), __float2half2_rn(6.103515625e-5f)) & __hne2_mask(bf2(w[i]), __float2bfloat162_rn(0.f));
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    const uint32_t lanes = __ballot_sync(0xffffffffu, ok && inexact != 0);
    if (lanes & ((threadIdx.x & 16) ? 0xFFFF0000u : 0xFFFFu)) return -back;
    v = make_uint4(w[0], w[1], w[2], w[3]);
    return back;
}
// floor(a * b / c) for a * b that may need 64 bits
__device__ __forceinline__ uint32_t sk_muldiv(uint32_t a, uint32_t b, uint32_t c, bool fits32) {
    if (fits32) return (a * b) / c;
    return (uint32_t)(((uint64_t)a * (uint64_t)b) / (uint64_t)c);
}

// One unit the way of BF16 operands, of which all BF16 numbers are exact: the lane's codes decoded under their scales, x (64 bytes apart, in
// shared memory) as it came.  Returns the sums of rows gid and gid + 8.  Accumulators of its own, as the FP16 way has: in an MMA what
// stands in the accumulator loses the bits that lie below the largest product, which cancels in such a unit as like as not.
template <int BITS>
__device__ __forceinline__ float2 sk_unit_bf16(const unsigned char* code, const unsigned char* scale, const unsigned char* x) {
    const uint32_t scw = sk_lds32(scale);
    uint32_t w[2][BITS], lo[16], hi[16];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < BITS; ++k) w[h][k] = sk_lds32(code + k * 256 + h * 128);
    const __nv_bfloat162 sc = __float22bfloat162_rn(__half22float2(*reinterpret_cast<const __half2*>(&scw)));
    const uint32_t sb = *reinterpret_cast<const uint32_t*>(&sc);
    potl::pot_decode32_bf16<BITS, 1>(w[0], 0, __byte_perm(sb, 0, 0x1010), lo);
    potl::pot_decode32_bf16<BITS, 1>(w[1], 0, __byte_perm(sb, 0, 0x3232), hi);
    float c[2][4] = {};  // (two: half the length of the dependent chain)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 v = sk_lds128(x + 64 * i);
        sk_mma_bf16(c[0], lo[4 * i], hi[4 * i], lo[4 * i + 1], hi[4 * i + 1], v.x, v.y);
        sk_mma_bf16(c[1], lo[4 * i + 2], hi[4 * i + 2], lo[4 * i + 3], hi[4 * i + 3], v.z, v.w);
    }
    return make_float2(c[0][0] + c[1][0], c[0][2] + c[1][2]);
}
// Out of line, for the two-CTA builds, whose registers are few (inlined it cost them spills, and launches without such units 1 - 4 %).
template <int BITS>
__device__ __noinline__ float2 sk_unit_bf16_call(const unsigned char* code, const unsigned char* scale, const unsigned char* x) {
    return sk_unit_bf16<BITS>(code, scale, x);
}
// ---- what both streaming kernels do with a unit and with the activations
// The activations of a launch to shared memory (xs), in the order in which the MMA loop reads them, and what goes with them; behind_loads() is called once by
// every warp, behind its first loads.  True: BF16 numbers of this thread's are not FP16 numbers times their unit's factor.
template <int TOK, int W, bool UNSC, bool FACTORS, class Args, class Hook>
__device__ __forceinline__ bool sk_stage_x(const Args& sa, unsigned char* smem, unsigned char* xs, float* factors, Hook&& behind_loads) {
    bool inexact = false;
    uint4* dst = reinterpret_cast<uint4*>(xs);
    const uint4* src = reinterpret_cast<const uint4*>(sa.X);
    const int kc = (int)(sa.K / 8);  // 16-byte chunks per token
    if constexpr (UNSC && TOK == 1)
        if (threadIdx.x < SK_ZERO_BYTES / 16) *reinterpret_cast<uint4*>(smem + sa.zeros_at + threadIdx.x * 16) = make_uint4(0, 0, 0, 0);
    if constexpr (TOK == 1) {
        // chunk (quarter t, part j) of a unit goes to position j * 4 + t: lanes tig = 0..3 read 64 contiguous bytes
        // (four loads in flight per thread before the first store: one round trip for K <= 32 * 32 W)
        // (a bound for whole warps, here and below: 0.5 - 0.8 % of an eight-layer token in the two-CTA build)
        if ((int)(threadIdx.x & ~31u) >= kc) behind_loads();  // (a warp that loads nothing)
        for (int i0 = threadIdx.x; (i0 & ~31) < kc; i0 += 4 * W * 32) {
            uint4 v[4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (i0 + p * W * 32 < kc) v[p] = ld_dependent16(src + i0 + p * W * 32);
            if (i0 == threadIdx.x) behind_loads();
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int i = i0 + p * W * 32;
                if constexpr (FACTORS) {  // lanes 0-15 and 16-31 hold one unit each
                    const float f = sk_normalize(v[p], i < kc);
                    inexact = inexact || (i < kc && f < 0.f);
                    if (i < kc && (i & 15) == 0) factors[i >> 4] = f * potl::POT_UNIT_SCALE;
                }
                if (i < kc) dst[(i & ~15) | ((i & 3) << 2) | ((i >> 2) & 3)] = v[p];
            }
        }
    } else {
        // T = 2, 4 or 8 token slots (the smallest that holds M).  Chunk (token, unit, quarter t, part j) goes to
        // 16-byte slot (unit * 4 + j) * 4 T + (token / 2) * 8 + (token % 2) * 4 + t: the eight lanes of a quarter-warp
        // of the MMA loop (tokens 2q and 2q + 1, quarters 0..3) read one 128-byte line, a warp 4 lines -- no bank
        // conflict (token-major slots cost four-way conflicts: 11 against 8 us in the loop at 5+ tokens).  With fewer
        // than 8 slots the MMA columns beyond T repeat the first T tokens; they are never delivered, like the
        // tokens >= M.  The threads are numbered so that a quarter-warp also STORES one line: t fastest, then the
        // token's parity, then j -- a warp loads the 256 contiguous bytes of a unit for two tokens.
        const int ts = sa.token_shift;
        const int total = kc << ts;
        if ((int)(threadIdx.x & ~31u) >= total) behind_loads();
        for (int e0 = threadIdx.x; (e0 & ~31) < total; e0 += 8 * W * 32) {  // eight loads in flight per thread
            uint4 v[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const int e = e0 + p * W * 32;
                const int t = e & 3, par = (e >> 2) & 1, j = (e >> 3) & 3, hi = (e >> 5) & ((1 << (ts - 1)) - 1), unit_ = e >> (4 + ts);
                const int token = (hi << 1) | par;
                if (e < total && token < sa.M) v[p] = ld_dependent16(src + (int64_t)token * kc + unit_ * 16 + t * 4 + j);
            }
            if (e0 == threadIdx.x) behind_loads();
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const int e = e0 + p * W * 32;
                const int t = e & 3, par = (e >> 2) & 1, j = (e >> 3) & 3, hi = (e >> 5) & ((1 << (ts - 1)) - 1), unit_ = e >> (4 + ts);
                const int token = (hi << 1) | par;
                if (e < total && token < sa.M) dst[(((unit_ << 2) + j) << (2 + ts)) + (hi << 3) + (par << 2) + t] = v[p];
            }
        }
    }
    return inexact;
}
// One unit of PoT codes -> this lane's 32 half2 of the A fragments
template <int BITS, int DT, bool UNSC, class Args>
__device__ __forceinline__ void sk_decode_pot(const Args& sa, const unsigned char* code, const unsigned char* param, int spg, int lane, int gid, int tig, uint32_t (&lo)[16], uint32_t (&hi)[16]) {
    // the scale words {row gid, row gid + 8} of this lane's group
    const uint32_t poff = ((spg == 2 ? (uint32_t)(tig >> 1) * 8u : 0u) + (uint32_t)gid) * 4u;
    // plane k of a unit holds word k of every (row, quarter): this lane's word sits at byte 4 * lane
    uint32_t w[2][BITS];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < BITS; ++k) w[h][k] = sk_lds32(code + (uint32_t)(k * 256 + h * 128) + (uint32_t)lane * 4u);
    if constexpr (UNSC) {
        potl::pot_units32<BITS>(w[0], sa.p2, sa.bias, lo);
        potl::pot_units32<BITS>(w[1], sa.p2, sa.bias, hi);
        return;
    }
    const uint32_t scw = sk_lds32(param + poff);  // {row gid, row gid + 8}
    if constexpr (DT == 0) {
        potl::pot_decode32<BITS, 1>(w[0], 0, __byte_perm(scw, 0, 0x1010), lo);
        potl::pot_decode32<BITS, 1>(w[1], 0, __byte_perm(scw, 0, 0x3232), hi);
    } else {  // the FP16 scale rounded once to BF16
        const uint32_t s0 = __bfloat16_as_ushort(__float2bfloat16_rn(__half2float(__ushort_as_half((uint16_t)(scw & 0xFFFFu)))));
        const uint32_t s1 = __bfloat16_as_ushort(__float2bfloat16_rn(__half2float(__ushort_as_half((uint16_t)(scw >> 16)))));
        potl::pot_decode32_bf16<BITS, 1>(w[0], 0, s0 * 0x10001u, lo);
        potl::pot_decode32_bf16<BITS, 1>(w[1], 0, s1 * 0x10001u, hi);
    }
}
// ... a decoded unit times its activations: eight MMAs, and without the scale in the codes the scale after them.  xcol, xstep: this lane's column of B (GEMV)
template <int TOK, bool XSMEM, int DT, bool UNSC, bool FACTORS, class Args>
__device__ __forceinline__ void sk_multiply(const Args& sa, const uint32_t (&lo)[16], const uint32_t (&hi)[16], const unsigned char* param, uint32_t cbu, int spg, int gid, int tig,
                                            const unsigned char* xs, const unsigned char* xcol, uint32_t xstep, const float* factors, float (&acc)[2][4]) {
    // activations of quarter tig (of token gid): the B fragments of the eight MMAs
    uint32_t xq[16];
    if constexpr (XSMEM) {
        const unsigned char* xa = TOK == 1 ? xcol + cbu * xstep
                                           : xs + ((((cbu * 16u) << sa.token_shift) + ((((uint32_t)gid & ((1u << sa.token_shift) - 1u)) >> 1) << 3) +
                                                    (((uint32_t)gid & 1u) << 2) + (uint32_t)tig) << 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint4 v = sk_lds128(xa + (TOK == 1 ? 64u : (64u << sa.token_shift)) * i);
            xq[4 * i + 0] = v.x; xq[4 * i + 1] = v.y; xq[4 * i + 2] = v.z; xq[4 * i + 3] = v.w;
        }
    } else {
        const bool live = TOK == 1 || gid < sa.M;
        const uint4* xp = reinterpret_cast<const uint4*>(sa.X) + (TOK == 1 || !live ? 0 : (int64_t)gid * (sa.K / 8)) +
                          (int64_t)cbu * 16 + tig * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint4 v = make_uint4(0, 0, 0, 0);
            if (live) v = ld_dependent16(xp + i);
            xq[4 * i + 0] = v.x; xq[4 * i + 1] = v.y; xq[4 * i + 2] = v.z; xq[4 * i + 3] = v.w;
        }
    }
    if constexpr (UNSC) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 8; ++j) sk_mma(c, lo[2 * j], hi[2 * j], lo[2 * j + 1], hi[2 * j + 1], xq[2 * j], xq[2 * j + 1]);
        const uint32_t scw = sk_lds32(param + ((spg == 2 ? (uint32_t)(tig >> 1) * 8u : 0u) + (uint32_t)gid) * 4u);  // {row gid, row gid + 8}
        float2 sc = __half22float2(*reinterpret_cast<const __half2*>(&scw));
        if constexpr (!FACTORS) {
            acc[0][0] = fmaf(c[0], sc.x, acc[0][0]);
            acc[0][2] = fmaf(c[2], sc.y, acc[0][2]);
            if constexpr (TOK > 1) {
                acc[0][1] = fmaf(c[1], sc.x, acc[0][1]);
                acc[0][3] = fmaf(c[3], sc.y, acc[0][3]);
            }
        } else {  // the FP16 scale rounded once to BF16; times the unit's factor last, so that no product leaves FP32's range early
            sc = __bfloat1622float2(__float22bfloat162_rn(sc));
            const float f = factors[cbu];
            acc[0][0] = fmaf(c[0] * sc.x, f, acc[0][0]);
            acc[0][2] = fmaf(c[2] * sc.y, f, acc[0][2]);
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)  // two accumulators: half the length of the dependent chain
        if constexpr (DT == 0) sk_mma(acc[j & 1], lo[2 * j], hi[2 * j], lo[2 * j + 1], hi[2 * j + 1], xq[2 * j], xq[2 * j + 1]);
        else sk_mma_bf16(acc[j & 1], lo[2 * j], hi[2 * j], lo[2 * j + 1], hi[2 * j + 1], xq[2 * j], xq[2 * j + 1]);
}

// DT = 0: FP16 activations, weights and output; DT = 1: BF16 (PoT codes only: the scale is rounded once to BF16 and the
// exponent is added at bit 7).
// KIND: SK_POT / SK_UINT.  TOK = 1: GEMV (x in every B column).  TOK = 8: up to 8 tokens, one per B column.
// XSMEM: the activations are staged in shared memory in fragment order (else they are read through L1 from global).
// W consumer warps per CTA; OCC = 2 leaves room for a second CTA on the SM (64 registers per thread, half the shared
// memory), so that the next launch in the stream can become resident and fill its rings while this one still computes.
// UNSC: the codes are decoded without their scale (pot_units32) and a unit's FP32 sums are multiplied by it.  With two groups per
// unit (G = 64, GEMV only) columns 0-3 of B hold x of the first group's quarters and zeros for the others, columns 4-7 the
// opposite, so that the two groups' sums come out in different lanes.  BF16: FP16 codes cannot meet BF16 numbers in one MMA, and the
// decode to BF16 costs 41 instead of 25 logic operations per 32 codes, so that x is staged as FP16 numbers relative to the largest of
// 128 columns -- where that is exact.  A unit where it might not be (see sk_normalize) is marked, x stays BF16 there, and its codes are
// decoded to BF16 under their scale; only chunks that hold a marked unit leave the straight-line code.  us, all units decoded under
// the scale -> no / one / every eighth / every unit marked: 28672 x 8192, 4 bits, 37.5 -> 28.3 / 29.2 / 32.1 / 38.8; 8192 x 28672, 3 bits, 37.3 -> 30.7 / 31.6 /
// 34.7 / 40.0; with two CTAs per SM 12288 x 4096, 3 bits, 10.5 -> 9.5 / 10.2 / 11.6 / 13.3, 11008 x 4096, 4 bits, 9.9 -> 9.0 / 9.7 / 10.6 / 13.5.  (A loop for whole
// launches of marked units beside this one, x turned back: 11.7 instead of 13.5, but spills, and 2 - 4 % where no unit is marked.)
template <int BITS, int KIND, int TOK, bool XSMEM, int W, int OCC, int SK_Q, int DT, bool UNSC>
__device__ __forceinline__ void stream_body(const StreamKernelArgs<UNSC>& sa, int* __restrict__ err) {
    constexpr int UB = sk_unit_bytes(BITS);
    constexpr bool UNIFORM = (KIND == SK_UINT);
    constexpr int NPARAM = UNIFORM ? 2 : 1;
    static_assert(!UNSC || (!UNIFORM && XSMEM && (DT == 0 || TOK == 1)), "the decode without the scale: PoT codes, x in shared memory, BF16 one token");
    constexpr bool FACTORS = UNSC && DT == 1;
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = lane >> 2, tig = lane & 3;  // MMA fragment coordinates: rows gid and gid + 8, quarter tig
    const int S = sa.stages;
    const int spg = 128 / sa.group;
    const uint32_t PB = 32u * (uint32_t)spg;                 // parameter bytes of one unit
    const uint32_t slot_bytes = SK_Q * (UB + NPARAM * PB);
    const uint32_t smem0 = smem_u32(smem);
    const uint32_t bars = smem0 + (uint32_t)warp * 64u;      // this warp's full barriers (S <= 8)
    constexpr int HDR = sk_header_bytes(W, TOK);
    // Values a warp needs only when it requests a chunk or delivers sums live in shared memory, not in registers (the
    // two-CTAs-per-SM build has 64 registers per thread): [0] a, [1] n, [2] first row block, [3] last row block,
    // [4] slot of the first segment, [5] contributors of the first segment, [6] of the last, [7] bit 0 / 1: the first / last
    // segment is combined inside the CTA
    uint32_t* wst = reinterpret_cast<uint32_t*>(smem + W * 64) + warp * 8;
    unsigned* lcnt = reinterpret_cast<unsigned*>(smem + W * 96);               // local arrival counters
    float* lslots = reinterpret_cast<float*>(smem + W * 96 + W * 4);           // [warp][first, last][16 TOK]
    const unsigned char* xs = smem + HDR;
    const unsigned char* ringp = xs + sa.x_bytes + (uint32_t)warp * (uint32_t)S * slot_bytes;  // this warp's ring
    const uint32_t ring = smem0 + (uint32_t)HDR + (uint32_t)sa.x_bytes + (uint32_t)warp * (uint32_t)S * slot_bytes;

    // ---- this warp's range of units [a, b) ---------------------------------------------------------------
    // Unit split (sa.aligned == 0): the U units are cut into GW equal ranges, warp gw = blockIdx * W + warp takes range gw.
    // Row-block split (sa.aligned == 1): CTA c takes the row blocks [c nrb / grid, (c + 1) nrb / grid) and its W warps
    // cut that range of units into W equal ranges -- no row block is shared between CTAs.
    const bool f32 = sa.fits32 != 0;
    uint32_t base = 0, U = sa.units, GW = sa.gw_total, gw = blockIdx.x * W + warp;
    if (sa.aligned) {
        const uint32_t r0 = sk_muldiv(blockIdx.x, (uint32_t)sa.nrb, gridDim.x, f32), r1 = sk_muldiv(blockIdx.x + 1, (uint32_t)sa.nrb, gridDim.x, f32);
        base = r0 * (uint32_t)sa.ncb;
        U = (r1 - r0) * (uint32_t)sa.ncb;
        GW = W;
        gw = (uint32_t)warp;
    }
    const uint32_t a = base + (gw < GW ? sk_muldiv(gw, U, GW, f32) : 0u), b = base + (gw < GW ? sk_muldiv(gw + 1, U, GW, f32) : 0u);
    const uint32_t n = b - a;
    const uint32_t nchunks = (n + SK_Q - 1) / SK_Q;

    // chunk j of the range holds units [a + Q j, a + Q j + Q) (fewer at the end) and lives in slot j % S
    auto issue = [&](uint32_t a_, uint32_t n_, uint32_t j, uint32_t s) {  // one lane: request chunk j into slot s
        const uint32_t left_j = n_ - j * SK_Q;
        const uint32_t cnt = left_j < (uint32_t)SK_Q ? left_j : (uint32_t)SK_Q;
        const uint32_t bar = bars + s * 8u, dst = ring + s * slot_bytes;
        const size_t u0 = (size_t)a_ + (size_t)j * SK_Q;
        if (!in_range(s < (uint32_t)S && u0 + cnt <= sa.units && cnt >= 1 && cnt <= (uint32_t)SK_Q, err, 0x110)) return;
        mbar_expect_tx(bar, cnt * (UB + NPARAM * PB));
        bulk_g2s(dst, sa.packed + u0 * UB, cnt * UB, bar);
        bulk_g2s(dst + SK_Q * UB, sa.scales + u0 * PB, cnt * PB, bar);
        if constexpr (UNIFORM) bulk_g2s(dst + SK_Q * (UB + PB), sa.zeros + u0 * PB, cnt * PB, bar);
    };
    if (lane < S) {  // lane s sets up slot s and requests chunk s: the weights do not depend on the predecessor
        mbar_init(bars + (uint32_t)lane * 8u, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if ((uint32_t)lane < nchunks) issue(a, n, (uint32_t)lane, (uint32_t)lane);
    }
    __syncwarp();
    pdl_launch_dependents();

    // ---- row blocks of the range; which of its segments are partial, and their place among the contributors
    const uint32_t ncb = (uint32_t)sa.ncb;
    uint32_t rb = a / ncb, cb = a - rb * ncb;
    const uint32_t rb0 = rb, rbL = n ? (b - 1) / ncb : rb;
    uint32_t slot0 = 0, exp0 = 0, expL = 0;  // exp == 0: the segment covers its whole row block
    auto owner = [&](uint32_t u) {  // the warp (numbered like gw) whose range holds unit u
        u -= base;
        return f32 ? ((u + 1) * GW - 1) / U : (uint32_t)((((uint64_t)u + 1) * GW - 1) / U);
    };
    if (n) {
        if (cb != 0 || b < (rb0 + 1) * ncb) {
            const uint32_t lo = owner(rb0 * ncb), hi = owner((rb0 + 1) * ncb - 1);
            slot0 = gw - lo;
            exp0 = hi - lo + 1;
        }
        if (rbL != rb0 && b != (rbL + 1) * ncb) expL = owner((rbL + 1) * ncb - 1) - gw + 1;  // this warp is its first contributor
    }
    // a row block whose contributors all sit in this CTA is combined in shared memory
    const uint32_t cta_lo = sa.aligned ? 0u : blockIdx.x * W;
    const bool loc0 = exp0 && gw - slot0 >= cta_lo && gw - slot0 + exp0 <= cta_lo + W;
    const bool locL = expL && gw + expL <= cta_lo + W;
    if (lane == 0) {
        wst[0] = a; wst[1] = n; wst[2] = rb0; wst[3] = rbL;
        wst[4] = slot0; wst[5] = exp0; wst[6] = expL; wst[7] = (loc0 ? 1u : 0u) | (locL ? 2u : 0u);
    }
    if (threadIdx.x < W) lcnt[threadIdx.x] = 0u;

    pdl_wait();  // x, Y and the workspace may belong to the previous kernel in the stream
    float* factors = nullptr;  // BF16 without the scale: one per unit
    if constexpr (FACTORS) factors = reinterpret_cast<float*>(smem + sa.factors_at);
    bool inexact = false;
    if constexpr (XSMEM) {
        inexact = sk_stage_x<TOK, W, UNSC, FACTORS>(sa, smem, smem + HDR, factors, [] {});
    }
    if constexpr (FACTORS) inexact = __syncthreads_or(inexact);
    else __syncthreads();

    float acc[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;

    // ---- delivery of the sums of rows [16 rb, 16 rb + 16) accumulated so far ---------------------------------
    auto deliver = [&](uint32_t rbd) {
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[e] = acc[0][e] + acc[1][e];
            acc[0][e] = 0.f;
            acc[1][e] = 0.f;
        }
        if constexpr (UNSC) {
            if constexpr (TOK == 1) {
                if (spg == 2) {  // the second group's sums sit in lanes tig = 2, 3
                    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
                    v[2] += __shfl_xor_sync(0xffffffffu, v[2], 2);
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if constexpr (!FACTORS) v[e] *= potl::POT_UNIT_SCALE;
        }
        const bool first = rbd == wst[2];
        const uint32_t expect = first ? wst[5] : (rbd == wst[3] ? wst[6] : 0u);
        const uint32_t slot = first ? wst[4] : 0u;
        const int64_t row0 = (int64_t)rbd * 16;
        if (expect == 0) {
            if constexpr (TOK == 1) {
                if (tig == 0 && in_range(row0 + gid + 8 < sa.N, err, 0x120)) {
                    sa.Y[row0 + gid] = sk_out<DT>(v[0]);
                    sa.Y[row0 + gid + 8] = sk_out<DT>(v[2]);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int token = 2 * tig + (e & 1);
                    if (token < sa.M && in_range(row0 + gid + 8 * (e >> 1) < sa.N, err, 0x121))
                        sa.Y[(int64_t)token * sa.N + row0 + gid + 8 * (e >> 1)] = sk_out<DT>(v[e]);
                }
            }
            return;
        }
        if ((wst[7] >> (first ? 0 : 1)) & 1u) {
            // slot of warp w: [w][1] if w is the row block's first contributor, else [w][0]
            const uint32_t wl = (uint32_t)warp - slot;  // first contributor (local warp index)
            if (!in_range(slot <= (uint32_t)warp && wl + expect <= (uint32_t)W && row0 + 16 <= sa.N, err, 0x130)) return;
            float* mine = lslots + ((size_t)warp * 2 + (slot == 0 ? 1 : 0)) * (16 * TOK);
            if constexpr (TOK == 1) {
                if (tig == 0) {
                    mine[gid] = v[0];
                    mine[gid + 8] = v[2];
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) mine[(2 * tig + (e & 1)) * 16 + gid + 8 * (e >> 1)] = v[e];
            }
            __threadfence_block();
            __syncwarp();
            unsigned prev = 0;
            if (lane == 0) prev = atomicAdd(&lcnt[wl], 1u);
            prev = __shfl_sync(0xffffffffu, prev, 0);
            if (prev == expect - 1u) {
                __threadfence_block();
                for (int e = lane; e < 16 * (TOK == 1 ? 1 : sa.M); e += 32) {
                    float sum = 0.f;
                    for (uint32_t q = 0; q < expect; ++q) sum += lslots[((size_t)(wl + q) * 2 + (q == 0 ? 1 : 0)) * (16 * TOK) + e];
                    sa.Y[(int64_t)(e >> 4) * sa.N + row0 + (e & 15)] = sk_out<DT>(sum);
                }
            }
            return;
        }
        if (!in_range(rbd < (uint32_t)sa.nrb && slot < (uint32_t)sa.max_slots && expect <= (uint32_t)sa.max_slots && sa.partial != nullptr,
                      err, 0x140))
            return;
        float* base = sa.partial + ((size_t)rbd * (size_t)sa.max_slots) * (16 * TOK);
        float* mine = base + (size_t)slot * (16 * TOK);
        if constexpr (TOK == 1) {
            if (tig == 0) {
                mine[gid] = v[0];
                mine[gid + 8] = v[2];
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int token = 2 * tig + (e & 1);
                if (token < sa.M) mine[token * 16 + gid + 8 * (e >> 1)] = v[e];
            }
        }
        __threadfence();
        __syncwarp();
        // Arrivals are counted down: the first one finds zero, or more than the counter can hold, and puts expect - 1 there, the last one finds one and leaves
        // zero.  So a counter need not be zero before the call: from row block 64 on it lies where a product of more tokens on the same matrix
        // (gemm_prefill.cu) leaves FP32 partial sums.  As whole numbers these are larger than any count (38 there), but for sums from 2^-149 to 38 x 2^-149,
        // which no FP16 product has, and a BF16 one only of activations some 2^-100 times the usual ones.
        // (A sign that no sum can have, raised by a second atomic operation: 2048 x 8192 6.7 -> 7.3 us; bytes in the first 64 words as counters: 7.6.)
        unsigned prev = 0;
        if (lane == 0) prev = atomicDec(&sa.counters[rbd], expect - 1u);
        prev = __shfl_sync(0xffffffffu, prev, 0);
        if (prev == 1u) {  // this warp delivered the last slot of the row block: add them in ascending order
            __threadfence();
            for (int e = lane; e < 16 * (TOK == 1 ? 1 : sa.M); e += 32) {
                float sum = 0.f;
                for (uint32_t q = 0; q < expect; ++q) sum += __ldcg(base + (size_t)q * (16 * TOK) + e);
                sa.Y[(int64_t)(e >> 4) * sa.N + row0 + (e & 15)] = sk_out<DT>(sum);
            }
        }
    };

    // ---- one unit: 2 x 32 codes of this lane -> 32 half2 (decode: needs no activations) -> eight MMAs (multiply) ----
    auto unit_ok = [&](const unsigned char* code, const unsigned char* param, uint32_t cbu) {
        return in_range(code >= ringp && code + UB <= ringp + (size_t)S * slot_bytes && param + NPARAM * PB <= ringp + (size_t)S * slot_bytes &&
                            cbu < ncb && (!XSMEM || ((size_t)(cbu + 1) * 256u << sa.token_shift) <= (size_t)sa.x_bytes),
                        err, 0x150);
    };
    auto decode = [&](const unsigned char* code, const unsigned char* param, uint32_t (&lo)[16], uint32_t (&hi)[16]) {
        if constexpr (!UNIFORM) {
            sk_decode_pot<BITS, DT, UNSC>(sa, code, param, spg, lane, gid, tig, lo, hi);
        } else {
            // the scale words {row gid, row gid + 8} of this lane's group
            const uint32_t poff = ((spg == 2 ? (uint32_t)(tig >> 1) * 8u : 0u) + (uint32_t)gid) * 4u;
            // the quarter's words sit at record words 2 tig, 2 tig + 1 (n = 2), 2 tig, 2 tig + 1, 8 + tig (n = 3) or
            // 4 tig .. 4 tig + 3 (n = 4); record word w is byte (w / 4) * 256 + row * 16 + (w % 4) * 4
            const uint32_t scw = sk_lds32(param + poff);
            const uint32_t zw = sk_lds32(param + SK_Q * PB + poff);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t q[BITS == 3 ? 9 : BITS];
#pragma unroll
                for (int k = 0; k < BITS; ++k) {
                    const int wi = BITS == 4 ? 4 * tig + k : (k < 2 ? 2 * tig + k : 8 + tig);
                    q[(BITS == 3 && k == 2) ? 8 : k] =
                        sk_lds32(code + (uint32_t)((wi >> 2) * 256 + (wi & 3) * 4 + h * 128) + (uint32_t)gid * 16u);
                }
                potl::UintParams pr;
                pr.s2 = potl::bits_h2(__byte_perm(scw, 0, h ? 0x3232 : 0x1010));
                pr.z = potl::bits_h2(__byte_perm(zw, 0, h ? 0x3232 : 0x1010));
                uint32_t a8[8], b8[8];
                potl::uint_decode_pairs16<BITS>(q, 0, pr, a8);
                potl::uint_decode_pairs16<BITS>(q, 1, pr, b8);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    (h ? hi : lo)[i] = a8[i];
                    (h ? hi : lo)[8 + i] = b8[i];
                }
            }
        }
    };
    // this lane's column of B (GEMV): x, or zeros if the column belongs to the other group
    auto zeros = [&]() -> const unsigned char* {
        if constexpr (UNSC) return smem + sa.zeros_at;
        else return xs;
    };
    const bool zero_column = UNSC && TOK == 1 && spg == 2 && (gid >> 2) != (tig >> 1);
    const unsigned char* xcol = zero_column ? zeros() + tig * 16 : xs + tig * 16;
    const uint32_t xstep = zero_column ? 0u : 256u;
    auto multiply = [&](const uint32_t (&lo)[16], const uint32_t (&hi)[16], const unsigned char* param, uint32_t cbu) {
        sk_multiply<TOK, XSMEM, DT, UNSC, FACTORS>(sa, lo, hi, param, cbu, spg, gid, tig, xs, xcol, xstep, factors, acc);
    };
    auto unit = [&](const unsigned char* code, const unsigned char* param, uint32_t cbu) {
        if (!unit_ok(code, param, cbu)) return;
        uint32_t lo[16], hi[16];
        decode(code, param, lo, hi);
        multiply(lo, hi, param, cbu);
    };
    // a unit whose activations are not FP16 numbers times one factor
    auto unit_bf16 = [&](const unsigned char* code, const unsigned char* param, uint32_t cbu) {
        if (!unit_ok(code, param, cbu)) return;
        const unsigned char* sp = param + ((spg == 2 ? (uint32_t)(tig >> 1) * 8u : 0u) + (uint32_t)gid) * 4u;
        float2 v;
        if constexpr (OCC == 2) v = sk_unit_bf16_call<BITS>(code + (uint32_t)lane * 4u, sp, xcol + cbu * xstep);
        else v = sk_unit_bf16<BITS>(code + (uint32_t)lane * 4u, sp, xcol + cbu * xstep);
        acc[0][0] += v.x;
        acc[0][2] += v.y;
    };
    // ---- main loop over this warp's chunks; MARKS: x has marked units.  False: a copy never arrived -----------------------------
    // (Two loops: with the marks looked for in the one that most launches run these took 2 - 4 % longer.)
    auto main_loop = [&](auto marks) -> bool {
        constexpr bool MARKS = decltype(marks)::value;
        uint32_t s = 0, phase = 0, left = n;
        for (uint32_t j = 0; left > 0; ++j) {
            const unsigned char* code = ringp + s * slot_bytes;
            const unsigned char* param = code + SK_Q * UB;
            const uint32_t bar = bars + s * 8u;
            if (!mbar_test(bar, phase) && !mbar_wait(bar, phase)) {
                // Record it, request nothing more, deliver nothing more (the rows this warp still owed stay unwritten: the error
                // word says so), wait -- bounded again -- for the chunks already requested, leave.
                if (err && lane == 0) atomicCAS(err, 0, 2 | (int)(j << 8) | (warp << 24));
                uint32_t s2 = s, ph2 = phase;
                for (uint32_t k = 1; k < (uint32_t)S && (j + k) * SK_Q < wst[1]; ++k) {
                    if (++s2 == (uint32_t)S) {
                        s2 = 0;
                        ph2 ^= 1u;
                    }
                    mbar_wait(bars + s2 * 8u, ph2);
                }
                return false;
            }
            const bool full = left >= (uint32_t)SK_Q && cb + (uint32_t)SK_Q <= ncb;
            bool some = false, all = MARKS;  // some, all units of a full chunk are marked
            if constexpr (MARKS) {
                if (full) {
#pragma unroll
                    for (int i = 0; i < SK_Q; ++i) {
                        const bool m = factors[cb + i] < 0.f;
                        some = some || m;
                        all = all && m;
                    }
                }
            }
            if (full && !some) {
                // the common case: a full chunk inside one row block, straight-line code
#pragma unroll
                for (int i = 0; i < SK_Q; ++i) unit(code + i * UB, param + (uint32_t)i * PB, cb + (uint32_t)i);
                cb += SK_Q;
                left -= SK_Q;
                if (cb == ncb) {
                    deliver(rb);
                    cb = 0;
                    ++rb;
                }
            } else if (MARKS && OCC == 1 && full && all) {
                if constexpr (MARKS) {
#pragma unroll
                    for (int i = 0; i < SK_Q; ++i) unit_bf16(code + i * UB, param + (uint32_t)i * PB, cb + (uint32_t)i);
                }
                cb += SK_Q;
                left -= SK_Q;
                if (cb == ncb) {
                    deliver(rb);
                    cb = 0;
                    ++rb;
                }
            } else {
                const uint32_t cnt = left < (uint32_t)SK_Q ? left : (uint32_t)SK_Q;
                for (uint32_t i = 0; i < cnt; ++i) {
                    if constexpr (MARKS) {
                        if (factors[cb] < 0.f) unit_bf16(code, param, cb);
                        else unit(code, param, cb);
                    } else {
                        unit(code, param, cb);
                    }
                    code += UB;
                    param += PB;
                    if (++cb == ncb) {
                        deliver(rb);
                        cb = 0;
                        ++rb;
                    }
                }
                left -= cnt;
            }
            __syncwarp();  // every lane has read the slot: it may be refilled
            if (lane == 0 && (j + (uint32_t)S) * SK_Q < wst[1]) issue(wst[0], wst[1], j + (uint32_t)S, s);
            if (++s == (uint32_t)S) {
                s = 0;
                phase ^= 1u;
            }
        }
        return true;
    };
    if (FACTORS && inexact) {
        if constexpr (FACTORS)
            if (!main_loop(std::true_type())) return;
    } else {
        if (!main_loop(std::false_type())) return;
    }
    if (n && cb != 0) deliver(rb);
}

template <int BITS, int KIND, int TOK, bool XSMEM, int W, int OCC, int SK_Q, int DT, bool UNSC>
__global__ void __launch_bounds__(W * 32, OCC) stream_kernel(const __grid_constant__ StreamKernelArgs<UNSC> sa, int* __restrict__ err) {
    stream_body<BITS, KIND, TOK, XSMEM, W, OCC, SK_Q, DT, UNSC>(sa, err);
}
// The same with the parameters by value, for the uniform twin at 2 bits: read from constant memory they cost its two-CTA build
// (64 registers) spills of 96 / 112 bytes, 4096 x 4096 4.2 -> 5.7 us, 12288 x 4096 9.6 -> 12.2 us.  At 3 bits constant memory is 3 %
// the faster one (14.1 -> 13.7 us), at 4 bits between 3 % slower and 2 % faster.
template <int BITS, int KIND, int TOK, bool XSMEM, int W, int OCC, int SK_Q, int DT, bool UNSC>
__global__ void __launch_bounds__(W * 32, OCC) stream_kernel_by_value(const StreamArgs sa, int* __restrict__ err) {
    stream_body<BITS, KIND, TOK, XSMEM, W, OCC, SK_Q, DT, UNSC>(sa, err);
}
template <int BITS, int KIND, int TOK, bool XSMEM, int W, int OCC, int SK_Q, int DT, bool UNSC>
constexpr auto stream_kernel_of() {
    if constexpr (KIND == SK_UINT && BITS == 2) return stream_kernel_by_value<BITS, KIND, TOK, XSMEM, W, OCC, SK_Q, DT, UNSC>;
    else return stream_kernel<BITS, KIND, TOK, XSMEM, W, OCC, SK_Q, DT, UNSC>;
}
#endif  // __CUDACC__

}  // namespace pot
#include "stream_even.cuh"
namespace pot {

// ---- host side --------------------------------------------------------------------------------------------
inline StreamArgs stream_args(const StreamPlan& p, const void* packed, const void* scales, const void* zeros, int64_t N,
                              int64_t K, int group, const void* X, int M, void* Y, void* workspace) {
    StreamArgs sa;
    sa.packed = (const unsigned char*)packed;
    sa.scales = (const unsigned char*)scales;
    sa.zeros = (const unsigned char*)zeros;
    sa.X = (const uint16_t*)X;
    sa.Y = (uint16_t*)Y;
    sa.counters = (unsigned*)workspace;
    sa.partial = workspace ? (float*)((char*)workspace + p.ws_counters) : nullptr;
    sa.N = N;
    sa.K = K;
    sa.units = p.units;
    sa.gw_total = p.gw_total;
    sa.aligned = p.aligned ? 1 : 0;
    sa.nrb = p.nrb;
    sa.ncb = p.ncb;
    sa.group = group;
    sa.stages = p.stages;
    sa.x_bytes = (int)p.x_bytes;
    sa.max_slots = p.max_slots;
    sa.M = M;
    sa.token_shift = p.token_shift;
    sa.fits32 = ((uint64_t)p.units + 1) * ((uint64_t)sa.gw_total + 1) < (uint64_t(1) << 32) ? 1 : 0;
    return sa;
}

#ifdef __CUDACC__
template <int BITS, int KIND, int TOK, int W, int OCC = 1, int DT = 0>
pot_status_t launch_stream(const void* packed, const void* scales, const void* zeros, int64_t N, int64_t K, int group,
                           const void* X, int M, void* Y, void* workspace, int* err, cudaStream_t s) {
    const StreamPlan p = plan_stream(N, K, M, BITS, group, KIND, TOK, W, OCC, DT);
    if (!p.ok) return POT_ERR_SHAPE;
    StreamArgsUnscaled args;
    static_cast<StreamArgs&>(args) = stream_args(p, packed, scales, zeros, N, K, group, X, M, Y, workspace);
    args.bias = potl::POT_UNIT_BIAS;
    // (cleared whether needed or not: a condition in the kernel cost 0.7 % of an eight-layer token with G = 64.  With one group per
    // unit that is the start of the slots of partial sums, which are written after the prologue's barrier)
    args.zeros_at = group == 64 ? (uint32_t)sk_header_bytes(W, TOK) + (uint32_t)K * 2 : (uint32_t)W * 100;
    static_assert(W * 2 * 16 * TOK * 4 >= SK_ZERO_BYTES && W * 100 % 16 == 0, "the zeros fit into the partial-sum slots");
    for (int i = 0; i < potl::POT_UNIT_SHIFTS; ++i) args.p2[i] = 1u << i;
    args.factors_at = (uint32_t)sk_header_bytes(W, TOK) + (uint32_t)K * 2u + (group == 64 ? SK_ZERO_BYTES : 0);
    auto run = [&](auto kernel) -> pot_status_t {
        auto launch = [&](const auto& a) { return launch_pdl_cluster(kernel, dim3((unsigned)p.grid), dim3(W * 32), p.smem_bytes, 1, true, s, a, err); };
        if constexpr (std::is_same<decltype(kernel), void (*)(StreamArgs, int*)>::value) return launch(static_cast<const StreamArgs&>(args));
        else return launch(args);
    };
    constexpr bool POT = KIND == SK_POT;
    auto pick = [&](auto q) -> pot_status_t {  // q units per slot
        constexpr int Q = decltype(q)::value;
        if constexpr (POT) {
            if (p.even) {
                StreamArgsEven even;
                static_cast<StreamArgsUnscaled&>(even) = args;
                if (group == 128) even.zeros_at = (uint32_t)sk_even_slots_at(W);
                even.cta_blocks = p.cta_blocks;
                even.cta_more = p.cta_more;
                even.ncb_shift = 31;  // (Granlund and Montgomery 1994, "Division by invariant integers using multiplication")
                while ((int64_t(1) << (even.ncb_shift - 31)) < p.ncb) ++even.ncb_shift;
                even.ncb_mul = (uint32_t)(((uint64_t(1) << even.ncb_shift) + (uint64_t)p.ncb - 1) / (uint64_t)p.ncb);
                auto run_even = [&](auto kernel) -> pot_status_t {
                    return launch_pdl_cluster(kernel, dim3((unsigned)p.grid), dim3(W * 32), p.smem_bytes, 1, true, s, even, err);
                };
                if constexpr (TOK > 1)  // (more than four tokens come here only with their activations in shared memory)
                    if (M > 4 && p.x_in_smem) {
                        if constexpr (DT == 0)
                            if (p.unscaled) return run_even(stream_even_kernel<BITS, TOK, true, W, OCC, Q, DT, true, true>);
                        return run_even(stream_even_kernel<BITS, TOK, true, W, OCC, Q, DT, false, true>);
                    }
                if constexpr (DT == 0 || TOK == 1)
                    if (p.unscaled) return run_even(stream_even_kernel<BITS, TOK, true, W, OCC, Q, DT, true>);
                if constexpr (!(DT == 0 && TOK == 1))
                    if (p.x_in_smem) return run_even(stream_even_kernel<BITS, TOK, true, W, OCC, Q, DT, false>);
                if constexpr (OCC == 1 && Q == 2) return run_even(stream_even_kernel<BITS, TOK, false, W, OCC, Q, DT, false>);
                else return POT_ERR_SHAPE;
            }
        }
        if constexpr (POT && (DT == 0 || TOK == 1))
            if (p.unscaled) return run(stream_kernel_of<BITS, KIND, TOK, true, W, OCC, Q, DT, true>());
        if constexpr (!(POT && DT == 0 && TOK == 1))
            if (p.x_in_smem) return run(stream_kernel_of<BITS, KIND, TOK, true, W, OCC, Q, DT, false>());
        // (x that does not fit in shared memory leaves no room for longer slots, and is never planned with two CTAs per SM)
        if constexpr (OCC == 1 && Q == 2) return run(stream_kernel_of<BITS, KIND, TOK, false, W, OCC, Q, DT, false>());
        else return POT_ERR_SHAPE;
    };
    if (p.q == 2) return pick(std::integral_constant<int, 2>());
    if constexpr (OCC == 1 && TOK == 1)
        if (p.q == 8) return pick(std::integral_constant<int, 8>());
    return pick(std::integral_constant<int, SK_QMAX>());
}
#endif

}  // namespace pot
