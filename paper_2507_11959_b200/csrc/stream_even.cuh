// The streaming kernel of stream.cuh with the units dealt out evenly to the CTAs (PoT codes; plan_stream says where).  As there: warps with rings of
// their own, decode, MMAs.  Different: which units a warp works on, and the way of the sums.
//
// CTA c takes the blocks of units c * cta_blocks + min(c, cta_more) .., as much as every other CTA but for one block.  A range that begins
// inside a row block begins with a part that the CTA before has the rest of.  All warps work on this part first, and its sums are left in the
// workspace for that CTA, which adds them to its own when it has come to its end -- or the other way round, where a CTA starts late: the
// second one adds.  No CTA waits for another.  Then the warps cut up the other units.  Row blocks that warps share are added up in shared
// memory by the last one that delivers; the order of additions is fixed.
// What bounds it: as in stream.cuh.  What the split takes away is the unequal ends: of whole row blocks (28672 x 8192: 16 CTAs have 13 row blocks, 132
// have 12), of a row block's many contributors (unit split).  Where the kernel has an SM to itself nothing hides its launch: it asks for one
// chunk per warp, then for the activations, then for the rest of the ring (with all chunks first the activations arrive behind them:
// 28672 x 8192 24.3 us, so 23.1), and divisions by the number of column blocks are multiplications (the ranges took 1200 cycles).  Before -> after:
// 28672 x 8192 25.0 -> 23.1 us (3 bits), 28.2 -> 28.0 (4 bits, BF16, G = 64), 5120 x 13824 12.4 -> 11.4, 2400 x 8192 6.9 -> 5.95, 4 tokens x 15360 x 5120 13.4 -> 12.6.
#pragma once
#include "stream.cuh"

#ifdef __CUDACC__
namespace pot {

__device__ __forceinline__ void st_relaxed64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long exch_relaxed64(unsigned long long* p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.exch.relaxed.gpu.global.b64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}
// A sum on its way from CTA to CTA: the number in the lower half, a mark in the upper one.  What else may lie there is zero or the partial sums of a
// product of more tokens (gemm_prefill.cu), pairs of FP32 numbers.  The mark is a signaling NaN, which no operation returns, and not PF_NO_SUM.
constexpr uint32_t SK_SUM_MARK = 0x7F95C0DEu;
__device__ __forceinline__ unsigned long long sk_marked_sum(float v) { return ((unsigned long long)SK_SUM_MARK << 32) | __float_as_uint(v); }
__device__ __forceinline__ bool sk_is_sum(unsigned long long v) { return (uint32_t)(v >> 32) == SK_SUM_MARK; }
// shared-memory header: as sk_header_bytes, with four words between the local arrival counters and the slots of partial sums
__host__ __device__ constexpr int sk_even_counters_at(int warps) { return warps * 96; }
__host__ __device__ constexpr int sk_even_slots_at(int warps) { return warps * 100 + 16; }

// Template parameters as of stream_kernel; MANY: more than four tokens.
template <int BITS, int TOK, bool XSMEM, int W, int OCC, int SK_Q, int DT, bool UNSC, bool MANY = false>
__global__ void __launch_bounds__(W * 32, OCC) stream_even_kernel(const __grid_constant__ StreamArgsEven sa, int* __restrict__ err) {
    constexpr int UB = sk_unit_bytes(BITS);
    static_assert(!UNSC || (XSMEM && (DT == 0 || TOK == 1)), "the decode without the scale: x in shared memory, BF16 one token");
    constexpr bool FACTORS = UNSC && DT == 1;
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = lane >> 2, tig = lane & 3;  // MMA fragment coordinates: rows gid and gid + 8, quarter tig
    const int S = sa.stages;
    const int spg = 128 / sa.group;
    const uint32_t PB = 32u * (uint32_t)spg;                 // parameter bytes of one unit
    const uint32_t slot_bytes = SK_Q * (UB + PB);
    const uint32_t smem0 = smem_u32(smem);
    const uint32_t bars = smem0 + (uint32_t)warp * 64u;      // this warp's full barriers (S <= 8)
    constexpr int HDR = sk_header_bytes(W, TOK);
    static_assert(sk_even_slots_at(W) + W * 2 * 16 * TOK * 4 <= HDR && sk_even_slots_at(W) % 16 == 0 && SK_ZERO_BYTES <= W * 2 * 16 * TOK * 4, "the header holds it");
    // What a warp needs only when it requests a chunk or delivers sums: [0] first unit, [1] number of units of its own range; [2], [3] the same of its
    // part of the CTA's first row block; [4] first, [5] last row block of its range; [6] the warps of the CTA that share the first (lower half)
    // and the last (upper half) of these; [7] number of chunks
    uint32_t* wst = reinterpret_cast<uint32_t*>(smem + W * 64) + warp * 8;
    // local arrival counters; [W] the same of the CTA's part of its first row block, [W + 1] its sums have been added up, [W + 2] the warps that
    // have a part, [W + 3] the row block that the next CTA has a part of
    unsigned* lcnt = reinterpret_cast<unsigned*>(smem + sk_even_counters_at(W));
    float* lslots = reinterpret_cast<float*>(smem + sk_even_slots_at(W));           // [warp][first, last][16 TOK]
    const unsigned char* xs = smem + HDR;
    const unsigned char* ringp = xs + sa.x_bytes + (uint32_t)warp * (uint32_t)S * slot_bytes;  // this warp's ring
    const uint32_t ring = smem0 + (uint32_t)HDR + (uint32_t)sa.x_bytes + (uint32_t)warp * (uint32_t)S * slot_bytes;

    // ---- this warp's ranges ----------------------------------------------------------------------------------
    const uint32_t ncb = (uint32_t)sa.ncb;
    constexpr uint32_t BLOCK = sk_block(SK_Q);
    auto div_ncb = [&](uint32_t u) { return (uint32_t)(((uint64_t)u * sa.ncb_mul) >> sa.ncb_shift); };
    auto part = [&](uint32_t blocks, uint32_t w) { return w * (blocks / W) + min(w, blocks % W); };
    const uint32_t base = (blockIdx.x * sa.cta_blocks + min(blockIdx.x, sa.cta_more)) * BLOCK;  // the CTA's units
    const uint32_t units = min(base + (sa.cta_blocks + (blockIdx.x < sa.cta_more ? 1u : 0u)) * BLOCK, sa.units) - base;
    const uint32_t first_rb = div_ncb(base), inside = base - first_rb * ncb;
    const uint32_t lead = inside ? ncb - inside : 0u, rest = units - lead;                      // ... of a row block that the CTA before began; the others
    const uint32_t lead_blocks = (lead + BLOCK - 1) / BLOCK, all_blocks = lead_blocks + (rest + BLOCK - 1) / BLOCK;
    const uint32_t l0 = part(lead_blocks, warp), l1 = part(lead_blocks, warp + 1);
    const uint32_t la = base + min(l0 * BLOCK, lead), ln = base + min(l1 * BLOCK, lead) - la;
    const uint32_t a = base + lead + min((part(all_blocks, warp) - l0) * BLOCK, rest);
    const uint32_t n = base + lead + min((part(all_blocks, warp + 1) - l1) * BLOCK, rest) - a;
    const uint32_t lchunks = (ln + SK_Q - 1) / SK_Q, nchunks = lchunks + (n + SK_Q - 1) / SK_Q;

    // chunk j holds units [a + Q j, a + Q j + Q) (fewer at the end) and lives in slot j % S; the part of the shared row block comes first
    auto issue = [&](uint32_t a_, uint32_t n_, uint32_t la_, uint32_t ln_, uint32_t j, uint32_t s) {  // one lane: request chunk j into slot s
        const uint32_t lc = (ln_ + SK_Q - 1) / SK_Q, jj = j < lc ? j : j - lc;
        const uint32_t u0 = (j < lc ? la_ : a_) + jj * SK_Q, left_j = (j < lc ? ln_ : n_) - jj * SK_Q;
        const uint32_t cnt = left_j < (uint32_t)SK_Q ? left_j : (uint32_t)SK_Q;
        const uint32_t bar = bars + s * 8u, dst = ring + s * slot_bytes;
        if (!in_range(s < (uint32_t)S && (uint64_t)u0 + cnt <= sa.units && cnt >= 1 && cnt <= (uint32_t)SK_Q, err, 0x110)) return;
        mbar_expect_tx(bar, cnt * (UB + PB));
        bulk_g2s(dst, sa.packed + (size_t)u0 * UB, cnt * UB, bar);
        bulk_g2s(dst + SK_Q * UB, sa.scales + (size_t)u0 * PB, cnt * PB, bar);
    };
    constexpr bool late = OCC == 1 && XSMEM;   // only the first chunk before the activations
    if (lane < S) {  // lane s sets up slot s and requests chunk s: the weights do not depend on the predecessor
        mbar_init(bars + (uint32_t)lane * 8u, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    auto request = [&](uint32_t from, uint32_t to) {
        if ((uint32_t)lane >= from && (uint32_t)lane < to && lane < S && (uint32_t)lane < nchunks) issue(a, n, la, ln, (uint32_t)lane, (uint32_t)lane);
    };
    // Two CTAs per SM: this one's first copies, 100 KB, would be in the way of the activations that the one beside it, of the launch before, is
    // just waiting for.  us with this pause / without it / without it and with all but the first chunk behind the activations: eight layers of
    // 3200 / 8576 240.1 / 247.3 / 243.7, of 2048 / 5504 226.3 / 222.2 / 226.2, of 2816 / 7040 202.2 / 203.8 / 204.3, of 2560 / 6912 at 2 bits 171.5 /
    // 174.1 / 176.6.  Behind another kernel, which does not let this one in early, it is lost time: 2480 x 4096 6.7 / 6.2 / 6.3 (unit split 8.0),
    // 7136 x 4096 10.2 / 9.7 / 9.3 (11.4), 5120 x 13824 16.0 / 15.5 / 14.6 (16.4).  A pause that ends with the previous kernel: 240 -> 238 and 226
    // -> 228, but 2480 x 2048 at 2 bits 2.8 -> 3.1; with both orders in one launch the chains took 1 - 4 % longer.
    if constexpr (OCC == 2) __nanosleep(1000);
    request(0, late ? 1u : 8u);
    __syncwarp();
    pdl_launch_dependents();

    // ---- row blocks of the range; which of its segments are partial, and their place among the contributors
    uint32_t rb = 0, cb = 0;
    auto row_blocks = [&]() {
        const uint32_t start = base + lead, r1 = first_rb + (lead ? 1u : 0u), m0 = a - start;
        const uint32_t q0 = div_ncb(m0), qL = n ? div_ncb(m0 + n - 1) : q0, full = div_ncb(rest);
        rb = r1 + q0;
        cb = m0 - q0 * ncb;
        // the warps whose ranges touch the first and the last row block of this one's
        const uint32_t w = min((uint32_t)lane, (uint32_t)W - 1u);
        const uint32_t f = min((part(all_blocks, w) - part(lead_blocks, w)) * BLOCK, rest), e = min((part(all_blocks, w + 1) - part(lead_blocks, w + 1)) * BLOCK, rest);
        const uint32_t m_first = __ballot_sync(0xffffffffu, lane < W && f < e && f < (q0 + 1) * ncb && e > q0 * ncb);
        const uint32_t m_last = __ballot_sync(0xffffffffu, lane < W && f < e && f < (qL + 1) * ncb && e > qL * ncb);
        if (lane == 0) {
            wst[0] = a; wst[1] = n; wst[2] = la; wst[3] = ln; wst[4] = rb; wst[5] = r1 + qL;
            wst[6] = m_first | (m_last << 16);
        }
        if (threadIdx.x == 0) {
            lcnt[W + 2] = 0xFFFFu >> (16u - min(lead_blocks, (uint32_t)W));
            lcnt[W + 3] = rest != full * ncb ? r1 + full : 0xffffffffu;
        }
        static_assert(W <= 16, "sets of warps in 16 bits");
        if (lane == 0) wst[7] = nchunks;
        if (threadIdx.x < W + 2) lcnt[threadIdx.x] = 0u;
    };
    // Two CTAs per SM: this one waits anyway.  One: its predecessor on the SM has gone, and so, most of the time, has the previous kernel;
    // the activations are asked for first.
    if (!late) row_blocks();
    [[maybe_unused]] auto behind_loads = [&]() {
        if (late) {
            request(1, 8);
            row_blocks();
        }
    };

    pdl_wait();  // x, Y and the workspace may belong to the previous kernel in the stream
    float* factors = nullptr;  // BF16 without the scale: one per unit
    if constexpr (FACTORS) factors = reinterpret_cast<float*>(smem + sa.factors_at);
    bool inexact = false;
    if constexpr (XSMEM) {
        inexact = sk_stage_x<TOK, W, UNSC, FACTORS>(sa, smem, smem + HDR, factors, behind_loads);
    }
    if constexpr (FACTORS) inexact = __syncthreads_or(inexact);
    else __syncthreads();

    float acc[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;

    // ---- delivery of the sums of rows [16 rb, 16 rb + 16) accumulated so far ---------------------------------
    auto deliver = [&](uint32_t rbd, bool shared_first) {
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
        const int64_t row0 = (int64_t)rbd * 16;
        auto store = [&]() {
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
        };
        // the warps of this CTA that have a part of the row block; whether the next CTA has one
        const uint4 mine4 = *reinterpret_cast<const uint4*>(wst + 4), cta4 = *reinterpret_cast<const uint4*>(lcnt + W);
        const bool next_cta = !shared_first && rbd == cta4.w;
        const uint32_t sharers = shared_first ? cta4.z : (rbd == mine4.x ? mine4.z & 0xFFFFu : (rbd == mine4.y ? mine4.z >> 16 : 1u << warp));
        if (!shared_first && !next_cta && (sharers & (sharers - 1u)) == 0) {
            store();
            return;
        }
        // slot of warp w: [w][1] if w is the row block's first contributor, else [w][0]; the shared first row block, which is done before a
        // warp begins with its own range: [w][0]
        const uint32_t wl = (uint32_t)__ffs(sharers) - 1u, wh = 31u - (uint32_t)__clz(sharers);
        const bool begins = !shared_first && (uint32_t)warp == wl;
        if (!in_range(row0 + 16 <= sa.N && ((sharers >> warp) & 1u) && wh < (uint32_t)W && (!(shared_first || next_cta) || sa.counters != nullptr), err, 0x131)) return;
        if (!shared_first && !begins && wst[3] != 0) {  // [w][0] may still hold sums of the shared row block
            volatile unsigned* taken = lcnt + W + 1;
            uint32_t i = 0;
            while (*taken == 0 && ++i < kSpinLimit) {}
            __syncwarp();
            if (__any_sync(0xffffffffu, i >= kSpinLimit)) {
                if (err && lane == 0) atomicCAS(err, 0, 3 | (warp << 24));
                return;
            }
        }
        float* mine = lslots + ((size_t)warp * 2 + (begins ? 1 : 0)) * (16 * TOK);
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
        if (lane == 0) prev = atomicAdd(&lcnt[shared_first ? (uint32_t)W : wl], 1u);
        prev = __shfl_sync(0xffffffffu, prev, 0);
        if (prev != (unsigned)__popc(sharers) - 1u) return;
        __threadfence_block();
        // Where two CTAs have sums of the row block, the one that finds the other's in the workspace adds the two (in either order the same number),
        // and clears them for the next call.  Neither waits for the other, which may not have started (another stream's kernel on its SM).
        // A bounded wait of the first CTA and a plain store in the second were as fast but for 0 - 0.5 us where a launch has an SM to
        // itself (2400 x 8192 5.45 -> 5.84 us on one GPU, 5.96 -> 5.98 on another; 28672 x 8192 23.0, 5120 x 13824 11.4, both).
        if constexpr (!MANY) {
            for (int e = lane; e < 16 * (TOK == 1 ? 1 : sa.M); e += 32) {
                const float* at = lslots + e;
                float sum = at[(wl * 2u + (shared_first ? 0u : 1u)) * (16 * TOK)];
                for (uint32_t w = wl + 1; w <= wh; w += 4) {  // (four loads at a time; a warp between them that has no part of the row block adds nothing)
                    float p[4];
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u) p[u] = at[min(w + u, wh) * 2u * (16 * TOK)];
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u)
                        if (w + u <= wh && ((sharers >> (w + u)) & 1u)) sum += p[u];
                }
                if (shared_first || next_cta) {
                    unsigned long long* box = reinterpret_cast<unsigned long long*>(sa.counters) + (size_t)(blockIdx.x + (next_cta ? 1u : 0u)) * (16 * TOK) + e;
                    unsigned long long got = shared_first ? 0ull : ld_relaxed64(box);  // (the CTA after this one is nearly always the first)
                    if (!sk_is_sum(got)) got = exch_relaxed64(box, sk_marked_sum(sum));
                    if (!sk_is_sum(got)) continue;
                    st_relaxed64(box, 0ull);
                    sum += __uint_as_float((uint32_t)got);
                }
                sa.Y[(int64_t)(e >> 4) * sa.N + row0 + (e & 15)] = sk_out<DT>(sum);
            }
        } else {
            // Three or four sums per lane: all requests are on their way before the first answer is looked at (in the loop above 5 - 8 tokens take 4 - 10 %
            // longer, 6 x 3552 x 5888 10.9 us, so 9.95, and on some matrices longer than with the unit split; one or two sums are the loop's: 2
            // tokens 2 - 5 %, 4 tokens 1 %, and an instantiation of its own because both in one took them 1 - 2 % longer).
            static_assert(TOK > 1, "several tokens");
            constexpr int R = TOK / 2;
            const int last = 16 * sa.M;
            float sum[R];
            uint32_t done = 0;  // bit r: sum r is complete
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (lane + 32 * r >= last) continue;
                const float* at = lslots + lane + 32 * r;
                sum[r] = at[(wl * 2u + (shared_first ? 0u : 1u)) * (16 * TOK)];
                for (uint32_t w = wl + 1; w <= wh; w += 4) {
                    float p[4];
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u) p[u] = at[min(w + u, wh) * 2u * (16 * TOK)];
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u)
                        if (w + u <= wh && ((sharers >> (w + u)) & 1u)) sum[r] += p[u];
                }
                done |= 1u << r;
            }
            if (shared_first || next_cta) {
                unsigned long long* box = reinterpret_cast<unsigned long long*>(sa.counters) + (size_t)(blockIdx.x + (next_cta ? 1u : 0u)) * (16 * TOK) + lane;
                unsigned long long got[R];
#pragma unroll
                for (int r = 0; r < R; ++r) got[r] = !shared_first && ((done >> r) & 1u) ? ld_relaxed64(box + 32 * r) : 0ull;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (((done >> r) & 1u) && !sk_is_sum(got[r])) got[r] = exch_relaxed64(box + 32 * r, sk_marked_sum(sum[r]));
                done = 0;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (lane + 32 * r < last && sk_is_sum(got[r])) {
                        st_relaxed64(box + 32 * r, 0ull);
                        sum[r] += __uint_as_float((uint32_t)got[r]);
                        done |= 1u << r;
                    }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int e = lane + 32 * r;
                if ((done >> r) & 1u) sa.Y[(int64_t)(e >> 4) * sa.N + row0 + (e & 15)] = sk_out<DT>(sum[r]);
            }
        }
        if (shared_first) {
            __threadfence_block();
            __syncwarp();
            if (lane == 0) *(volatile unsigned*)(lcnt + W + 1) = 1u;
        }
    };

    // ---- one unit: 2 x 32 codes of this lane -> 32 half2 (decode: needs no activations) -> eight MMAs (multiply) ----
    auto unit_ok = [&](const unsigned char* code, const unsigned char* param, uint32_t cbu) {
        return in_range(code >= ringp && code + UB <= ringp + (size_t)S * slot_bytes && param + PB <= ringp + (size_t)S * slot_bytes &&
                            cbu < ncb && (!XSMEM || ((size_t)(cbu + 1) * 256u << sa.token_shift) <= (size_t)sa.x_bytes),
                        err, 0x150);
    };
    auto decode = [&](const unsigned char* code, const unsigned char* param, uint32_t (&lo)[16], uint32_t (&hi)[16]) {
        sk_decode_pot<BITS, DT, UNSC>(sa, code, param, spg, lane, gid, tig, lo, hi);
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
        bool shared_first = ln != 0;  // (the part of the row block that the CTA before began)
        if (shared_first) {
            left = ln;
            rb = first_rb;
            cb = la - first_rb * ncb;
        }
        for (uint32_t j = 0; left > 0; ++j) {
            const unsigned char* code = ringp + s * slot_bytes;
            const unsigned char* param = code + SK_Q * UB;
            const uint32_t bar = bars + s * 8u;
            if (!mbar_test(bar, phase) && !mbar_wait(bar, phase)) {
                // Record it, request nothing more, deliver nothing more (the rows this warp still owed stay unwritten: the error
                // word says so), wait -- bounded again -- for the chunks already requested, leave.
                if (err && lane == 0) atomicCAS(err, 0, 2 | (int)(j << 8) | (warp << 24));
                uint32_t s2 = s, ph2 = phase;
                for (uint32_t k = 1; k < (uint32_t)S && j + k < wst[7]; ++k) {
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
                if (cb == ncb || left == 0) {
                    deliver(rb, shared_first);
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
                if (cb == ncb || left == 0) {
                    deliver(rb, shared_first);
                    cb = 0;
                    ++rb;
                }
            } else {
                const uint32_t cnt = left < (uint32_t)SK_Q ? left : (uint32_t)SK_Q;
                left -= cnt;
                for (uint32_t i = 0; i < cnt;) {
                    uint32_t step = 1;
                    if (BLOCK < SK_Q && !MARKS && i + BLOCK <= cnt && cb + BLOCK <= ncb) {
#pragma unroll
                        for (uint32_t u = 0; u < BLOCK; ++u) unit(code + u * UB, param + u * PB, cb + u);
                        step = BLOCK;
                    } else if constexpr (MARKS) {
                        if (factors[cb] < 0.f) unit_bf16(code, param, cb);
                        else unit(code, param, cb);
                    } else {
                        unit(code, param, cb);
                    }
                    code += step * UB;
                    param += step * PB;
                    i += step;
                    cb += step;
                    if (cb == ncb || (left == 0 && i == cnt)) {
                        deliver(rb, shared_first);
                        cb = 0;
                        ++rb;
                    }
                }
            }
            __syncwarp();  // every lane has read the slot: it may be refilled
            if (lane == 0 && j + (uint32_t)S < wst[7]) issue(wst[0], wst[1], wst[2], wst[3], j + (uint32_t)S, s);
            if (++s == (uint32_t)S) {
                s = 0;
                phase ^= 1u;
            }
            if (left == 0 && shared_first) {
                shared_first = false;
                left = wst[1];
                rb = wst[4];
                cb = wst[0] - rb * ncb;
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
}

}  // namespace pot
#endif
