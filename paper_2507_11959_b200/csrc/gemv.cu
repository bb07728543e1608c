// Batch-1 decode GEMV, y = W~ x, fused with the dequantization (the weights never touch HBM as FP16).
//
//  * tiled layout (the fast path): the streaming kernel of stream.cuh.  Every warp streams its own contiguous
//    range of 16-row x 128-column units through a private shared-memory ring (bulk copies), decodes the codes in
//    registers with the mask / shift / integer-add of Sec. 4.2 and feeds them, as A fragments, to warp-level
//    tensor-core MMAs whose B columns all hold x; row blocks that span warps are combined in a fixed order.
//  * canonical layout (any N): warps of 16 rows on the same MMAs, codes straight from global memory into registers and decoded
//    with byte look-ups; the uniform twin, and vectors too long for shared memory, run on CUDA cores with one warp per row, 8
//    codes per lane per step, products accumulated in FP32 with the mixed-precision FMA and reduced with warp shuffles.
//
// Programmatic dependent launch: weights and scales do not depend on the previous kernel in the stream, x does.
// The streaming kernel and the canonical kernel on the tensor cores request their first weights before they execute
// griddepcontrol.wait, and touch x, y and the workspace only after it; the one with a warp per row waits first.
#include "common.cuh"
#include "layout.cuh"
#include "stream.cuh"

namespace pot {

// two FP16 x FP16 products accumulated in FP32 (mixed-precision FMA: no conversion instructions)
__device__ __forceinline__ void rg_fma2(float& acc0, float& acc1, uint32_t w2, uint32_t x2) {
    asm("{\n\t"
        ".reg .b16 wl, wh, xl, xh;\n\t"
        "mov.b32 {wl, wh}, %2;\n\t"
        "mov.b32 {xl, xh}, %3;\n\t"
        "fma.rn.f32.f16 %0, wl, xl, %0;\n\t"
        "fma.rn.f32.f16 %1, wh, xh, %1;\n\t"
        "}"
        : "+f"(acc0), "+f"(acc1)
        : "r"(w2), "r"(x2));
}


// ------------------------------------------------------------------------------------------
// canonical layout, one warp per row
// ------------------------------------------------------------------------------------------
// BF16 pairs: a BF16 number is the upper half of an FP32 pattern, so the conversions are a shift and a mask
__device__ __forceinline__ void rg_fma2_bf16(float& acc0, float& acc1, uint32_t w2, uint32_t x2) {
    acc0 = fmaf(__uint_as_float(w2 << 16), __uint_as_float(x2 << 16), acc0);
    acc1 = fmaf(__uint_as_float(w2 & 0xFFFF0000u), __uint_as_float(x2 & 0xFFFF0000u), acc1);
}

// DT = 0: FP16 activations / weights / output; DT = 1: BF16 (PoT only: scale rounded once to BF16, E added at bit 7)
template <int BITS, bool UNIFORM, int DT = 0>
__global__ void __launch_bounds__(256) gemv_canonical_kernel(const uint32_t* __restrict__ packed,
                                                             const uint16_t* __restrict__ scales,
                                                             const uint16_t* __restrict__ zeros, int64_t N, int64_t K,
                                                             int G, const uint4* __restrict__ x, uint16_t* __restrict__ y) {
    constexpr int EBIT = DT == 0 ? 10 : 7;
    constexpr uint32_t CM = (1u << BITS) - 1u;
    constexpr uint32_t QM2 = (uint32_t)qmax_of(BITS) * 0x10001u;
    constexpr uint32_t SM2 = (1u << (BITS - 1)) * 0x10001u;
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= N) return;
    const int64_t pieces = K / 8;
    const uint32_t* rowp = packed + row * (K * BITS / 32);
    const uint16_t* srow = scales + row * (K / G);
    const uint16_t* zrow = UNIFORM ? zeros + row * (K / G) : nullptr;
    float acc0 = 0.f, acc1 = 0.f;
    pdl_wait();
    for (int64_t c = lane; c < pieces; c += 32) {
        const uint32_t v = read_bits(rowp, c * (8 * BITS), 8 * BITS);
        uint32_t s16 = __ldg(srow + (c * 8) / G);
        if (DT == 1) s16 = __bfloat16_as_ushort(__float2bfloat16_rn(__half2float(__ushort_as_half((uint16_t)s16))));
        const uint4 xv = ld_dependent16(x + c);
        const uint32_t xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t t = v >> (2 * j * BITS);
            const uint32_t pr = (t & CM) | ((t << (16 - BITS)) & (CM << 16));
            uint32_t w2;
            if constexpr (!UNIFORM) {
                w2 = s16 * 0x10001u + (((pr & QM2) << EBIT) | ((pr & SM2) << (16 - BITS)));
            } else {
                const __half2 zm2 = __hadd2(__half2half2(__ushort_as_half(__ldg(zrow + (c * 8) / G))), __float2half2_rn(1024.0f));
                const uint32_t h = pr | 0x64006400u;
                const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), zm2);
                const __half2 w = __hmul2(d, __half2half2(__ushort_as_half((uint16_t)s16)));
                w2 = *reinterpret_cast<const uint32_t*>(&w);
            }
            if (DT == 0) rg_fma2(acc0, acc1, w2, xs[j]);
            else rg_fma2_bf16(acc0, acc1, w2, xs[j]);
        }
    }
    float acc = acc0 + acc1;
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) y[row] = sk_out<DT>(acc);
}

// ------------------------------------------------------------------------------------------
// canonical layout, PoT: 16 rows per warp on the tensor cores
// ------------------------------------------------------------------------------------------
// Lane (gid, tig) holds its part of the A fragments of m16n8k16 MMAs: rows gid and gid + 8.  The order of the K columns is
// free as long as A and B agree, so in a step of 512 columns lane tig takes the WHOLE column block 4 step + tig of its two rows:
// BITS 16-byte loads per row from contiguous memory, and each register is loaded for the next step as soon as it has been
// decoded.  x is staged in shared memory (272 bytes per column block: the four blocks that the lanes of a fragment read lie
// in different banks) and sits in every column of B; at 2 bits in the order in which the codes leave the words most cheaply.
// CTAs of eight warps, two per SM, or of four: while one of them finishes, another (of the next launch, too) sets itself up.  The steps of
// a row block are dealt to 1, 2, 4 or 8 warps of a CTA and, where few row blocks leave SMs idle, to the CTAs of a cluster; the sums are
// added in warp order, then in CTA order.  (One CTA of 16 warps per SM with a contiguous, equal share of the steps per warp was
// 5 - 20 % slower: its launches do not overlap.)
// Bound by instruction issue (16 rows x 128 columns: 70 - 110 instructions to decode, 8 MMAs, 12 loads) and by fixed latencies (launch,
// x).  HBM-cold, 10007 x 4096: 6.95 us at 2 bits, 9.25 us at 3, 10.5 us at 4 bits in BF16 (one warp per row on CUDA cores: 26.5,
// 31.9, 26.5 us); 4099 x 11008 at 3 bits: 36.1 -> 9.75 us.
constexpr int GC_WARPS = 8;                      // (or half as many)
constexpr int GC_X_STRIDE = 272;                 // bytes per staged column block
constexpr int64_t GC_MAX_K = 64 * 1024;          // x takes 136 KB at this length
struct CanonPlan { int wk_shift, warps, cluster; unsigned grid; };  // log2 of the warps per row block, warps per CTA, CTAs per row block
// Four warps per row block: CTAs of four warps with one row block, or of eight with two.  The small ones stage x twice as often and deal the
// row blocks out more finely: they win where an SM gets an odd number of them, which the large ones round up.  Back to back, eight ->
// four warps, us, FP16, 2 / 3 bits: 10500 x 4096 (five per SM) 9.0 / 11.7 -> 8.2 / 10.1, x 16384 25.5 / 34.8 -> 25.1 / 32.3; 16000 x 8192
// (seven) 18.8 / 24.9 -> 17.4 / 22.8; 2300 x 2944 (one) 3.4 / 4.4 -> 2.9 / 2.9.  An even number: 12000 x 16384 25.7 / 34.9 -> 28.8 / 36.9, 18900 x
// 8192 19.1 / 25.0 -> 19.5 / 25.4, 9472 x 8192 10.7 / 13.8 -> 11.5 / 14.6, 4099 x 2944 3.5 / 4.4 -> 4.0 / 4.4.  With more to decode and few columns
// the wait for the codes counts for more than x, and four warps win with even numbers too (3 bits: 12000 x 4096 11.8 -> 11.0, 9472 x
// 2944 8.2 -> 7.3).  At 2 bits three per SM depend on how they fall (K = 2944: 5000 rows 0.85 of the time, 6000 - 7000 rows 1.10), and on long
// rows there is nothing to gain (593 row blocks x 16384 1.04).  (x has to fit into shared memory four times: K <= 24576.)
static bool four_warp_ctas(int wk_shift, int64_t rbs, int64_t K, int bits) {
    if (wk_shift != 2 || K > 24 * 1024) return false;
    const int64_t per_sm = (rbs + kSmCount - 1) / kSmCount;
    if (bits == 2) return per_sm % 2 == 1 && per_sm != 3 && K <= 12 * 1024;
    return per_sm % 2 == 1 || (K <= 5 * 1024 && per_sm > 2);
}
static CanonPlan plan_canonical(int64_t N, int64_t K, int bits) {
    const int64_t rbs = (N + 15) / 16, steps = (K / 128 + 3) / 4;
    CanonPlan p{0, GC_WARPS, 1, 0};
    while (p.wk_shift < 3 && (rbs << p.wk_shift) < 2 * GC_WARPS * kSmCount && (2 << p.wk_shift) <= steps) ++p.wk_shift;
    while (p.cluster < 4 && p.wk_shift == 3 && rbs * p.cluster * 2 <= kSmCount && 2 * p.cluster * GC_WARPS <= steps) p.cluster *= 2;
    p.warps = four_warp_ctas(p.wk_shift, rbs, K, bits) ? GC_WARPS / 2 : GC_WARPS;
    const int64_t per_cta = p.warps >> p.wk_shift;
    p.grid = (unsigned)((rbs + per_cta - 1) / per_cta * p.cluster);
    return p;
}

// (CTAs per SM: as many as 128 registers leave; at 2 bits 102 registers are enough, and a fifth 4-warp CTA is worth 8.5 -> 8.2 us)
constexpr int gc_ctas_per_sm(int bits, int warps) { return warps == GC_WARPS ? 2 : (bits == 2 ? 5 : 4); }
template <int BITS, int DT, int W>
__global__ void __launch_bounds__(W * 32, gc_ctas_per_sm(BITS, W)) gemv_canonical_mma_kernel(const uint4* __restrict__ packed, const uint16_t* __restrict__ scales,
                                                                              int64_t N, int ncb, int spg, const uint4* __restrict__ x,
                                                                              uint16_t* __restrict__ y, int wk_shift, int cluster, int* __restrict__ err) {
    extern __shared__ __align__(16) unsigned char xs[];
    __shared__ float part[W][16];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = lane >> 2, tig = lane & 3;
    const int WK = 1 << wk_shift;
    const int crank = (int)blockIdx.x % cluster;
    const int64_t rb = (int64_t)(blockIdx.x / cluster) * (W >> wk_shift) + (warp >> wk_shift);
    const int64_t row0 = min(rb * 16 + gid, N - 1), row1 = min(rb * 16 + gid + 8, N - 1);  // (rows past the end repeat the last one and are not stored)
    const int steps = (ncb + 3) / 4, stride = WK * cluster;

    uint32_t w[2][4 * BITS], sc[2][2];
    const uint4* src[2];
    const uint16_t* ssrc[2];
    auto point = [&](int step) {  // the codes and scales of this lane's column block (a block past the end repeats the last one)
        const int cb = min(4 * step + tig, ncb - 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t block = (h ? row1 : row0) * ncb + cb;
            src[h] = packed + block * BITS;
            ssrc[h] = scales + block * spg;
        }
    };
    auto load_codes = [&](int t) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 q = __ldg(src[h] + t);
            w[h][4 * t + 0] = q.x; w[h][4 * t + 1] = q.y; w[h][4 * t + 2] = q.z; w[h][4 * t + 3] = q.w;
        }
    };
    auto load_scales = [&](int hb) {
#pragma unroll
        for (int h = 0; h < 2; ++h) sc[h][hb] = __ldg(ssrc[h] + (spg == 2 ? hb : 0));
    };
    const bool fits = in_range((uint32_t)(ncb + 1) * GC_X_STRIDE <= dynamic_smem_bytes() && WK <= W && crank < cluster, err, 0x160);
    int step = fits ? crank * WK + (warp & (WK - 1)) : steps;
    if (step < steps) {
        point(step);
#pragma unroll
        for (int t = 0; t < BITS; ++t) load_codes(t);
        load_scales(0);
        load_scales(1);
    }
    // x and y may belong to the previous kernel in the stream; the codes and scales do not, and are on their way (us, before -> behind the wait: 10007 x
    // 4096 at 2 / 3 / 4 bits 8.05 / 9.7 / 11.1 -> 6.95 / 9.25 / 10.5, 4099 x 11008 11.1 -> 9.75, 1001 x 4096 2.95 -> 2.45).  The next launch is let in
    // behind the wait: before it, CTAs of several launches share some SMs and leave others empty (4099 x 2944 6.4 us instead of 4.0).
    pdl_wait();
    pdl_launch_dependents();
    if constexpr (BITS == 2) {  // the order of canon_decode32_any
        for (int i = threadIdx.x; fits && i < ncb * 8; i += W * 32) {
            const uint4 a = ld_dependent16(x + 2 * i), b = ld_dependent16(x + 2 * i + 1);
            uint4* dst = reinterpret_cast<uint4*>(xs + (i >> 3) * GC_X_STRIDE + (i & 7) * 32);
            dst[0] = make_uint4(potl::prmt(a.x, a.y, 0x5410), potl::prmt(a.z, a.w, 0x5410), potl::prmt(b.x, b.y, 0x5410), potl::prmt(b.z, b.w, 0x5410));
            dst[1] = make_uint4(potl::prmt(a.x, a.y, 0x7632), potl::prmt(a.z, a.w, 0x7632), potl::prmt(b.x, b.y, 0x7632), potl::prmt(b.z, b.w, 0x7632));
        }
    } else {
        for (int i = threadIdx.x; fits && i < ncb * 16; i += W * 32)
            *reinterpret_cast<uint4*>(xs + (i >> 4) * GC_X_STRIDE + (i & 15) * 16) = ld_dependent16(x + i);
    }
    if (fits && threadIdx.x < 16) *reinterpret_cast<uint4*>(xs + ncb * GC_X_STRIDE + threadIdx.x * 16) = make_uint4(0, 0, 0, 0);  // x of the block past the end
    __syncthreads();

    float acc[2][4] = {};
    for (; step < steps; step += stride) {
        const unsigned char* xb = xs + min(4 * step + tig, ncb) * GC_X_STRIDE;
        const bool more = step + stride < steps;
        if (more) point(step + stride);
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) {
            uint32_t s0 = sc[0][hb], s1 = sc[1][hb];
            if (DT == 1) {
                s0 = __bfloat16_as_ushort(__float2bfloat16_rn(__half2float(__ushort_as_half((uint16_t)s0))));
                s1 = __bfloat16_as_ushort(__float2bfloat16_rn(__half2float(__ushort_as_half((uint16_t)s1))));
            }
            const potl::CanonLut<BITS, DT> lut0(s0), lut1(s1);
            if (more) load_scales(hb);
#pragma unroll
            for (int T = 2 * hb; T < 2 * hb + 2; ++T) {
                uint32_t lo[16], hi[16], xq[16];
                potl::canon_decode32_any<BITS, DT>(w[0] + T * BITS, lut0, lo);
                potl::canon_decode32_any<BITS, DT>(w[1] + T * BITS, lut1, hi);
                if (more) {  // the 16-byte pieces whose last word belongs to this quarter
#pragma unroll
                    for (int t = 0; t < BITS; ++t)
                        if ((4 * t + 3) / BITS == T) load_codes(t);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = *reinterpret_cast<const uint4*>(xb + T * 64 + i * 16);
                    xq[4 * i + 0] = v.x; xq[4 * i + 1] = v.y; xq[4 * i + 2] = v.z; xq[4 * i + 3] = v.w;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if constexpr (DT == 0) sk_mma(acc[j & 1], lo[2 * j], hi[2 * j], lo[2 * j + 1], hi[2 * j + 1], xq[2 * j], xq[2 * j + 1]);
                    else sk_mma_bf16(acc[j & 1], lo[2 * j], hi[2 * j], lo[2 * j + 1], hi[2 * j + 1], xq[2 * j], xq[2 * j + 1]);
            }
        }
    }
    if (tig == 0) {
        part[warp][gid] = acc[0][0] + acc[1][0];
        part[warp][gid + 8] = acc[0][2] + acc[1][2];
    }
    __syncthreads();
    // the first warp of a row block adds the sums of its warps, the first CTA of a cluster those of its CTAs
    float sum = 0.f;
    const bool first = (warp & (WK - 1)) == 0 && lane < 16;
    if (first)
        for (int q = 0; q < WK; ++q) sum += part[warp + q][lane];
    if (cluster > 1) {
        __syncthreads();
        if (first) part[warp][lane] = sum;
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        if (first && crank == 0)
            for (int z = 1; z < cluster; ++z) {
                uint32_t addr;
                float v;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_u32(&part[warp][lane])), "r"(z));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
                sum += v;
            }
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");  // the sums have been read
    }
    if (first && crank == 0 && rb * 16 + lane < N && in_range(fits && rb >= 0, err, 0x161)) y[rb * 16 + lane] = sk_out<DT>(sum);
}

// CTAs per SM of the streaming GEMV (16 consumer warps each).  Two: the next launch in the stream becomes resident,
// sets itself up and fills its rings while this one computes, which hides the launch and the prologue (about 2.5 us);
// the price is 64 registers per thread and half the ring, i.e. a slower loop (about 15 %).  Worth it while a CTA's
// share of the matrix is small; one CTA per SM otherwise, and whenever the half-size ring could not hold two slots.
constexpr size_t kTwoCtaMaxShare = 300 * 1024;  // bytes of codes + scales per CTA
static int gemv_occupancy(int64_t N, int64_t K, int bits, int group, int kind, int dt = 0) {
    const StreamPlan p2 = plan_stream(N, K, 1, bits, group, kind, 1, 16, 2, dt);
    if (!p2.ok || !p2.x_in_smem || p2.ring_capacity < 2 || p2.grid < kSmCount) return 1;
    const size_t share = (size_t)(N / 16) * (size_t)(K / 128) * (size_t)sk_unit_total_bytes(bits, group, kind) / (size_t)p2.grid;
    return share <= kTwoCtaMaxShare ? 2 : 1;
}

template <int KIND, int DT = 0>
static pot_status_t launch_gemv_stream(const void* packed, const void* scales, const void* zeros, int64_t N, int64_t K,
                                       int bits, int group, const void* x, void* y, void* workspace, cudaStream_t s) {
    int* err = error_ptr(ERR_GEMV);
#define POT_SG(B, O) return launch_stream<B, KIND, 1, 16, O, DT>(packed, scales, zeros, N, K, group, x, 1, y, workspace, err, s)
    if (gemv_occupancy(N, K, bits, group, KIND, DT) == 2) {
        if (bits == 2) POT_SG(2, 2);
        if (bits == 3) POT_SG(3, 2);
        POT_SG(4, 2);
    }
    if (bits == 2) POT_SG(2, 1);
    if (bits == 3) POT_SG(3, 1);
    POT_SG(4, 1);
#undef POT_SG
}

template <int DT>
static pot_status_t launch_gemv_canonical(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group,
                                          const void* x, void* y, cudaStream_t s) {
    if (K <= GC_MAX_K) {
        const CanonPlan p = plan_canonical(N, K, bits);
        auto run = [&](auto kernel) -> pot_status_t {
            const size_t smem = (size_t)(K / 128 + 1) * GC_X_STRIDE;
            return launch_pdl_cluster(kernel, dim3(p.grid), dim3((unsigned)p.warps * 32), smem, p.cluster, smem > 46 * 1024, s, (const uint4*)packed,
                                      (const uint16_t*)scales, N, (int)(K / 128), 128 / group, (const uint4*)x, (uint16_t*)y, p.wk_shift, p.cluster, error_ptr(ERR_GEMV));
        };
        auto pick = [&](auto w) -> pot_status_t {
            constexpr int W = decltype(w)::value;
            if (bits == 2) return run(gemv_canonical_mma_kernel<2, DT, W>);
            if (bits == 3) return run(gemv_canonical_mma_kernel<3, DT, W>);
            return run(gemv_canonical_mma_kernel<4, DT, W>);
        };
        return p.warps == GC_WARPS ? pick(std::integral_constant<int, GC_WARPS>()) : pick(std::integral_constant<int, GC_WARPS / 2>());
    }
    const dim3 grid((unsigned)((N + 7) / 8)), block(256);
    auto* P = (const uint32_t*)packed;
    auto* S = (const uint16_t*)scales;
    const uint16_t* Z = nullptr;
    if (bits == 2) return launch_pdl(gemv_canonical_kernel<2, false, DT>, grid, block, 0, s, P, S, Z, N, K, group, (const uint4*)x, (uint16_t*)y);
    if (bits == 3) return launch_pdl(gemv_canonical_kernel<3, false, DT>, grid, block, 0, s, P, S, Z, N, K, group, (const uint4*)x, (uint16_t*)y);
    return launch_pdl(gemv_canonical_kernel<4, false, DT>, grid, block, 0, s, P, S, Z, N, K, group, (const uint4*)x, (uint16_t*)y);
}

// the FP16 / BF16 GEMV for pot_gemm's single-token case
pot_status_t gemv_canonical_launch(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group, const void* x,
                                   void* y, cudaStream_t s, int dt) {
    return dt == 0 ? launch_gemv_canonical<0>(packed, scales, N, K, bits, group, x, y, s)
                   : launch_gemv_canonical<1>(packed, scales, N, K, bits, group, x, y, s);
}
pot_status_t gemv_stream_launch(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group, const void* x,
                                void* y, void* workspace, cudaStream_t s, int dt) {
    if (dt == 0) return launch_gemv_stream<SK_POT, 0>(packed, scales, nullptr, N, K, bits, group, x, y, workspace, s);
    return launch_gemv_stream<SK_POT, 1>(packed, scales, nullptr, N, K, bits, group, x, y, workspace, s);
}

// (the partial-sum layout depends neither on the kind of codes nor on the occupancy)
static size_t gemv_stream_workspace(int64_t N, int64_t K, int bits, int group, int tok) {
    const StreamPlan p = plan_stream(N, K, 1, bits, group, SK_UINT, tok, 16);
    return p.ok ? p.ws_bytes : 0;
}

}  // namespace pot

using namespace pot;

// Host arithmetic only: how pot_gemv / uint_gemv would run a tiled shape (tests assert which variants they reach).
extern "C" pot_status_t pot_debug_gemv_plan(int64_t N, int64_t K, int bits, int group, int uniform, int* ctas_per_sm,
                                            int* row_block_split, int* ring_slots, int* units_per_slot, int* x_in_smem) {
    if (!ctas_per_sm || !row_block_split || !ring_slots || !units_per_slot || !x_in_smem) return POT_ERR_NULL;
    pot_status_t st = check_shape(N, K, bits, group);
    if (st != POT_OK) return st;
    if (N % 16 != 0) return POT_ERR_SHAPE;
    const int kind = uniform ? SK_UINT : SK_POT;
    const int occ = gemv_occupancy(N, K, bits, group, kind);
    const StreamPlan p = plan_stream(N, K, 1, bits, group, kind, 1, 16, occ);
    if (!p.ok) return POT_ERR_SHAPE;
    *ctas_per_sm = occ;
    *row_block_split = p.aligned ? 1 : 0;
    *ring_slots = p.stages;
    *units_per_slot = p.q;
    *x_in_smem = p.x_in_smem ? 1 : 0;
    return POT_OK;
}
extern "C" pot_status_t pot_debug_gemv_split(int64_t M, int64_t N, int64_t K, int bits, int group, int bf16, int* split) {
    if (!split) return POT_ERR_NULL;
    const pot_status_t st = check_shape(N, K, bits, group);
    if (st != POT_OK) return st;
    if (M < 1 || M > 8 || N % 16 != 0) return POT_ERR_SHAPE;
    const int dt = bf16 ? 1 : 0, tok = M == 1 ? 1 : 8, occ = M == 1 ? gemv_occupancy(N, K, bits, group, SK_POT, dt) : 1;
    const StreamPlan p = plan_stream(N, K, M, bits, group, SK_POT, tok, 16, occ, dt);
    if (!p.ok) return POT_ERR_SHAPE;
    *split = p.even ? 2 : (p.aligned ? 0 : 1);
    return POT_OK;
}
extern "C" pot_status_t pot_debug_canonical_gemv_plan(int64_t N, int64_t K, int bits, int* warps_per_row_block, int* warps_per_cta, int* ctas_per_row_block) {
    if (!warps_per_row_block || !warps_per_cta || !ctas_per_row_block) return POT_ERR_NULL;
    const pot_status_t st = check_shape(N, K, bits, 128);
    if (st != POT_OK) return st;
    const bool mma = K <= GC_MAX_K;  // (longer rows: one warp each, eight to a CTA)
    const CanonPlan p = plan_canonical(N, K, bits);
    *warps_per_row_block = mma ? 1 << p.wk_shift : 0;
    *warps_per_cta = mma ? p.warps : 8;
    *ctas_per_row_block = mma ? p.cluster : 0;
    return POT_OK;
}
extern "C" pot_status_t pot_debug_gemv_decode(int64_t N, int64_t K, int bits, int group, int bf16, int* ctas_per_sm, int* unscaled) {
    if (!ctas_per_sm || !unscaled) return POT_ERR_NULL;
    const pot_status_t st = check_shape(N, K, bits, group);
    if (st != POT_OK) return st;
    if (N % 16 != 0) return POT_ERR_SHAPE;
    const int dt = bf16 ? 1 : 0, occ = gemv_occupancy(N, K, bits, group, SK_POT, dt);
    const StreamPlan p = plan_stream(N, K, 1, bits, group, SK_POT, 1, 16, occ, dt);
    if (!p.ok) return POT_ERR_SHAPE;
    *ctas_per_sm = occ;
    *unscaled = p.unscaled ? 1 : 0;
    return POT_OK;
}

extern "C" size_t pot_gemv_workspace_bytes(int64_t N, int64_t K, int bits, int group) {
    if (check_shape(N, K, bits, group) != POT_OK || N % 16 != 0) return 0;
    return gemv_stream_workspace(N, K, bits, group, 1);  // row-block arrival counters + FP32 partial slots
}

// every argument check of pot_gemv, run before anything is enqueued (also by the wrappers that enqueue copies first)
static pot_status_t check_gemv_args(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group,
                                    pot_layout_t layout, const void* x, const void* y, const void* workspace, size_t ws_bytes) {
    if (!packed || !scales || !x || !y) return POT_ERR_NULL;
    pot_status_t st = check_shape(N, K, bits, group);
    if (st != POT_OK) return st;
    if (layout != POT_LAYOUT_CANONICAL && layout != POT_LAYOUT_TILED) return POT_ERR_UNSUPPORTED;
    if (!aligned16(packed) || !aligned16(scales) || !aligned16(x) || !aligned16(y) || !aligned16(workspace))
        return POT_ERR_ALIGN;
    if (layout == POT_LAYOUT_TILED) {
        if (N % 16 != 0) return POT_ERR_SHAPE;
        const StreamPlan p = plan_stream(N, K, 1, bits, group, SK_POT, 1, 16);
        if (!p.ok) return POT_ERR_SHAPE;
        if (p.ws_bytes > 0 && (!workspace || ws_bytes < p.ws_bytes)) return POT_ERR_WORKSPACE;
    }
    return POT_OK;
}

template <int DT>
static pot_status_t gemv_impl(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group,
                              pot_layout_t layout, const void* x, void* y, void* workspace, size_t ws_bytes, void* stream) {
    const pot_status_t st = check_gemv_args(packed, scales, N, K, bits, group, layout, x, y, workspace, ws_bytes);
    if (st != POT_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (layout == POT_LAYOUT_CANONICAL) return launch_gemv_canonical<DT>(packed, scales, N, K, bits, group, x, y, s);
    return launch_gemv_stream<SK_POT, DT>(packed, scales, nullptr, N, K, bits, group, x, y, workspace, s);
}

extern "C" pot_status_t pot_gemv(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group,
                                 pot_layout_t layout, const void* x, void* y, void* workspace, size_t ws_bytes,
                                 void* stream) {
    return gemv_impl<0>(packed, scales, N, K, bits, group, layout, x, y, workspace, ws_bytes, stream);
}

extern "C" pot_status_t pot_gemv_bf16(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group,
                                      pot_layout_t layout, const void* x, void* y, void* workspace, size_t ws_bytes,
                                      void* stream) {
    return gemv_impl<1>(packed, scales, N, K, bits, group, layout, x, y, workspace, ws_bytes, stream);
}

extern "C" pot_status_t pot_gemv_host(const void* packed, const void* scales, int64_t N, int64_t K, int bits, int group,
                                      pot_layout_t layout, const void* x_host, void* y_host, void* d_x, void* d_y,
                                      void* workspace, size_t ws_bytes, void* stream) {
    if (!x_host || !y_host) return POT_ERR_NULL;
    pot_status_t st = check_gemv_args(packed, scales, N, K, bits, group, layout, d_x, d_y, workspace, ws_bytes);
    if (st != POT_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemcpyAsync(d_x, x_host, (size_t)K * 2, cudaMemcpyHostToDevice, s) != cudaSuccess) return POT_ERR_CUDA;
    st = pot_gemv(packed, scales, N, K, bits, group, layout, d_x, d_y, workspace, ws_bytes, stream);
    if (st != POT_OK) return st;
    if (cudaMemcpyAsync(y_host, d_y, (size_t)N * 2, cudaMemcpyDeviceToHost, s) != cudaSuccess) return POT_ERR_CUDA;
    return POT_OK;
}

extern "C" pot_status_t uint_gemv(const void* packed, const void* scales, const void* zeros, int64_t N, int64_t K,
                                  int bits, int group, pot_layout_t layout, const void* x, void* y, void* workspace,
                                  size_t ws_bytes, void* stream) {
    if (!packed || !scales || !zeros || !x || !y) return POT_ERR_NULL;
    pot_status_t st = check_shape(N, K, bits, group);
    if (st != POT_OK) return st;
    if (layout != POT_LAYOUT_CANONICAL && layout != POT_LAYOUT_TILED) return POT_ERR_UNSUPPORTED;
    if (!aligned16(packed) || !aligned16(scales) || !aligned16(zeros) || !aligned16(x) || !aligned16(y) ||
        !aligned16(workspace))
        return POT_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    auto* S = (const uint16_t*)scales;
    auto* Z = (const uint16_t*)zeros;
    if (layout == POT_LAYOUT_CANONICAL) {
        const dim3 grid((unsigned)((N + 7) / 8)), block(256);
        auto* P = (const uint32_t*)packed;
        if (bits == 2) return launch_pdl(gemv_canonical_kernel<2, true>, grid, block, 0, s, P, S, Z, N, K, group, (const uint4*)x, (uint16_t*)y);
        if (bits == 3) return launch_pdl(gemv_canonical_kernel<3, true>, grid, block, 0, s, P, S, Z, N, K, group, (const uint4*)x, (uint16_t*)y);
        return launch_pdl(gemv_canonical_kernel<4, true>, grid, block, 0, s, P, S, Z, N, K, group, (const uint4*)x, (uint16_t*)y);
    }
    if (N % 16 != 0) return POT_ERR_SHAPE;
    const size_t need = pot_gemv_workspace_bytes(N, K, bits, group);
    if (need > 0 && (!workspace || ws_bytes < need)) return POT_ERR_WORKSPACE;
    // same kernel as pot_gemv (tensor-core path); only the decode differs
    return launch_gemv_stream<SK_UINT>(packed, scales, zeros, N, K, bits, group, x, y, workspace, s);
}

// ------------------------------------------------------------------------------------------
// pot_gemv_noalloc: the split-K GEMV for callers that are not allowed to allocate device memory.
// ------------------------------------------------------------------------------------------
// Some hosts of this library own all device memory themselves and hand their plug-ins a fixed
// budget: an inference server whose serving loop must never hit the implicit device-wide
// synchronisation of cudaMalloc/cudaFree, or an embedding application whose allocator the
// library cannot reach.  Such a caller cannot provide the split-K workspace that pot_gemv asks
// for.  For them the scratch lives in the library image itself: a fixed-size array in device
// memory that every GPU which loads the library carries until the process exits.
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(1) << 20;  // 1 MiB per GPU
constexpr int kNoAllocMaxDevices = 64;
}  // namespace

// In host code this name is only a handle for the runtime (it is NOT a device address); the
// device address is looked up per GPU with cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {
std::atomic<void*> g_noalloc_ptr[kNoAllocMaxDevices];
}

extern "C" size_t pot_gemv_noalloc_max_scratch_bytes(void) { return kNoAllocScratchBytes; }

extern "C" pot_status_t pot_gemv_noalloc(const void* packed_tiled, const void* scales, int64_t N, int64_t K, int bits,
                                         int group, const void* x, void* y, void* stream) {
    if (!packed_tiled || !scales || !x || !y) return POT_ERR_NULL;
    pot_status_t st = check_shape(N, K, bits, group);
    if (st != POT_OK) return st;
    if (N % 16 != 0) return POT_ERR_SHAPE;
    const size_t need = pot_gemv_workspace_bytes(N, K, bits, group);
    if (need > kNoAllocScratchBytes) return POT_ERR_WORKSPACE;  // shape needs more scratch than the built-in array holds
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return POT_ERR_CUDA;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return POT_ERR_UNSUPPORTED;
    // Set-up, once per device, with that device current: ask the runtime where this GPU's copy of the
    // array lives.  (Racing first calls both get the same answer, so a plain atomic store is enough.)
    void* scratch = g_noalloc_ptr[dev].load(std::memory_order_acquire);
    if (!scratch) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return POT_ERR_CUDA;
        g_noalloc_ptr[dev].store(p, std::memory_order_release);
        scratch = p;
    }
    st = check_gemv_args(packed_tiled, scales, N, K, bits, group, POT_LAYOUT_TILED, x, y, scratch, kNoAllocScratchBytes);
    if (st != POT_OK) return st;  // nothing has been enqueued yet
    if (need == 0) return pot_gemv(packed_tiled, scales, N, K, bits, group, POT_LAYOUT_TILED, x, y, nullptr, 0, stream);
    // The array keeps whatever the previous call, of any shape, left in it.  Only the arrival counters, or the places of the sums that go
    // from CTA to CTA, have to start without counts or marks (partial sums are fully overwritten before they are read), so clear just those.
    size_t clear = plan_stream(N, K, 1, bits, group, SK_POT, 1, 16).ws_counters;
    if (clear < sk_box_bytes(1)) clear = sk_box_bytes(1);
    if (cudaMemsetAsync(scratch, 0, clear, (cudaStream_t)stream) != cudaSuccess) return POT_ERR_CUDA;
    return pot_gemv(packed_tiled, scales, N, K, bits, group, POT_LAYOUT_TILED, x, y, scratch, need, stream);
}

