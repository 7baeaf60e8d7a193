// Training-forward statistic of Algorithm 2 on sm_100a: psum[i] = sum_n P_{n,i}, the column sums of the row-wise
// softmax over all M experts (Eq. app_softmax, Eq. app_psum), given each token's log-sum-exp from the routing sweep.
// This is Algorithm 2's second sweep: the logit tiles are produced again and reduced along the TOKEN axis, and the
// T x M probabilities never exist in memory.
//
// The first half of the kernel is the router's: TMA streams X and R1, tcgen05.mma accumulates z = X_blk R1 for a
// block of 128 or 160 ... 256 tokens in TMEM, the epilogue threads narrow it to bf16 hi + lo in shared memory.  The second
// contraction is issued TRANSPOSED, D[expert][token] = R2[:, tile]^T z^T: the R2 tile is the (MN-major) A operand,
// z the (K-major) B operand, so a TMEM lane is an expert and its columns are tokens.  Each epilogue thread then owns
// one expert of the tile and adds exp(y - lse_token) over its share of the block's token columns in registers -- a column
// sum with no cross-lane traffic -- and finishes with one atomic add into psum.  (In the router the lanes are tokens,
// because there the reduction runs along the expert axis.)
//
// Warp roles, shared-memory ring, barriers and the bounded waits are those of the router kernel, but for 16 epilogue warps:
// four per lane quarter, two for the first 128 tokens, which take 64 token columns each, and two for what the block has beyond
// them, 16 to 64 columns each (none up to 128 tokens).  Bound by the exponentials: 12 of 16 go
// through the special-function unit (16 results per clock and SM), four through the FMA pipe, and with 32 epilogue warps
// per SM the latencies around them are hidden (16 warps, which could each hold twice the registers: 53 % of the issue
// slots used).
#include "sm100_common.cuh"

#include <math.h>

#include <type_traits>

namespace more {

namespace {

constexpr int kPsumEpi = 512;
constexpr int kPsumThreads = 64 + kPsumEpi;
// Up to 128 tokens: the second half does nothing, X tiles are half as tall, and four stages of them fit where otherwise two do (the
// first contraction is a chain of trips to memory then: T = 4, h = 2152, r = 32, M = 1584 25.0 -> 16.7 us, T = 24, h = 3360, r = 56, M = 20224 36.8 -> 20.7).
constexpr int kFewTokens = 128, kFewStages = 4, kFewXBytes = kXTileBytes / 2, kFewStageBytes = kFewXBytes + 64 * 128;
static_assert(kFewStages * kFewStageBytes <= kRingBytes, "phase-1 stages do not fit");

// 16 consecutive fp32 columns of this thread's tensor-memory lane, complete on return.  (Load and wait in one statement:
// with the destination registers tied to a separate wait the compiler copies them.)
__device__ __forceinline__ void tmem_get16(uint32_t taddr, float (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
          "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr)
        : "memory");
}

struct PsumParams {
    int T, h, r, M, msplit, tiles_total;
    int block;           // tokens of a block: a multiple of 32, 128 or 160 ... 256 (what a CTA computes z for beyond them is not used)
    const float* lse;    // [T] natural-log log-sum-exp of every token's logits
    float* psum;         // [M], zeroed before the launch
    int* status;
};

template <int RPAD>
__global__ void __launch_bounds__(kPsumThreads, 2)
psum_tcgen05_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_r1,
                    const __grid_constant__ CUtensorMap map_r2, const PsumParams p)
{
    constexpr int kKSteps = RPAD / 16;
    constexpr int kZopOne = (RPAD == 64) ? 32768 : 16384;       // [hi | lo] operand of one 128-token half
    constexpr int kZopBytes = 2 * kZopOne;
    constexpr int kLseBytes = 1024;                              // 256 floats: log2-scaled lse of the block's tokens
    constexpr int kR2StageBytes = RPAD * 256;
    constexpr int kStagesP2 = (RPAD == 64) ? 2 : 4;
    static_assert(kZopBytes + kLseBytes + kStagesP2 * kR2StageBytes <= kRingBytes, "phase-2 layout does not fit");
    constexpr float kLog2e = 1.4426950408889634f;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    uint8_t* ring_ptr = smem_raw + (ring - raw);
    uint8_t* ctl = ring_ptr + kRingBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(ctl);
    constexpr int B_FULL1 = 0, B_EMPTY1 = B_FULL1 + kFewStages, B_ZACC = B_EMPTY1 + kFewStages, B_ZOP = B_ZACC + 1,
                  B_FULL2 = B_ZOP + 1, B_EMPTY2 = B_FULL2 + 8, B_ACCF = B_EMPTY2 + 8, B_ACCE = B_ACCF + 2,
                  B_COUNT = B_ACCE + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ctl + B_COUNT * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(ctl + B_COUNT * 8 + 4);
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = blockIdx.x / p.msplit, split = blockIdx.x % p.msplit;
    const int tok0 = blk * p.block;
    const int tile_lo = (int)(((long long)p.tiles_total * split) / p.msplit);
    const int tile_hi = (int)(((long long)p.tiles_total * (split + 1)) / p.msplit);
    const int ntiles = tile_hi - tile_lo;
    const int ktiles1 = (p.h + 63) / 64;
    const bool few = p.block <= kFewTokens;
    const int stages1 = few ? kFewStages : kStagesP1, x_bytes = few ? kFewXBytes : kXTileBytes, st1_bytes = few ? kFewStageBytes : kP1StageBytes;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kFewStages; ++i) { mbar_init(bar(B_FULL1 + i), 1); mbar_init(bar(B_EMPTY1 + i), 1); }
        mbar_init(bar(B_ZACC), 1);
        mbar_init(bar(B_ZOP), kEpilogueThreads);
        for (int i = 0; i < 8; ++i) { mbar_init(bar(B_FULL2 + i), 1); mbar_init(bar(B_EMPTY2 + i), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(bar(B_ACCF + i), 1); mbar_init(bar(B_ACCE + i), kPsumEpi / 32 / 2); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t zop = ring;
    float* lse2 = reinterpret_cast<float*>(ring_ptr + kZopBytes);
    const uint32_t r2ring = ring + kZopBytes + kLseBytes;

    if (warp == 0) {
        // ===================================================================================== TMA producer
        if (lane == 0) {
            bool ok = true;
            for (int kt = 0, s = 0, ph = 1; kt < ktiles1 && ok; ++kt) {
                ok = mbar_wait(bar(B_EMPTY1 + s), ph, abort_flag, p.status);
                if (!ok) break;
                const uint32_t dst = ring + s * st1_bytes;
                mbar_expect_tx(bar(B_FULL1 + s), st1_bytes);
                tma_load_2d(dst, &map_x, bar(B_FULL1 + s), kt * 64, tok0);
                tma_load_2d(dst + x_bytes, &map_r1, bar(B_FULL1 + s), 0, kt * 64);
                if (++s == stages1) { s = 0; ph ^= 1; }
            }
            ok = ok && mbar_wait(bar(B_ZACC), 0, abort_flag, p.status);
            for (int it = 0; it < ntiles && ok; ++it) {
                const int s = it % kStagesP2;
                if (it >= kStagesP2) ok = mbar_wait(bar(B_EMPTY2 + s), ((it / kStagesP2) - 1) & 1, abort_flag, p.status);
                if (!ok) break;
                const uint32_t dst = r2ring + s * kR2StageBytes;
                const int e0 = (tile_lo + it) * kTileExperts;
                mbar_expect_tx(bar(B_FULL2 + s), kR2StageBytes);
                tma_load_2d(dst, &map_r2, bar(B_FULL2 + s), e0, 0);
                tma_load_2d(dst + RPAD * 128, &map_r2, bar(B_FULL2 + s), e0 + 64, 0);
            }
        }
    } else if (warp == 1) {
        // ======================================================================================= MMA issuer
        // The whole warp runs this code converged and one elected lane issues each instruction; the descriptors are
        // words computed once plus integer offsets (see tc_mma_bf16_ss_elect).
        constexpr unsigned kFull = 0xffffffffu;
        bool ok = true;
        constexpr uint32_t idesc1 = umma_idesc(64);
        // second contraction transposed: A = R2 tile (MN-major), B = z operand (K-major), 128 experts x 128 tokens
        constexpr uint32_t idesc2 = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (0u << 16) |
                                    ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        {
            const uint64_t xd = umma_desc_sw128(ring, 16, 1024), rd = umma_desc_sw128(ring + x_bytes, 8192, 1024);
            const uint32_t x_lo0 = (uint32_t)xd, x_hi = (uint32_t)(xd >> 32), r_lo0 = (uint32_t)rd, r_hi = (uint32_t)(rd >> 32);
            for (int kt = 0, s = 0, ph = 0; kt < ktiles1 && ok; ++kt) {
                ok = __all_sync(kFull, mbar_wait(bar(B_FULL1 + s), ph, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
                const uint32_t x_lo = x_lo0 + s * (st1_bytes >> 4), r_lo = r_lo0 + s * (st1_bytes >> 4);
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    if (a == 1 && few) break;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma_bf16_ss_elect(tmem_base + a * kTileExperts, x_lo + a * (16384 >> 4) + kk * 2, x_hi,
                                             r_lo + kk * (2048 >> 4), r_hi, idesc1, (kt | kk) != 0);
                }
                tc_commit_elect(bar(B_EMPTY1 + s));
                if (++s == stages1) { s = 0; ph ^= 1; }
            }
        }
        if (ok) tc_commit_elect(bar(B_ZACC));
        ok = __all_sync(kFull, ok && mbar_wait(bar(B_ZOP), 0, abort_flag, p.status));
        tc_fence_after();
        const uint32_t idesc_tail = (idesc2 & ~(0x3fu << 17)) | ((uint32_t)((p.block - 128) >> 3) << 17);    // the second half's tokens
        const uint64_t ad0 = umma_desc_sw128(r2ring, RPAD * 128, 1024), zd0 = umma_desc_sw128(zop, 16, 1024);
        const uint32_t a_lo0 = (uint32_t)ad0, a_hi = (uint32_t)(ad0 >> 32), z_lo0 = (uint32_t)zd0, z_hi = (uint32_t)(zd0 >> 32);
        for (int it = 0; it < ntiles && ok; ++it) {
            const int s = it % kStagesP2;
            ok = __all_sync(kFull, mbar_wait(bar(B_FULL2 + s), (it / kStagesP2) & 1, abort_flag, p.status));
            if (!ok) break;
            const uint32_t a_lo = a_lo0 + s * (kR2StageBytes >> 4);
#pragma unroll
            for (int a = 0; a < 2; ++a) {            // token half a -> TMEM columns a*128 ..
                if (a == 1 && few) break;
                ok = __all_sync(kFull, ok && mbar_wait(bar(B_ACCE + a), (it & 1) ^ 1, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int j = 0; j < 2 * kKSteps; ++j) {
                    const uint32_t zbyte = j * 32;                                       // K offset in [hi | lo]
                    tc_mma_bf16_ss_elect(tmem_base + a * 128, a_lo + (j % kKSteps) * (2048 >> 4), a_hi,
                                         z_lo0 + ((a * kZopOne + (zbyte >> 7) * 16384 + (zbyte & 127)) >> 4), z_hi,
                                         a == 0 ? idesc2 : idesc_tail, j != 0);
                }
                tc_commit_elect(bar(B_ACCF + a));
            }
            if (!ok) break;
            tc_commit_elect(bar(B_EMPTY2 + s));
        }
    } else {
        // ========================================================================================= epilogue
        const int q = warp & 3;                              // TMEM lane group: token rows (phase 1), experts (phase 2)
        const int half = ((warp - 2) >> 2) & 1;              // which 128-token half
        const int part = (warp - 2) >> 3;                    // which half of its columns
        const int row_in_half = q * 32 + lane;
        const int row_in_blk = half * 128 + row_in_half;
        const int64_t row = (int64_t)tok0 + row_in_blk;
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16) + half * 128;
        bool ok = mbar_wait(bar(B_ZACC), 0, abort_flag, p.status);
        if (ok && part == 0 && half == 1 && few) {
            mbar_arrive(bar(B_ZOP));
        } else if (ok && part == 0) {
            tc_fence_after();
            // (the phase-1 ring is free now) minus the log2-scaled log-sum-exp of my token; -inf for rows past T, whose
            // zero-filled logits then contribute exp(-inf) = 0
            lse2[row_in_blk] = (row < p.T && row_in_blk < p.block) ? -p.lse[row] * kLog2e : -INFINITY;
            uint8_t* zrow = ring_ptr + half * kZopOne + row_in_half * 128;
#pragma unroll
            for (int c = 0; c < RPAD / 16; ++c) {
                float z[16];
                tmem_get16(t_lane + c * 16, z);
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const __nv_bfloat16 h0 = __float2bfloat16_rn(z[2 * e]), h1 = __float2bfloat16_rn(z[2 * e + 1]);
                    const __nv_bfloat16 l0 = __float2bfloat16_rn(z[2 * e] - __bfloat162float(h0));
                    const __nv_bfloat16 l1 = __float2bfloat16_rn(z[2 * e + 1] - __bfloat162float(h1));
                    hi[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                    lo[e] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                }
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int ch_hi = c * 2 + hf, ch_lo = RPAD / 8 + c * 2 + hf;
                    const int slab_hi = ch_hi >> 3, slab_lo = ch_lo >> 3;
                    uint4 vh = make_uint4(hi[hf * 4], hi[hf * 4 + 1], hi[hf * 4 + 2], hi[hf * 4 + 3]);
                    uint4 vl = make_uint4(lo[hf * 4], lo[hf * 4 + 1], lo[hf * 4 + 2], lo[hf * 4 + 3]);
                    *reinterpret_cast<uint4*>(zrow + slab_hi * 16384 + (((ch_hi & 7) ^ (row_in_half & 7)) << 4)) = vh;
                    *reinterpret_cast<uint4*>(zrow + slab_lo * 16384 + (((ch_lo & 7) ^ (row_in_half & 7)) << 4)) = vl;
                }
            }
            fence_async_smem();
            tc_fence_before();
            mbar_arrive(bar(B_ZOP));
        }
        // all 256 lse2 entries must be visible before anyone reads them in the sweep
        asm volatile("bar.sync 1, 512;" ::: "memory");

        ok = __all_sync(0xffffffffu, ok);
        // The sweep, for a number of 16-column chunks that the compiler knows.
        auto sweep = [&](auto chunks_c) {
            constexpr int kChunks = decltype(chunks_c)::value;
            const ulonglong2* lse4 = reinterpret_cast<const ulonglong2*>(lse2 + half * 128 + part * kChunks * 16);
            const uint64_t scale = pack2(kLog2e, kLog2e);
            for (int it = 0; it < ntiles && ok; ++it) {
                const int expert = (tile_lo + it) * kTileExperts + q * 32 + lane;     // my lane's expert in this tile
                ok = __all_sync(0xffffffffu, mbar_wait(bar(B_ACCF + half), it & 1, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
                uint64_t acc01 = 0, acc23 = 0;
#pragma unroll
                for (int c = 0; c < kChunks; ++c) {
                    float v[16];
                    tmem_get16(t_lane + (part * kChunks + c) * 16, v);
                    if (c + 1 == kChunks) {                      // all columns are in registers: hand the accumulator back
                        tc_fence_before();
                        warp_arrive(bar(B_ACCE + half), lane);
                    }
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const ulonglong2 l = lse4[c * 4 + g];    // same address in every lane: a broadcast
                        float x0, x1, x2, x3;
                        unpack2(fma2(pack2(v[4 * g], v[4 * g + 1]), scale, l.x), x0, x1);
                        unpack2(fma2(pack2(v[4 * g + 2], v[4 * g + 3]), scale, l.y), x2, x3);
                        // (one exponential in four on the FMA pipe: the special-function unit's 16 results per clock per SM
                        // are this loop's narrowest resource)
                        acc01 = add2(acc01, pack2(ex2f(x0), ex2f(x1)));
                        acc23 = add2(acc23, pack2(ex2f(x2), ex2_poly(x3)));
                    }
                }
                float a0, a1, a2, a3;
                unpack2(acc01, a0, a1);
                unpack2(acc23, a2, a3);
                if (expert < p.M) atomicAdd(p.psum + expert, (a0 + a1) + (a2 + a3));
            }
        };
        const int chunks = half == 0 ? 4 : (p.block - 128) / 32;
        if (chunks == 4) sweep(std::integral_constant<int, 4>{});
        else if (chunks == 3) sweep(std::integral_constant<int, 3>{});
        else if (chunks == 2) sweep(std::integral_constant<int, 2>{});
        else if (chunks == 1) sweep(std::integral_constant<int, 1>{});
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

template <int RPAD>
int launch_psum_rpad(const CUtensorMap& mx, const CUtensorMap& m1, const CUtensorMap& m2, const PsumParams& pp, int ctas,
                     cudaStream_t st)
{
    static unsigned long long configured = 0;
    auto kern = psum_tcgen05_kernel<RPAD>;
    int dev = 0;
    cudaGetDevice(&dev);
    if (!(configured >> (dev & 63) & 1ull)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess)
            return MORE_ERR_CUDA;
        configured |= 1ull << (dev & 63);
    }
    kern<<<ctas, kPsumThreads, kSmemBytes, st>>>(mx, m1, m2, pp);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? MORE_OK : MORE_ERR_CUDA;
}

// Tokens of a block, and CTAs per block, by a model of the time.  CTAs that have an SM each take less than half of what two on an
// SM do where the projection counts, as 256 rows of X per k-tile, whatever the block, are bound by the SM's share of L2, and all
// of them together slow each other down (T = 2737, h = 3800, M = 7136: 77 CTAs 51 us, 220 of them 82; T = 18993, h = 744, M = 184:
// 75 CTAs 18.9 us, 119 22.7).  Microseconds, fitted to 300 shapes (T = 129 ... 64 k, h = 128 ... 4096, r = 8 ... 64, M = 128 ... 128 k)
// at up to 35 pairs of block and split each.  On 200 others what is chosen takes 1.01 of the best pair's time on average and 1.12
// at most; blocks of 256 and two CTAs per SM wherever there are four tiles for each take 1.14, and stay only where no other pair
// should be 3 % better.
void choose_blocks(int T, int h, int tiles, int slots, int* block_out, int* split_out)
{
    const double ktiles = (h + 63) / 64;
    double best = 1e300;
    auto consider = [&](int block, int split, double handicap) {
        const int per = (tiles + split - 1) / split, s = (tiles + per - 1) / per;
        const long long ctas = (long long)((T + block - 1) / block) * s, waves = (ctas + slots - 1) / slots;
        const double chunks = block / 16.0;
        const double alone = 0.88 + 0.234 * ktiles + per * (0.623 + 0.0545 * chunks);
        const double shared = 2.14 + 0.537 * ktiles + per * (0.80 + 0.117 * chunks);
        const double last = 2 * (ctas - (waves - 1) * slots) <= slots ? alone : shared;      // the last wave
        const double us = (5.5 + (waves - 1) * shared + last + 0.0021 * ctas * ktiles) * handicap;
        if (us < best) { best = us; *block_out = block; *split_out = s; }
    };
    const int n = (T + kBlockTokens - 1) / kBlockTokens, most = slots / n < tiles / 4 ? slots / n : tiles / 4;
    consider(kBlockTokens, most < 1 ? 1 : (most < 64 ? most : 64), 0.97);
    for (int block = kBlockTokens; block >= 160; block -= 32) {
        const int blocks = (T + block - 1) / block;
        for (int all = slots; all >= slots / 2; all -= slots / 2)
            for (int part = 12; part >= 3; part -= 3) {
                const int split = all / blocks * part / 12;
                consider(block, split < 1 ? 1 : (split < tiles ? split : tiles), 1.0);
            }
    }
}

}  // namespace

void plan_psum(int T, int h, int M, int sm_count, int* block, int* split)
{
    const int slots = 2 * (sm_count > 0 ? sm_count : 148), tiles = (M + kTileExperts - 1) / kTileExperts;
    if (T > kFewTokens) return choose_blocks(T, h, tiles, slots, block, split);
    *block = kFewTokens;                           // a CTA per SM at most, two tiles or more
    *split = tiles / 2 < slots / 2 ? tiles / 2 : slots / 2;
    if (*split < 1) *split = 1;
}

int launch_psum_tcgen05(const __nv_bfloat16* X, const __nv_bfloat16* R1, const __nv_bfloat16* R2, int T, int h, int r,
                        int M, const float* lse, float* psum, DeviceCtx& ctx, cudaStream_t stream)
{
    CUtensorMap mx, m1, m2;
    const bool few = T <= kFewTokens;
    const int rpad = (r <= 16) ? 16 : (r <= 32 ? 32 : 64);
    int rc = get_tensor_map(X, T, h, few ? kFewTokens : kBlockTokens, 64, &mx);
    if (rc == MORE_OK) rc = get_tensor_map(R1, h, r, 64, 64, &m1);
    if (rc == MORE_OK) rc = get_tensor_map(R2, r, M, rpad, 64, &m2);
    if (rc != MORE_OK) return rc;
    PsumParams pp;
    pp.T = T; pp.h = h; pp.r = r; pp.M = M;
    pp.tiles_total = (M + kTileExperts - 1) / kTileExperts;
    pp.lse = lse; pp.psum = psum; pp.status = ctx.status;
    plan_psum(T, h, M, ctx.sm_count, &pp.block, &pp.msplit);
    const int s = pp.msplit, blocks = (T + pp.block - 1) / pp.block;
    switch (rpad) {
        case 16: return launch_psum_rpad<16>(mx, m1, m2, pp, blocks * s, stream);
        case 32: return launch_psum_rpad<32>(mx, m1, m2, pp, blocks * s, stream);
        default: return launch_psum_rpad<64>(mx, m1, m2, pp, blocks * s, stream);
    }
}

}  // namespace more
