// The low-rank router (Algorithm 1 with the gates of Section 2 / Eq. app_softmax and the per-expert counts) for few tokens
// and for long sweeps, as three kernels chained with programmatic dependent launches:
//
//   project_kernel   z = X R1, narrowed to a bf16 pair [hi | lo] per token, to scratch (T x 128 or 256 bytes).
//   sweep_kernel     y = z R2 tile by tile on the tensor cores, reduced on chip to a short list of candidates per token
//                    (and the online (max, sum) pair of Eq. app_online); the T x M logits never reach memory.
//   finish_*_kernel  the candidates of all of a token's expert ranges -> sorted top-k, gates, histogram.
//
// Why three.  The projection is bound by reading X, the sweep by the tensor cores and by looking at every logit; with z
// in scratch the sweep can be cut anywhere along tokens x experts (every CTA gets the same number of steps, whatever T
// and M are), a token block whose experts are shared by many CTAs is projected once instead of once per CTA, and shared
// and tensor memory belong to the sweep alone.  z costs 2 x T x 256 bytes of L2 traffic, 1/8 of X at h = 2048.
#include "more_topk.cuh"
#include "sm100_common.cuh"

#include <cuda_bf16.h>
#include <float.h>

#include <type_traits>

namespace more {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRows = 128;                         // tokens per block: the rows of one accumulator
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ============================================================================================== projection
// One cluster of `cs` CTAs per 128-token block; CTA `rank` contracts an even share of the h / 64 k-tiles.  With cs > 1
// the partial sums are exchanged through distributed shared memory: every CTA collects 128 / cs rows from all, adds them
// in rank order (so the result does not depend on timing) and narrows them.
constexpr int kPThreads = 192;                     // warp 0 TMA, warp 1 MMA, warps 2..5 one token per thread
constexpr int kPStages = 4;
constexpr int kPStageBytes = kRows * 128 + 64 * 128;      // X tile 128 x 64, R1 tile 64 x 64 (columns >= r zero-filled)
constexpr int kPExchange = kRows * 64 * 4;         // [rank][row share][64] fp32
constexpr int kPCtl = 1024;

struct ProjectParams {
    int T, h, cs, cs_bits, n, zc;                           // n: columns of z computed (16, 32, 48, 64); zc: bf16 per row of z
    uint32_t* z;                                   // [blocks * 128][zc / 2]
    int32_t* counts;                               // cleared here: [M] (null for the later chunks of one call)
    int M;
    int* status;
};

__device__ __forceinline__ void narrow2(float a, float b, uint32_t& hi, uint32_t& lo)
{
    const __nv_bfloat16 h0 = __float2bfloat16_rn(a), h1 = __float2bfloat16_rn(b);
    const __nv_bfloat16 l0 = __float2bfloat16_rn(a - __bfloat162float(h0)), l1 = __float2bfloat16_rn(b - __bfloat162float(h1));
    hi = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
    lo = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
}

__global__ void __launch_bounds__(kPThreads)
project_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_r1, const ProjectParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    uint8_t* ring_ptr = smem_raw + (ring - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(ring_ptr + kPStages * kPStageBytes);
    constexpr int B_FULL = 0, B_EMPTY = kPStages, B_DONE = 2 * kPStages, B_COUNT = B_DONE + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    float* exch = reinterpret_cast<float*>(ring_ptr + kPStages * kPStageBytes + kPCtl);
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cs = p.cs, rank = blockIdx.x & (cs - 1), blk = blockIdx.x >> p.cs_bits;
    const int nkt = (p.h + 63) / 64;
    const int kt_lo = nkt * rank >> p.cs_bits, kt_hi = nkt * (rank + 1) >> p.cs_bits;
    const int live = min(kRows, p.T - blk * kRows);

    if (threadIdx.x == 0) {
        for (int i = 0; i < B_COUNT; ++i) mbar_init(bar(i), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (cs > 1) cluster_sync();                    // every CTA of the cluster is running before anyone writes into it
    pdl_wait();                                    // the set-up above overlaps the end of what ran before
    // The sweep may be placed next to this kernel from here on: this CTA's tensor memory is allocated, so the sweep's
    // own allocation can only wait for it, never take it away.
    pdl_launch_dependents();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            for (int kt = kt_lo, i = 0; kt < kt_hi && ok; ++kt, ++i) {
                const int s = i % kPStages;
                if (i >= kPStages) ok = mbar_wait(bar(B_EMPTY + s), ((i / kPStages) - 1) & 1, abort_flag, p.status);
                if (!ok) break;
                const uint32_t dst = ring + s * kPStageBytes;
                mbar_expect_tx(bar(B_FULL + s), kPStageBytes);
                tma_load_2d(dst, &map_x, bar(B_FULL + s), kt * 64, blk * kRows);
                tma_load_2d(dst + kRows * 128, &map_r1, bar(B_FULL + s), 0, kt * 64);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        bool ok = true;
        const uint32_t idesc = umma_idesc(p.n);
        const uint64_t xd = umma_desc_sw128(ring, 16, 1024), rd = umma_desc_sw128(ring + kRows * 128, 8192, 1024);
        const uint32_t x_lo0 = (uint32_t)xd, x_hi = (uint32_t)(xd >> 32), r_lo0 = (uint32_t)rd, r_hi = (uint32_t)(rd >> 32);
        for (int kt = kt_lo, i = 0; kt < kt_hi && ok; ++kt, ++i) {
            const int s = i % kPStages;
            ok = __all_sync(kFull, mbar_wait(bar(B_FULL + s), (i / kPStages) & 1, abort_flag, p.status));
            if (!ok) break;
            tc_fence_after();
            const uint32_t x_lo = x_lo0 + s * (kPStageBytes >> 4), r_lo = r_lo0 + s * (kPStageBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)         // A: +32 B per K = 16; B: 16 K-rows of 128 B
                tc_mma_bf16_ss_elect(tmem_base, x_lo + kk * 2, x_hi, r_lo + kk * (2048 >> 4), r_hi, idesc, (i | kk) != 0);
            tc_commit_elect(bar(B_EMPTY + s));
        }
        if (ok) tc_commit_elect(bar(B_DONE));
        __syncwarp();
    } else {
        const int et = threadIdx.x - 64;           // 0..127
        if (p.counts)
            for (int e = blockIdx.x * kRows + et; e < p.M; e += gridDim.x * kRows) p.counts[e] = 0;
        const int row = (warp & 3) * 32 + lane;    // the tensor-memory lane this thread may read
        const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        const bool ok = __all_sync(kFull, mbar_wait(bar(B_DONE), 0, abort_flag, p.status));
        tc_fence_after();
        if (cs == 1) {
            if (ok) {
                uint4* zr = reinterpret_cast<uint4*>(p.z + (size_t)(blk * kRows + row) * (p.zc / 2));
                const int lo_off = p.zc / 16;      // 16-byte chunks of the hi half
                for (int c = 0; c < p.zc / 32; ++c) {
                    float v[16];
                    if (c * 16 < p.n) {
                        tmem_ld16(t_lane + c * 16, v);
                        tmem_ld_wait16(v);
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = 0.f;
                    }
                    uint32_t hi[8], lo[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) narrow2(v[2 * e], v[2 * e + 1], hi[e], lo[e]);
                    zr[2 * c] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    zr[2 * c + 1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
                    zr[lo_off + 2 * c] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    zr[lo_off + 2 * c + 1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
                }
            }
        } else if (ok && row - lane < live) {      // (rows past the last token are not exchanged)
            const int share = kRows >> p.cs_bits, dst = row >> (7 - p.cs_bits);
            const uint32_t a = smem_u32(exch) + (uint32_t)((rank * share + (row & (share - 1))) * 64) * 4u;
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(a), "r"(dst));
            for (int c = 0; c * 16 < p.n; ++c) {
                float v[16];
                tmem_ld16(t_lane + c * 16, v);
                tmem_ld_wait16(v);
                if (row < live) {
#pragma unroll
                    for (int e = 0; e < 16; e += 4)
                        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};"
                                     ::"r"(remote + (c * 16 + e) * 4), "f"(v[e]), "f"(v[e + 1]), "f"(v[e + 2]), "f"(v[e + 3]) : "memory");
                }
            }
        }
    }
    tc_fence_before();
    if (cs > 1) {
        cluster_sync();
        if (warp >= 2) {
            const int share = kRows >> p.cs_bits, q4_bits = p.zc == 64 ? 3 : 4, q4 = 1 << q4_bits;        // float4s of one row of z
            // Rows past the last token, up to the 32 that a warp of the sweep looks at, are zero.  (What an earlier call left
            // there would be swept as tokens whose logits can be infinite, reach any threshold and fill their lists again
            // and again: T = 7284, M = 16384 2330 us instead of 83.)
            const int mine = live - rank * share, rows = min(share, ((live + 31) & ~31) - rank * share);
            for (int i = threadIdx.x - 64; i < rows * q4; i += kRows) {
                const int rr = i >> q4_bits, c4 = i & (q4 - 1);
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c4 * 4 < p.n && rr < mine) {
                    const float* e = exch + rr * 64 + c4 * 4;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if (q < cs) {
                            const float4 v = *reinterpret_cast<const float4*>(e + q * share * 64);
                            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
                        }
                    }
                }
                uint2 hi, lo;
                narrow2(s.x, s.y, hi.x, lo.x);
                narrow2(s.z, s.w, hi.y, lo.y);
                uint2* zr = reinterpret_cast<uint2*>(p.z + (size_t)(blk * kRows + rank * share + rr) * (p.zc / 2));
                zr[c4] = hi;
                zr[q4 + c4] = lo;
            }
        }
    }
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);         // copies still in flight land before the memory is released
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem_base) : "memory");
    }
}

// ================================================================================================== sweep
// Two CTAs per SM, 18 warps each: warp 0 TMA, warp 1 MMA, warps 2..17 selection.  The work is a line of blocks x steps
// units (unit = 128 tokens x 128 experts) cut into equal contiguous parts, one per CTA; what a CTA has of one token block
// is a segment.  Per unit 2 r / 16 MMAs (hi then lo) of 128 x 128 x 16 fill one of two accumulators; four warps per
// tensor-memory lane quarter look at 32 columns each, so a token is swept by four threads.  (What bounds the sweep is
// the selection's instructions and their latencies: 32 selecting warps per SM at 56 registers hide these about twice
// as well as 16 at 96, with any arrangement of the accumulators that was tried.)
//
// Selection.  A thread keeps the maxima of NB disjoint sets of its columns ("buckets": runs of 8 or 4 columns, by their
// position in the units) and a threshold.  The k-th largest of a token's 4 NB bucket maxima is reached by
// at least k of its logits, so nothing strictly below it can be selected; its expected rank is ~11 for k = 8 of 16
// buckets, ~22 for k = 16 of 32.  Every group of four whose maximum reaches the threshold is appended, values and first
// column, to the thread's list in global scratch: two predicated stores and an add, and nothing waits for them.  (Most of
// a list stays in L2.  What leaves it, 115 MB of a call with k = 16 of 131072 experts for 8192 tokens, is 18 us of DRAM
// time in a sweep of 510.)  A sweep starts with a threshold: the bucket maxima of its first units (lead_of: all of a short
// segment, the beginning of a long one) are formed before anything is selected; this costs their MMAs and the reading of their
// accumulators again, and saves the appends of the start, when nearly everything beats what has been seen.  Whenever half
// as much again of a long segment is done, the buckets are published in shared memory, one of the four warps of a lane
// quarter computes new thresholds from them, and the others pick these up when they see them (all values are monotone
// lower bounds, so no synchronisation is needed).  At the end of a segment a thread goes once through its list and passes
// on what reaches the final threshold (~11 logits per token for k = 8).
constexpr int kSThreads = 576;
constexpr int kEpi = 512;
constexpr int W = 128;                             // experts of a unit
constexpr int kCols = W / 4;                       // columns of a thread
constexpr int kMaxStages = 8;
constexpr int kListCap = 64;                       // places of a thread's list (fewer where so few units cannot fill them)
constexpr uint32_t kEntry = kEpi * 32;             // bytes between its entries (32 bytes each: four logits, the first one's column)

// Units whose bucket maxima are formed ahead of a segment of `steps` units.  All of a short one: its threshold is then the
// final one before the first candidate is kept, and a thread keeps one or two groups instead of the ten that a rising
// threshold lets through; what is saved is not the appending but the reading back at the end, a chain of trips to L2.
// T = 3000, M = 16384: 49.9 -> 41.7 us; T = 1024, M = 65536, k = 16: 164 -> 77 us; T = 64, M = 131072, k = 16: 40.7 -> 34.3.
// Only the beginning of a long one, where computing everything twice costs more.  The line is at 32 units for k <= 8 (at 41 units 84 us
// against 81) and at 64 for longer lists, which keep three times the candidates (T = 17000, M = 16384, k = 16, 57 units:
// 187 -> 143 us).  Up to 128 units a quarter, or half for longer lists: what a better first threshold saves in appends and in
// lists read back is more than the second reading costs (T = 32768, M = 16384, segments of 59 units on average: k = 8 168.7 us
// with 1/8, 162.6 with 1/4, 166.7 with 1/2; k = 16 214, 199, 192).  Longer ones an eighth (T = 32768, M = 65536 359 us, with 1/4
// 363, with 1/2 388).  On 250 drawn shapes with segments of 34 to 425 units, both gates, this costs 1.2 % on average against the
// best of all, 1/2, 1/4, 1/6, 1/8 and 1/16 for each shape, and in no range of lengths more than 2.3 % (always 1/4 1.4 %, always
// 1/8 1.5 %).  Up to two units stay in the two accumulators, more are computed again.
__host__ __device__ __forceinline__ int lead_of(int steps, bool longer)
{
    return steps <= (longer ? 64 : 32) ? steps : (steps > 128 ? steps / 8 : steps / (longer ? 2 : 4));
}

// The line of units and the CTAs that share it.  Every warp of a CTA starts by dividing, in code that is fetched as it runs: by
// multiplication with inverses from the host where total g fits 32 bits (inv_total = 0 where it does not).  With four 64-bit
// divisions T = 64, h = 4096, M = 131072, k = 16 took 36.3 us, with these 33.9, T = 1, M = 16384 14.6 and 13.8.
struct Cut {
    long long total;                               // units
    int nsteps, g;                                 // units per token block; CTAs
    uint32_t inv_total, inv_nsteps, inv_g;
};
Cut make_cut(long long total, int nsteps, int g)
{
    Cut t{total, nsteps, g, 0, 0, 0};
    if (total < (1ll << 32) / g) {                 // (then total g < 2^32)
        t.inv_total = 0xffffffffu / (uint32_t)total;
        t.inv_nsteps = 0xffffffffu / (uint32_t)nsteps;
        t.inv_g = 0xffffffffu / (uint32_t)g;
    }
    return t;
}

struct SweepParams {
    int T, M, k;
    Cut cut;
    int ks, rk, wide;                              // K-steps per half; rows of an R2 box; r > 32
    int maxseg, cap;                               // candidate lists per token block in scratch, entries per list and token
    int nst, st_bytes, zbufs, z_bytes;
    int off_r2, off_pub, off_ctl;
    int list_cap, list_shift;                      // places of a list; log2 of the CTAs whose lists lie side by side (0, 1, 2)
    uint8_t* list;                                 // [CTA >> shift][list_cap][512 = (CTA, 32-token quarter), column quarter, lane] x 32 bytes
    uint2* ent;                                    // [block][seg][128][cap] (logit bits, expert id)
    int* cnt;                                      // [block][seg][128]
    float2* mz;                                    // [block][seg][128] (max in log2 units, sum); LSE only
    int* status;
};

__device__ __forceinline__ uint32_t divide(uint32_t x, uint32_t d, uint32_t inv)        // x / d, inv = (2^32 - 1) / d
{
    const uint32_t q = __umulhi(x, inv);           // x / d or one less
    return x - q * d >= d ? q + 1 : q;
}
// CTA that owns unit u; the part of CTA c, [total c / g, total (c + 1) / g), as a block, a step in it and a count; which segment
// of that block its first one is.
__device__ __noinline__ int wide_owner(long long total, int g, long long u) { return (int)(((u + 1) * g - 1) / total); }
__device__ __forceinline__ int owner_of(const Cut& t, long long u)
{
    return t.inv_total ? (int)divide((uint32_t)(u + 1) * (uint32_t)t.g - 1u, (uint32_t)t.total, t.inv_total) : wide_owner(t.total, t.g, u);
}
struct Part {
    int blk, s0, units, seg;
};
__device__ __noinline__ Part wide_part(long long total, int g, int nsteps, int c)
{
    const long long lo = total * c / g, hi = total * (c + 1) / g;
    const int blk = (int)(lo / nsteps), s0 = (int)(lo - (long long)blk * nsteps);
    return Part{blk, s0, (int)(hi - lo), s0 == 0 ? 0 : c - wide_owner(total, g, lo - s0)};
}
__device__ __forceinline__ Part part_of(const Cut& t, int c)
{
    if (!t.inv_total) return wide_part(t.total, t.g, t.nsteps, c);
    const uint32_t total = (uint32_t)t.total, g = (uint32_t)t.g, n = (uint32_t)t.nsteps;
    const uint32_t lo = divide(total * (uint32_t)c, g, t.inv_g), hi = divide(total * (uint32_t)(c + 1), g, t.inv_g);
    const uint32_t blk = divide(lo, n, t.inv_nsteps), s0 = lo - blk * n;
    return Part{(int)blk, (int)s0, (int)(hi - lo), s0 == 0 ? 0 : c - owner_of(t, blk * n)};
}

// 16 consecutive fp32 columns of this thread's tensor-memory lane, complete on return.  (Load and wait in one statement:
// with the destination registers tied to a separate wait the compiler copies them.)
__device__ __forceinline__ void tmem_get16(uint32_t taddr, float (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(taddr)
                 : "memory");
}
// One arrival for a warp whose lanes have all completed their tensor-memory loads (the wait for these is warp-wide).
__device__ __forceinline__ void arrive_lane0(uint32_t bar, int lane)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar), "r"(lane) : "memory");
}
// Wait that lets the caller go on after a time-out (what it computes then is not used): the code that follows keeps its
// warp-uniform control flow and its barriers.
__device__ __forceinline__ void wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status)
{
    (void)mbar_wait(bar, parity, abort_flag, status);
}

// descending compare-exchange, and sorting networks over registers
__device__ __forceinline__ void cx(float& a, float& b)
{
    const float h = fmaxf(a, b);
    b = fminf(a, b);
    a = h;
}
__device__ __forceinline__ void sort8(float (&s)[8])
{
    cx(s[0], s[1]); cx(s[2], s[3]); cx(s[4], s[5]); cx(s[6], s[7]);
    cx(s[0], s[2]); cx(s[1], s[3]); cx(s[4], s[6]); cx(s[5], s[7]);
    cx(s[1], s[2]); cx(s[5], s[6]);
    cx(s[0], s[4]); cx(s[1], s[5]); cx(s[2], s[6]); cx(s[3], s[7]);
    cx(s[2], s[4]); cx(s[3], s[5]);
    cx(s[1], s[2]); cx(s[3], s[4]); cx(s[5], s[6]);
}
template <int N>
__device__ __forceinline__ void bitonic_down(float (&s)[N])
{
#pragma unroll
    for (int d = N / 2; d > 0; d >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i)
            if ((i & d) == 0) cx(s[i], s[i + d]);
}
// Append the groups of four (maxima t, values v, first column col + 4 i) that reach thr to a list that ends at `end`.  The
// four tests come first: only the adds to the list's end depend on each other.  No list's places lie on both sides of a multiple
// of 2^32 bytes (lists_at), and its end is one of them (the last place is never filled), so these are adds to the address's low word.
__device__ __forceinline__ void append4(uint64_t& end, float thr, const float* t, const float* v, int col)
{
#define MORE_APPEND(P, COL, A, B, C, D)                                                                     \
    "mov.b64 at, {lo, hi};\n\t@" P " st.global.v4.f32 [at], {" A ", " B ", " C ", " D "};\n\t@" P " st.global.b32 [at+16], " COL ";\n\t" \
    "@" P " add.u32 lo, lo, %22;\n\t"
    asm volatile(
        "{\n\t.reg .pred p0, p1, p2, p3;\n\t.reg .b32 c1, c2, c3, lo, hi;\n\t.reg .b64 at;\n\tmov.b64 {lo, hi}, %0;\n\t"
        "setp.ge.f32 p0, %2, %1;\n\tsetp.ge.f32 p1, %3, %1;\n\tsetp.ge.f32 p2, %4, %1;\n\tsetp.ge.f32 p3, %5, %1;\n\t"
        "add.u32 c1, %23, 4;\n\tadd.u32 c2, %23, 8;\n\tadd.u32 c3, %23, 12;\n\t"
        MORE_APPEND("p0", "%23", "%6", "%7", "%8", "%9") MORE_APPEND("p1", "c1", "%10", "%11", "%12", "%13")
        MORE_APPEND("p2", "c2", "%14", "%15", "%16", "%17") MORE_APPEND("p3", "c3", "%18", "%19", "%20", "%21")
        "mov.b64 %0, {lo, hi};\n\t}"
        : "+l"(end)
        : "f"(thr), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3]), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]),
          "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]),
          "f"(v[15]), "n"(kEntry), "r"(col)
        : "memory");
#undef MORE_APPEND
}
// the next float above x
__device__ __forceinline__ float just_above(float x)
{
    const int b = x == 0.f ? 0 : __float_as_int(x);
    const int key = (b ^ ((b >> 31) & 0x7fffffff)) + 1;      // ordered as the floats are
    return __int_as_float(key ^ ((key >> 31) & 0x7fffffff));
}

// A thread's list that overflows: rare, and not inlined, so that the sweep's code stays short (a call of a few units fetches
// it from L2 as it runs: T = 64, M = 16384 19.2 -> 18.7 us, T = 14, M = 4472 18.7 -> 18.4; long sweeps are the same).  The
// list's n entries start at `first`.
//
// k-th largest logit of a list (its bits in .x) and how many equal to it are wanted (.y; all of them in a short list).  Starting
// from NaN, which nothing reaches: an infinite logit, of finite inputs that overflow, is one like any other.
__device__ __noinline__ uint2 list_kth(uint64_t first, int n, int k)
{
    float cur = __int_as_float(0x7fffffff);
    int need = k;
    for (;;) {
        float m = -INFINITY;
        int c = 0;
#pragma unroll 1
        for (int i = 0; i < n; ++i) {
            const float4 e = *reinterpret_cast<const float4*>(first + (uint64_t)i * kEntry);
            const float x[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (!(x[j] >= cur)) {
                    if (x[j] > m) { m = x[j]; c = 1; }
                    else if (x[j] == m) ++c;
                }
        }
        if (c >= need || c == 0) return make_uint2(__float_as_uint(m), (uint32_t)need);
        need -= c;
        cur = m;
    }
}
// Drop what is below `known`, which k logits of the token reach, and cut a list that stays long to its k best (later equals
// then lose to those: larger ids).  Returns how many entries are left, and a new threshold.
__device__ __noinline__ uint2 make_room(uint64_t first, int n, float known, int k)
{
    auto keep = [&](float low, int equal) {
        int left = 0;
#pragma unroll 1
        for (int i = 0; i < n; ++i) {
            const uint64_t rd = first + (uint64_t)i * kEntry, wr = first + (uint64_t)left * kEntry;
            const float4 e = *reinterpret_cast<const float4*>(rd);
            const float m = fmaxf(max3(e.x, e.y, e.z), e.w);
            const bool take = m > low || (m == low && equal > 0);
            if (equal > 0) equal -= (e.x == low) + (e.y == low) + (e.z == low) + (e.w == low);
            if (take) {
                *reinterpret_cast<float4*>(wr) = e;
                *reinterpret_cast<int*>(wr + 16) = *reinterpret_cast<const int*>(rd + 16);
                ++left;
            }
        }
        n = left;
    };
    keep(known, INT_MAX);
    if (n > kListCap - kCols / 4) {
        const uint2 kth = list_kth(first, n, k);
        keep(__uint_as_float(kth.x), (int)kth.y);
        known = fmaxf(known, just_above(__uint_as_float(kth.x)));
    }
    return make_uint2((uint32_t)n, __float_as_uint(known));
}

__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate)
{
    if (accumulate)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, 0, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, 0, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc) : "memory");
}

// an accumulator's number, known to the compiler or not
__device__ __forceinline__ int number_of(int i) { return i; }
template <int I>
__device__ __forceinline__ constexpr int number_of(std::integral_constant<int, I>) { return I; }

__device__ __forceinline__ void quarter_sync(int q) { asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory"); }

// The loop over the units has a copy of its body for each accumulator, so that barriers, phases and tensor-memory addresses are
// constants: 92 -> 58 instructions per warp and unit without candidates, T = 32768, h = 512, M = 65536 405 -> 360 us.  SHORT:
// every CTA has few units (kShortUnits).  A call of that size fetches the code from L2 as it runs, so there is only one copy, for
// any unit (T = 1, M = 16384 15.4 -> 14.8 us, T = 64 19.4 -> 18.5; four units per CTA are slower that way: T = 2000, M = 8192
// 33.9 -> 34.4).
constexpr int kShortUnits = 2;
template <int KCAP, bool LSE, bool SHORT>
__global__ void __launch_bounds__(kSThreads, 2)
sweep_kernel(const __grid_constant__ CUtensorMap map_z, const __grid_constant__ CUtensorMap map_r2, const SweepParams p)
{
    constexpr int NB = KCAP <= 8 ? 4 : 8;          // buckets of a thread
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base_ptr + p.off_ctl);
    constexpr int B_ZF = 0, B_ZE = 2, B_RF = 4, B_RE = B_RF + kMaxStages, B_AF = B_RE + kMaxStages, B_AE = B_AF + 2,
                  B_COUNT = B_AE + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    const int warp = __shfl_sync(kFull, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;      // (the compiler sees a uniform value)
    const Part part = part_of(p.cut, (int)blockIdx.x);
    const int nsteps = p.cut.nsteps;

    if (threadIdx.x == 0) {
        for (int i = 0; i < B_AE; ++i) mbar_init(bar(i), 1);
        mbar_init(bar(B_AE), kEpi / 32);
        mbar_init(bar(B_AE + 1), kEpi / 32);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(256)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ===================================================================================== TMA producer
        if (lane == 0) {
            bool ok = true;
            int st = 0, ph = 0;
            const uint32_t r2 = base + p.off_r2;
            auto load_r2 = [&](int step) {
                ok = mbar_wait(bar(B_RE + st), ph ^ 1, abort_flag, p.status);
                if (!ok) return;
                mbar_expect_tx(bar(B_RF + st), p.st_bytes);
#pragma unroll
                for (int j = 0; j < W / 64; ++j)
                    tma_load_2d(r2 + st * p.st_bytes + j * p.rk * 128, &map_r2, bar(B_RF + st), step * W + j * 64, 0);
                if (++st == p.nst) { st = 0; ph ^= 1; }
            };
            int blk = part.blk, s0 = part.s0, seg = 0;
            for (int left = part.units; left > 0 && ok; ++blk, ++seg, s0 = 0) {
                const int steps = min(left, nsteps - s0);
                left -= steps;
                const int lead = lead_of(steps, KCAP > 8), total = steps + (lead > 2 ? lead : 0);
                auto step_of = [&](int v) { return s0 + (v >= lead && lead > 2 ? v - lead : v); };
                int v = 0;
                if (seg == 0) {
                    // R2 comes from the caller, not from the projection: the first stages are requested before waiting for it
                    for (; v < total && v < p.nst && ok; ++v) load_r2(step_of(v));
                    pdl_wait();
                }
                const int zb = seg % p.zbufs;
                if (seg >= p.zbufs) ok = ok && mbar_wait(bar(B_ZE + zb), ((seg / p.zbufs) - 1) & 1, abort_flag, p.status);
                if (!ok) break;
                mbar_expect_tx(bar(B_ZF + zb), p.z_bytes);
                tma_load_2d(base + zb * p.z_bytes, &map_z, bar(B_ZF + zb), 0, blk * kRows);
                if (p.wide) tma_load_2d(base + zb * p.z_bytes + kRows * 128, &map_z, bar(B_ZF + zb), 64, blk * kRows);
                for (; v < total && ok; ++v) load_r2(step_of(v));
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ======================================================================================= MMA issuer
        // One elected lane runs the whole loop, unrolled over the K-steps: with eight or nine other warps on its scheduler
        // every instruction here counts several times, and one unit's MMAs compute for 150 to 584 clocks only.
        constexpr uint32_t idesc = umma_idesc(W);
        auto run = [&](auto ksteps) {
            constexpr int KS = decltype(ksteps)::value;
            const uint64_t zd = umma_desc_sw128(base, 16, 1024), bd = umma_desc_sw128(base + p.off_r2, KS * 2048, 1024);
            const uint32_t lo_off = KS > 2 ? (kRows * 128) >> 4 : 4;     // from the hi half of z to the lo half, in 16 bytes
            int st = 0, ph = 0, seg = 0;
            uint32_t even = 1, odd = 1;                      // phases of the accumulators' "empty" barriers
            int s0 = part.s0;
            for (int left = part.units; left > 0; ++seg, s0 = 0) {
                const int steps = min(left, nsteps - s0);
                left -= steps;
                const int lead = lead_of(steps, KCAP > 8), total = steps + (lead > 2 ? lead : 0);
                const int zb = p.zbufs == 2 ? seg & 1 : 0, zuse = p.zbufs == 2 ? seg >> 1 : seg;
                wait_or_abort(bar(B_ZF + zb), zuse & 1, abort_flag, p.status);
                const uint64_t z = zd + zb * (p.z_bytes >> 4);
                for (int v = 0; v < total; ++v) {
                    const int buf = (lead > 2 && v >= lead ? v - lead : v) & 1;
                    const uint32_t free = buf ? odd : even;
                    (buf ? odd : even) ^= 1;
                    // (both are mostly complete: two tests, one branch)
                    if (!(mbar_try_wait(bar(B_RF + st), ph) & mbar_try_wait(bar(B_AE + buf), free))) {
                        wait_or_abort(bar(B_RF + st), ph, abort_flag, p.status);
                        wait_or_abort(bar(B_AE + buf), free, abort_flag, p.status);
                    }
                    tc_fence_after();
                    const uint64_t b = bd + st * (p.st_bytes >> 4);
                    const uint32_t d = tmem_base + buf * W;
                    // hi, then lo, into one accumulator: z K-major (+32 bytes per K-step), R2 MN-major (+16 rows of 128 bytes)
#pragma unroll
                    for (int j = 0; j < KS; ++j) mma_ss(d, z + 2 * j, b + 128 * j, idesc, j != 0);
#pragma unroll
                    for (int j = 0; j < KS; ++j) mma_ss(d, z + lo_off + 2 * j, b + 128 * j, idesc, true);
                    tc_commit(bar(B_AF + buf));
                    tc_commit(bar(B_RE + st));
                    if (++st == p.nst) { st = 0; ph ^= 1; }
                }
                tc_commit(bar(B_ZE + zb));
            }
        };
        if (elect_one()) {
            if (p.ks == 4) run(std::integral_constant<int, 4>{});
            else if (p.ks == 3) run(std::integral_constant<int, 3>{});
            else if (p.ks == 2) run(std::integral_constant<int, 2>{});
            else run(std::integral_constant<int, 1>{});
        }
        __syncwarp();
    } else {
        // ======================================================================================== selection
        const int q = warp & 3;                              // tensor-memory lane quarter
        const int sub = (warp - 2) >> 2;                     // column quarter
        const int row = q * 32 + lane;                       // token of the block
        const int M = p.M;
        const uint32_t t_col = tmem_base + ((uint32_t)(q * 32) << 16) + sub * kCols;
        // the thread's list; a unit adds at most 8 entries between two looks at its length
        // (A list of fewer than kListCap places is one whose last place so few units cannot reach; `warn` is then that place, and
        // nothing comes behind it.  Where only one or two quarters of the block hold tokens, four or two CTAs share an area: the
        // other quarters' warps touch no lists.)
        const uint32_t side = ((blockIdx.x & ((1u << p.list_shift) - 1)) << (2 - p.list_shift)) + q;
        const uint64_t first = reinterpret_cast<uint64_t>(p.list) + (uint64_t)(blockIdx.x >> p.list_shift) * (p.list_cap * kEntry) +
                               (side * (kEpi / 4) + sub * 32 + lane) * 32;
        const int warn_at = min(kListCap - kCols / 4, p.list_cap - 1);
        const uint64_t warn = first + warn_at * kEntry;
        // shared memory: published buckets [sub][128][NB], thresholds [128], counters [128], (m, Z) [sub - 1][128]
        const uint32_t pub0 = base + p.off_pub + row * (NB * 4);
        const uint32_t s_thr = base + p.off_pub + 4 * kRows * NB * 4 + row * 4;
        const uint32_t s_cnt = s_thr + kRows * 4;
        const uint32_t s_mz = base + p.off_pub + 4 * kRows * NB * 4 + kRows * 8 + row * 8;
        uint32_t even = 0, odd = 0;                          // phases of the accumulators' "full" barriers; a segment begins with the first
        float b[NB];
        float thr, m2, zsum;
        uint64_t ptr;                                        // where the next entry goes

        auto lds = [&](uint32_t a) { float v; asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory"); return v; };
        auto sts = [&](uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); };
        auto ent4 = [&](uint64_t o) { return *reinterpret_cast<const float4*>(o); };
        auto ent_col = [&](uint64_t o) { return *reinterpret_cast<const int*>(o + 16); };
        // (sorted: which bucket a set of columns is in does not matter, only that the sets are disjoint)
        auto publish = [&]() {
            if constexpr (NB == 4) {
                cx(b[0], b[1]); cx(b[2], b[3]); cx(b[0], b[2]); cx(b[1], b[3]); cx(b[1], b[2]);
            } else {
                sort8(b);
            }
#pragma unroll
            for (int i = 0; i < NB; i += 4)
                asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                             ::"r"(pub0 + sub * (kRows * NB * 4) + i * 4), "f"(b[i]), "f"(b[i + 1]), "f"(b[i + 2]), "f"(b[i + 3]) : "memory");
        };
        // threshold of the token from the published buckets of its four threads
        auto compute_thr = [&]() {
            auto fetch4 = [&](uint32_t at, float* x) {
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "r"(at) : "memory");
            };
            // 2 NB values at `at` and behind it, in descending order
            auto fetch_pair = [&](uint32_t at, float (&x)[2 * NB]) {
#pragma unroll
                for (int i = 0; i < NB; i += 4) fetch4(at + i * 4, x + i);
                float y[NB];
#pragma unroll
                for (int i = 0; i < NB; i += 4) fetch4(at + kRows * NB * 4 + i * 4, y + i);
#pragma unroll
                for (int i = 0; i < NB; ++i) x[NB + i] = y[NB - 1 - i];
                bitonic_down(x);
            };
            // the 2 NB best of two sorted lists: entry against mirrored entry
            float a[2 * NB], y[2 * NB];
            fetch_pair(pub0, a);
            fetch_pair(pub0 + 2 * kRows * NB * 4, y);
#pragma unroll
            for (int i = 0; i < 2 * NB; ++i) a[i] = fmaxf(a[i], y[2 * NB - 1 - i]);
            float kth = a[0];
            if (p.k == 2 * NB) {
#pragma unroll
                for (int i = 1; i < 2 * NB; ++i) kth = fminf(kth, a[i]);
            } else {
                bitonic_down(a);
                kth = a[0];
#pragma unroll
                for (int i = 1; i < 2 * NB; ++i) kth = (i < p.k) ? a[i] : kth;
            }
            return kth;
        };
        // Make room in the lists of a warp.  The bound that k logits are known to reach is not thr, which may lie just above logits
        // that the list has to keep: it was raised when enough of their equals were in.
        auto compact = [&]() {
            float known = lds(s_thr);
            if (p.k <= NB) {
                float mine = b[0];
#pragma unroll
                for (int i = 1; i < NB; ++i) mine = fminf(mine, b[i]);
                known = fmaxf(known, mine);
            }
            const uint2 left = make_room(first, (int)((ptr - first) / kEntry), known, p.k);
            ptr = first + (uint64_t)left.x * kEntry;
            thr = fmaxf(thr, __uint_as_float(left.y));
            __syncwarp();
        };
        // Candidates of the list that beat `low` -> scratch, and of those that equal it the first `equal`; with `every`, only
        // while fewer than `equal` have been passed on at all: where k of this thread are not below `low`, later equals lose.
        auto emit = [&](uint2* dst, float low, int equal, bool every) {
            constexpr int U = 4;                             // (independent loads: one round trip for four entries, columns and all;
                                                             // a trip for each column cost 2 % of most sweeps)
            for (uint64_t o = first; o < ptr; o += U * kEntry) {
                float4 e[U];
                int c[U];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    e[i] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                    c[i] = 0;
                    if (o + i * kEntry < ptr) { e[i] = ent4(o + i * kEntry); c[i] = ent_col(o + i * kEntry); }
                }
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    if (!(fmaxf(max3(e[i].x, e[i].y, e[i].z), e[i].w) >= low) || o + i * kEntry >= ptr) continue;
                    const float x[4] = {e[i].x, e[i].y, e[i].z, e[i].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool eq = x[j] == low && equal > 0;
                        if (x[j] > low || eq) {
                            equal -= eq || every ? 1 : 0;
                            int at;
                            asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(at) : "r"(s_cnt) : "memory");
                            if (at < p.cap) dst[at] = make_uint2(__float_as_uint(x[j]), (uint32_t)(c[i] + j));
                        }
                    }
                }
            }
        };

        // (units of this CTA as a block, a step in it and a count: 32-bit loop state)
        int blk = part.blk, s0 = part.s0;
        for (int left = part.units; left > 0; ++blk, s0 = 0) {
            const int steps = min(left, nsteps - s0);
            left -= steps;
            const int live = min(kRows, p.T - blk * kRows);
            const bool warp_live = q * 32 < live;
            const bool row_live = row < live;
#pragma unroll
            for (int i = 0; i < NB; ++i) b[i] = -INFINITY;
            thr = row_live ? -FLT_MAX : INFINITY;
            m2 = -INFINITY;
            zsum = 0.f;
            ptr = first;
            const int lead = lead_of(steps, KCAP > 8), again = lead > 2 ? lead : 0;      // units ahead, and how many of them come again
            int next = (lead + (lead + 1) / 2 + 1) & ~1, turn = 0;
            // A token whose logits are all equal (padding) would overflow its list again and again.  So, once, when some thread
            // of the warp first has more than `limit` groups: where the threshold is final from the start, those k reach it
            // and later ones that only equal it lose to them; elsewhere, if the first and the last group have the same
            // maximum, the same holds for the smallest maximum in the list.  (All tokens zero: T = 4096, M = 16384 450 us
            // -> 74, M = 65536 466 -> 135.)
            uint64_t limit = first + min(lead == steps ? max(p.k, 8) : max(p.k + 8, 16), warn_at) * kEntry;
            auto full = [&]() {
                if (limit < warn && ptr > limit) {
                    if (lead == steps) {
                        thr = fmaxf(thr, just_above(lds(s_thr)));
                    } else {
                        auto top = [&](uint64_t o) { const float4 e = ent4(o); return fmaxf(max3(e.x, e.y, e.z), e.w); };
                        float least = top(first);
                        if (least == top(ptr - kEntry)) {
#pragma unroll 1
                            for (uint64_t o = first + kEntry; o < ptr; o += kEntry) least = fminf(least, top(o));
                            thr = fmaxf(thr, just_above(least));
                        }
                    }
                }
                if (__any_sync(kFull, ptr > warn)) compact();
                limit = warn;
            };
            // maxima of 16 columns' groups of four; what lies beyond M is nothing (M is a multiple of 8)
            auto group_max = [&](auto masked, const float (&v)[16], int col, float (&t)[4]) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    t[i] = fmaxf(max3(v[4 * i], v[4 * i + 1], v[4 * i + 2]), v[4 * i + 3]);
                    if (decltype(masked)::value && col + 4 * i >= M) t[i] = -INFINITY;
                }
            };
            // buckets of 16 columns at h in a unit: a bucket per 8 columns, or per 4
            auto bucket = [&](int h, const float (&t)[4]) {
                if constexpr (NB == 4) {
                    b[h / 8] = max3(b[h / 8], t[0], t[1]);
                    b[h / 8 + 1] = max3(b[h / 8 + 1], t[2], t[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) b[h / 4 + i] = fmaxf(b[h / 4 + i], t[i]);
                }
            };
            // ---- the buckets of the first units, for a threshold to start with
            const int whole = min(steps, M / W - s0);    // units that do not reach beyond M
            auto lead_unit = [&](auto buf_c, auto masked, int s) {
                const int buf = number_of(buf_c);
                const int col0 = (s0 + s) * W + sub * kCols;
                wait_or_abort(bar(B_AF + buf), buf ? odd : even, abort_flag, p.status);
                if (again) (buf ? odd : even) ^= 1;          // (otherwise it is read where it is)
                const int valid = M - (s0 + s) * W;
                if (warp_live && NB == 4 && decltype(masked)::value && valid <= W / 2 && lead == steps) {
                    // Half a unit or less: in groups of four columns that go round the token's threads they fill up to all 16 of
                    // its buckets.  (Eight columns to a bucket gave 40 columns five: no threshold for k > 5, every logit a
                    // candidate and the scratch's share of them exceeded.  T = 256, h = 704, r = 40, M = 5800, one unit per CTA:
                    // k = 8 50.4 -> 26.1 us, k = 4 22.9 -> 19.7; T = 1, M = 16424 26.0 -> 14.0.)
                    tc_fence_after();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int c = 4 * (sub + 4 * i);
                        uint32_t x[4];
                        tmem_ld4(t_col - sub * kCols + buf * W + c, x);
                        tmem_ld_wait4(x);
                        const float m = fmaxf(max3(__uint_as_float(x[0]), __uint_as_float(x[1]), __uint_as_float(x[2])), __uint_as_float(x[3]));
                        if (c < valid) b[i] = fmaxf(b[i], m);
                    }
                } else if (warp_live) {
                    tc_fence_after();
#pragma unroll
                    for (int h = 0; h < kCols; h += 16) {
                        float v[16], t[4];
                        tmem_get16(t_col + buf * W + h, v);
                        group_max(masked, v, col0 + h, t);
                        bucket(h, t);
                    }
                }
                if (again) {
                    tc_fence_before();
                    arrive_lane0(bar(B_AE + buf), lane);
                }
            };
            constexpr std::integral_constant<int, 0> first_acc{};
            constexpr std::integral_constant<int, 1> second_acc{};
            {
                int s = 0;
                if constexpr (!SHORT) {
#pragma unroll 1
                    for (; s + 1 < min(lead, whole); s += 2) {
                        lead_unit(first_acc, std::false_type{}, s);
                        lead_unit(second_acc, std::false_type{}, s + 1);
                    }
                }
#pragma unroll 1
                for (; s < lead; ++s) lead_unit(s & 1, std::true_type{}, s);       // (left over, or reaching beyond M)
            }
            if (warp_live) {
                // (published by all four threads of a token before anyone reads: nothing of an earlier block is seen)
                publish();
                quarter_sync(q);
                const float t0 = compute_thr();
                sts(s_thr, t0);                              // (by all four, or a fast one could still read an earlier block's)
                thr = fmaxf(thr, t0);
                if (again) {                                 // (those units come again, and must not be in two buckets)
#pragma unroll
                    for (int i = 0; i < NB; ++i) b[i] = -INFINITY;
                }
            }
            // One unit.  (One that reaches beyond M is an instantiation of its own, so that the others carry no masking.)
            auto unit = [&](auto buf_c, auto masked, int s) {
                constexpr bool kMasked = decltype(masked)::value;
                const int buf = number_of(buf_c);
                const int col0 = (s0 + s) * W + sub * kCols;
                const uint32_t t_acc = t_col + buf * W;
                wait_or_abort(bar(B_AF + buf), buf ? odd : even, abort_flag, p.status);
                (buf ? odd : even) ^= 1;
                tc_fence_after();
                const float raised = lds(s_thr);             // (used after the accumulator's first columns have arrived)
#pragma unroll
                for (int h = 0; h < kCols; h += 16) {
                    const int col = col0 + h;
                    float v[16], t[4];
                    tmem_get16(t_acc + h, v);
                    if (h == 0) thr = fmaxf(thr, raised);
                    if (h + 16 == kCols) {
                        tc_fence_before();
                        arrive_lane0(bar(B_AE + buf), lane);         // everything is in registers: hand the accumulator back
                    }
                    group_max(masked, v, col, t);
                    const float m = fmaxf(max3(t[0], t[1], t[2]), t[3]);
                    if (LSE) {
                        const float c2 = m * kLog2e;
                        if (c2 > m2) { zsum *= ex2f(m2 - c2); m2 = c2; }
                        const uint64_t scale = pack2(kLog2e, kLog2e), low = pack2(-m2, -m2);
                        uint64_t a01 = 0, a23 = 0;
#pragma unroll
                        for (int i = 0; i < 16; i += 8) {
                            if (kMasked && col + i >= M) break;
#pragma unroll
                            for (int j = i; j < i + 8; j += 4) {
                                float x0, x1, x2, x3;
                                unpack2(fma2(pack2(v[j], v[j + 1]), scale, low), x0, x1);
                                unpack2(fma2(pack2(v[j + 2], v[j + 3]), scale, low), x2, x3);
                                a01 = add2(a01, pack2(ex2f(x0), ex2f(x1)));
                                a23 = add2(a23, pack2(ex2f(x2), ex2f(x3)));
                            }
                        }
                        float a0, a1;
                        unpack2(add2(a01, a23), a0, a1);
                        zsum += a0 + a1;
                    }
                    if (__any_sync(kFull, m >= thr)) {
                        // (a bucket matters only once it reaches the threshold, so it need not be kept up elsewhere)
                        bucket(h, t);
                        append4(ptr, thr, t, v, col);
                        if (__builtin_expect(__any_sync(kFull, (uint32_t)ptr > (uint32_t)limit), 0)) full();
                    }
                }
            };
            if (!warp_live) {
                for (int s = 0; s < steps; ++s) {
                    const int buf = s & 1;
                    wait_or_abort(bar(B_AF + buf), buf ? odd : even, abort_flag, p.status);
                    (buf ? odd : even) ^= 1;
                    arrive_lane0(bar(B_AE + buf), lane);
                }
            } else {
                int s = 0;
                while (!SHORT && s + 1 < whole) {
                    const int stop = min(whole - 1, next);           // a run of pairs, up to the next refresh of the threshold
#pragma unroll 1
                    for (; s < stop; s += 2) {
                        unit(first_acc, std::false_type{}, s);
                        unit(second_acc, std::false_type{}, s + 1);
                    }
                    if (s == next) {
                        publish();
                        if (sub == (turn & 3)) sts(s_thr, compute_thr());
                        ++turn;
                        next += ((next + 1) / 2 + 1) & ~1;
                    }
                }
#pragma unroll 1
                for (; s < steps; ++s) unit(s & 1, std::true_type{}, s);   // (left over, or reaching beyond M)
            }
            // ---- end of the segment: what still reaches the threshold goes to scratch
            if (warp_live) {
                const bool final = lead == steps;                    // (the threshold is that of all units already)
                if (!final) publish();
                if (sub == 0) asm volatile("st.shared.u32 [%0], 0;" ::"r"(s_cnt) : "memory");
                if (LSE && sub > 0)
                    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(s_mz + (sub - 1) * (kRows * 8)), "f"(m2), "f"(zsum) : "memory");
                quarter_sync(q);
                const float low = fmaxf(final ? lds(s_thr) : compute_thr(), -FLT_MAX);
                const int seg = blk == part.blk ? part.seg : 0;
                const size_t slot = (size_t)blk * p.maxseg + seg;
                uint2* dst = p.ent + (slot * kRows + row) * p.cap;
                if (row_live) emit(dst, low, p.k, true);
                quarter_sync(q);
                int total = __float_as_int(lds(s_cnt));
                if (__builtin_expect(__any_sync(kFull, total > p.cap), 0)) {              // (the same in all four warps)
                    // more than the scratch holds: the threads of such a token pass on their own k best each
                    quarter_sync(q);
                    if (sub == 0 && total > p.cap) sts(s_cnt, 0.f);
                    quarter_sync(q);
                    if (row_live && total > p.cap) {
                        const uint2 kth = list_kth(first, (int)((ptr - first) / kEntry), p.k);
                        emit(dst, __uint_as_float(kth.x), (int)kth.y, false);
                    }
                    quarter_sync(q);
                    total = __float_as_int(lds(s_cnt));
                }
                if (sub == 0 && row_live) {
                    p.cnt[slot * kRows + row] = min(total, p.cap);
                    if (LSE) {
                        float m = m2, z = zsum;
#pragma unroll
                        for (int o = 0; o < 3; ++o) {
                            float om, oz;
                            asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(om), "=f"(oz) : "r"(s_mz + o * (kRows * 8)) : "memory");
                            if (om > -INFINITY) {
                                const float nm = fmaxf(m, om);
                                z = z * ex2f(m - nm) + oz * ex2f(om - nm);
                                m = nm;
                            }
                        }
                        p.mz[slot * kRows + row] = make_float2(m, z);
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    pdl_launch_dependents();
    if (*abort_flag && threadIdx.x == 0)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);         // copies still in flight land before the memory is released
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(256) : "memory");
    }
}

// ================================================================================================= finish
struct FinishParams {
    int T, M, k, gate_mode;
    int share, maxseg, cap;
    Cut cut;
    const uint2* ent;
    const int* cnt;
    const float2* mz;
    int32_t* out_idx;
    float* out_gate;
    int32_t* out_counts;
    float* out_topval;
    float* out_lse;
};

__device__ __forceinline__ void join_mz(float& m, float& z, float om, float oz)
{
    if (om > -INFINITY) {
        const float nm = fmaxf(m, om);
        z = z * ex2f(m - nm) + oz * ex2f(om - nm);
        m = nm;
    }
}
// segments of token block blk
__device__ __forceinline__ int segments_of(const FinishParams& p, int blk)
{
    if (p.share > 0) return p.share;
    const long long u0 = (long long)blk * p.cut.nsteps;
    return owner_of(p.cut, u0 + p.cut.nsteps - 1) - owner_of(p.cut, u0) + 1;
}
__device__ __forceinline__ Cand load_cand(const uint2* at)
{
    const uint2 e = *at;
    return Cand{__uint_as_float(e.x), (int)e.y};
}
// entry `rank` of a token's result; gate = 2^(v log2e - ref2) inv
__device__ __forceinline__ void put_entry(const FinishParams& p, int tok, int rank, Cand c, float ref2, float inv)
{
    const int64_t o = (int64_t)tok * p.k + rank;
    p.out_idx[o] = c.id;
    p.out_gate[o] = ex2f(c.v * kLog2e - ref2) * inv;
    if (p.out_topval) p.out_topval[o] = c.v;
    if ((unsigned)c.id < (unsigned)p.M) atomicAdd(p.out_counts + c.id, 1);        // (non-finite inputs can leave a place unfilled)
}

// One or two segments per token (three where a part begins and ends inside a block): eight threads per token, which hold
// its candidates (k and a few more per segment) in registers and rank them by counting: every logit against every other,
// handed round by shuffles.  Bound by its instructions, so: logits alone are compared, and only if the ranks' sum shows
// that two were equal are the ids; and a warp does as many rounds as its longest token needs.
// (One thread per token that inserts into a sorted list took 27 us for 65536 tokens: one or two warps per scheduler, each
// a chain of dependent instructions.)
constexpr int kFewSegs = 3;
constexpr int kFewRounds = 8;
template <int R, class Fetch>
__device__ __forceinline__ void rank_few(const FinishParams& p, int tok, bool live, int n, int j, float m2, float z, Fetch fetch)
{
    const int k = p.k;
    Cand c[R];
    int rank[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        c[r] = j + 8 * r < n ? fetch(j + 8 * r) : no_cand();
        rank[r] = 0;
    }
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float o = __shfl_sync(kFull, c[q].v, e, 8);
#pragma unroll
            for (int r = 0; r < R; ++r) rank[r] += o > c[r].v ? 1 : 0;
        }
    int sum = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) sum += j + 8 * r < n ? rank[r] : 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o, 8);
    if (__any_sync(kFull, sum != n * (n - 1) / 2)) {                  // some token has equal logits
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll 1
            for (int e = 0; e < 8; ++e) {
                const float o = __shfl_sync(kFull, c[q].v, e, 8);
                const int id = __shfl_sync(kFull, c[q].id, e, 8);
#pragma unroll
                for (int r = 0; r < R; ++r) rank[r] += (o == c[r].v && id < c[r].id) ? 1 : 0;
            }
    }
    float inv, ref2;
    if (p.gate_mode == MORE_GATE_TOPK_SOFTMAX) {
        float v0 = c[0].v;
#pragma unroll
        for (int r = 1; r < R; ++r) v0 = fmaxf(v0, c[r].v);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v0 = fmaxf(v0, __shfl_xor_sync(kFull, v0, o, 8));
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (j + 8 * r < n && rank[r] < k) s += ex2f((c[r].v - v0) * kLog2e);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o, 8);
        inv = 1.f / s;
        ref2 = v0 * kLog2e;
    } else {
        inv = 1.f / z;
        ref2 = m2;
    }
    if (live) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (j + 8 * r < n && rank[r] < k) put_entry(p, tok, rank[r], c[r], ref2, inv);
        for (int q = n + j; q < k; q += 8) put_entry(p, tok, q, no_cand(), ref2, inv);
    }
}

__global__ void __launch_bounds__(256) finish_few_kernel(const FinishParams p)
{
    __shared__ int s_nseg;
    const int lane = threadIdx.x & 31, j = lane & 7;
    const int want = (blockIdx.x * 256 + threadIdx.x) >> 3;
    const bool live = want < p.T;
    const int tok = live ? want : p.T - 1;                    // (whole warps stay together; what is past the end writes nothing)
    const int blk = tok / kRows, row = tok % kRows;           // (a CTA's 32 tokens lie in one block)
    if (threadIdx.x == 0) s_nseg = segments_of(p, (blockIdx.x * 32) / kRows);
    __syncthreads();
    const int nseg = s_nseg;
    pdl_wait();
    int ends[kFewSegs];                                       // candidates in segments 0 .. s
    float m2 = -INFINITY, z = 0.f;
    {
        int sum = 0;
#pragma unroll
        for (int s = 0; s < kFewSegs; ++s) {
            if (s < nseg) {
                const size_t slot = ((size_t)blk * p.maxseg + s) * kRows + row;
                sum += p.cnt[slot];
                if (p.mz) {
                    const float2 o = p.mz[slot];
                    join_mz(m2, z, o.x, o.y);
                }
            }
            ends[s] = sum;
        }
    }
    const int n = ends[kFewSegs - 1];
    auto fetch = [&](int f) {                                 // candidate f of the token
        int s = 0, before = 0;
#pragma unroll
        for (int q = 0; q + 1 < kFewSegs; ++q)
            if (f >= ends[q]) { s = q + 1; before = ends[q]; }
        return load_cand(p.ent + (((size_t)blk * p.maxseg + s) * kRows + row) * p.cap + (f - before));
    };
    const int rounds = (__reduce_max_sync(kFull, n) + 7) >> 3;
    if (rounds <= 1) rank_few<1>(p, tok, live, n, j, m2, z, fetch);
    else if (rounds == 2) rank_few<2>(p, tok, live, n, j, m2, z, fetch);
    else if (rounds == 3) rank_few<3>(p, tok, live, n, j, m2, z, fetch);
    else if (rounds == 4) rank_few<4>(p, tok, live, n, j, m2, z, fetch);
    else if (rounds <= kFewRounds) rank_few<kFewRounds>(p, tok, live, n, j, m2, z, fetch);
    else {
        // more candidates than registers (many equal logits): k rounds of a maximum, twice, as the gates need their sum first
        const bool topk = p.gate_mode == MORE_GATE_TOPK_SOFTMAX;
        float sum = 0.f, v0 = 0.f;
        for (int pass = topk ? 0 : 1; pass < 2; ++pass) {
            Cand last{INFINITY, -1};
            for (int r = 0; r < p.k; ++r) {
                Cand top = no_cand();
                for (int f = j; f < n; f += 8) {
                    const Cand x = fetch(f);
                    if (ahead(last, x) && ahead(x, top)) top = x;
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    const Cand x{__shfl_xor_sync(kFull, top.v, o, 8), __shfl_xor_sync(kFull, top.id, o, 8)};
                    if (ahead(x, top)) top = x;
                }
                last = top;
                if (pass == 0) {
                    if (r == 0) v0 = top.v;
                    sum += ex2f((top.v - v0) * kLog2e);
                } else if (j == 0 && live) {
                    put_entry(p, tok, r, top, topk ? v0 * kLog2e : m2, topk ? 1.f / sum : 1.f / z);
                }
            }
        }
    }
    if (j == 0 && live && p.out_lse) p.out_lse[tok] = (m2 + log2f(z)) * kLn2;
}

// The result of one token from its k best, one per lane; called by a whole warp.
__device__ __forceinline__ void put_token(const FinishParams& p, int tok, Cand c, float m2, float z, int lane)
{
    float inv, ref2;
    if (p.gate_mode == MORE_GATE_TOPK_SOFTMAX) {
        const float v0 = __shfl_sync(kFull, c.v, 0);
        float s = lane < p.k ? ex2f((c.v - v0) * kLog2e) : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        inv = 1.f / s;
        ref2 = v0 * kLog2e;
    } else {
        inv = 1.f / z;
        ref2 = m2;
    }
    if (lane < p.k) put_entry(p, tok, lane, c, ref2, inv);
    if (lane == 0 && p.out_lse) p.out_lse[tok] = (m2 + log2f(z)) * kLn2;
}

// Up to kWarpSegs segments per token: a warp per token.
constexpr int kWarpSegs = 64;
// LONG: with up to 512 candidates held in registers, whose loads then are one trip to L2, and not one for each 128 of them, twice
// (T = 700, M = 1024, k = 16 22.5 -> 20.1 us; T = 900, M = 2048, k = 6 17.7 -> 16.5); short code otherwise, as it is fetched as it runs.
constexpr int kLongSure = 64;                      // candidates that are sure; there are 1.4 times as many, in places for up to three
template <bool LONG>
__global__ void __launch_bounds__(256) finish_warp_kernel(const FinishParams p)
{
    __shared__ Cand buf[8][64];
    __shared__ int counts[8][kWarpSegs];
    __shared__ int s_nseg;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tok = blockIdx.x * 8 + warp;
    if (threadIdx.x == 0) s_nseg = segments_of(p, (blockIdx.x * 8) / kRows);
    __syncthreads();
    const int nseg = s_nseg;
    pdl_wait();
    if (tok >= p.T) return;
    const int blk = tok / kRows, row = tok % kRows;
    const size_t slot0 = (size_t)blk * p.maxseg * kRows + row;
    float m2 = -INFINITY, z = 0.f;
    int most = 0;
    for (int s = lane; s < nseg; s += 32) {
        const int c = p.cnt[slot0 + (size_t)s * kRows];
        counts[warp][s] = c;
        most = max(most, c);
        if (p.mz) {
            const float2 o = p.mz[slot0 + (size_t)s * kRows];
            join_mz(m2, z, o.x, o.y);
        }
    }
    if (p.mz) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float om = __shfl_xor_sync(kFull, m2, o), oz = __shfl_xor_sync(kFull, z, o);
            join_mz(m2, z, om, oz);
        }
    }
    most = max(__reduce_max_sync(kFull, most), 1);
    __syncwarp();
    const uint32_t inv = most > 1 ? (uint32_t)(((1ull << 32) - 1) / (uint32_t)most) + 1u : 0u;      // f / most by multiplication
    auto get = [&](int f) {
        const int s = inv ? (int)__umulhi((uint32_t)f, inv) : f, i = f - s * most;
        return i < counts[warp][s] ? load_cand(p.ent + (slot0 + (size_t)s * kRows) * p.cap + i) : no_cand();
    };
    const int n = nseg * most;
    Cand c;
    if (!LONG || n <= 128 || n > 512) c = warp_topk<4>(n, p.k, get, buf[warp], lane);
    else if (n <= 256) c = warp_topk<8>(n, p.k, get, buf[warp], lane);
    else c = warp_topk<16>(n, p.k, get, buf[warp], lane);
    put_token(p, tok, c, m2, z, lane);
}

// More segments than that (a few tokens, whose experts are spread over the whole GPU): a CTA per token, 16 threads per
// segment.  A chain of latencies, so what can be is requested at once: the counts of all of a thread's segments, then their
// entries; 512 threads' maxima are joined to 64, of which the k-th largest bounds the k-th best entry; what reaches it is
// ranked by counting.  Code that runs once is fetched from L2 as it runs, so it is kept short (entries held in registers and
// 20 unrolled tests took 2.5 us where reading them again takes 1).
constexpr int kManyThreads = 512;
constexpr int kSomeThreads = 128;                  // where there are more tokens and fewer segments
constexpr int kManyPer = 10;                       // segments per half warp
constexpr int kManySegs = kManyPer * (kManyThreads / 16);
static_assert(kWarpSegs <= kManyPer * (kSomeThreads / 16), "the smaller CTAs take what a warp takes");
// More near the top than `keep` holds: many logits that equal the bound, of which those with the smallest ids count.  The k-th
// smallest of the 64 groups' smallest ids bounds the k-th smallest of them; collected again with it.  Returns how many.  (Not
// inlined: in the kernel's way it costs every call 0.5 us of instruction fetches.)
constexpr int kKeep = 512;
template <int THREADS>
__device__ __noinline__ int collect_equals(const int* cnt, const uint2* ent, size_t next_ent, int nseg, int k, float thr, int* ids,
                                           Cand* keep, int* count, int* bound)
{
    const int half = threadIdx.x >> 4, hl = threadIdx.x & 15;
    auto each = [&](auto what) {
        const uint2* e = ent;
        const int* c = cnt;
#pragma unroll 1
        for (int s = half; s < nseg; s += THREADS / 16, e += next_ent, c += THREADS / 16 * kRows) {
            const int n = *c;
#pragma unroll 1
            for (int i = hl; i < n; i += 16) {
                const Cand x = load_cand(e + (i - hl));
                if (x.v >= thr && x.v > -INFINITY) what(x);
            }
        }
    };
    int least = INT_MAX;
    each([&](Cand x) { if (x.v == thr) least = min(least, x.id); });
#pragma unroll
    for (int o = 1; o < THREADS / 64; o <<= 1) least = min(least, __shfl_xor_sync(kFull, least, o));
    if (threadIdx.x % (THREADS / 64) == 0) ids[threadIdx.x / (THREADS / 64)] = least;
    __syncthreads();                                          // (also: everyone has read the count)
    if (threadIdx.x == 0) *count = 0;
    if (threadIdx.x < 64) {
        const int mine = ids[threadIdx.x];
        int rank = 0;
#pragma unroll 1
        for (int j = 0; j < 64; ++j) rank += (ids[j] < mine) | ((ids[j] == mine) & (j < (int)threadIdx.x));
        if (rank == k - 1) *bound = mine;
    }
    __syncthreads();
    const int last = *bound;
    each([&](Cand x) {
        if (x.v > thr || x.id <= last) {
            const int at = atomicAdd(count, 1);
            if (at < kKeep) keep[at] = x;
        }
    });
    __syncthreads();
    return *count;
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS) finish_many_kernel(const FinishParams p)
{
    constexpr int kWarps = THREADS / 32, kGroup = THREADS / 64;
    __shared__ __align__(16) float maxima[64];
    __shared__ float2 smz[kWarps];
    __shared__ Cand keep[kKeep];
    __shared__ Cand buf[64];
    __shared__ int s_count, s_nseg, s_last;
    __shared__ float s_thr;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tok = blockIdx.x;
    const int blk = tok / kRows, row = tok % kRows;
    if (threadIdx.x == 0) { s_nseg = segments_of(p, blk); s_count = 0; }
    if (threadIdx.x < 64) buf[threadIdx.x] = no_cand();
    __syncthreads();
    const int nseg = s_nseg;
    const size_t slot0 = (size_t)blk * p.maxseg * kRows + row;
    const int half = threadIdx.x >> 4, hl = threadIdx.x & 15;
    const int* const my_cnt = p.cnt + slot0 + (size_t)half * kRows;
    const uint2* const my_ent = p.ent + (slot0 + (size_t)half * kRows) * p.cap + hl;
    const size_t next_ent = (size_t)(THREADS / 16) * kRows * p.cap;
    pdl_wait();
    int c[kManyPer];
#pragma unroll
    for (int u = 0; u < kManyPer; ++u)
        c[u] = half + u * (THREADS / 16) < nseg ? my_cnt[u * (THREADS / 16) * kRows] : 0;
    float m2 = -INFINITY, z = 0.f;
    if (p.mz) {
        for (int s = threadIdx.x; s < nseg; s += THREADS) {
            const float2 o = p.mz[slot0 + (size_t)s * kRows];
            join_mz(m2, z, o.x, o.y);
        }
    }
    float m = -INFINITY;
    {
        float x[kManyPer], y[kManyPer];
        const uint2* e = my_ent;
#pragma unroll
        for (int u = 0; u < kManyPer; ++u, e += next_ent) {
            x[u] = hl < c[u] ? __uint_as_float(e->x) : -INFINITY;
            y[u] = hl + 16 < c[u] ? __uint_as_float(e[16].x) : -INFINITY;
        }
        e = my_ent;
#pragma unroll
        for (int u = 0; u < kManyPer; ++u, e += next_ent) {
            m = max3(m, x[u], y[u]);
            for (int i = hl + 32; i < c[u]; i += 16) m = fmaxf(m, __uint_as_float(e[i - hl].x));
        }
    }
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));     // a group of threads' maximum: 64 of them
    if (lane % kGroup == 0) maxima[threadIdx.x / kGroup] = m;
    if (p.mz) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float om = __shfl_xor_sync(kFull, m2, o), oz = __shfl_xor_sync(kFull, z, o);
            join_mz(m2, z, om, oz);
        }
        if (lane == 0) smz[warp] = make_float2(m2, z);
    }
    __syncthreads();
    if (threadIdx.x < 64) {
        const int me = threadIdx.x;
        const float mine = maxima[me];
        int rank = 0;
#pragma unroll
        for (int j = 0; j < 64; j += 4) {
            const float4 o = *reinterpret_cast<const float4*>(maxima + j);
            rank += (o.x > mine) + (o.y > mine) + (o.z > mine) + (o.w > mine);
            rank += ((o.x == mine) & (j < me)) + ((o.y == mine) & (j + 1 < me)) + ((o.z == mine) & (j + 2 < me)) + ((o.w == mine) & (j + 3 < me));
        }
        if (rank == p.k - 1) s_thr = mine;
    }
    __syncthreads();
    const float thr = s_thr;
    if (m >= thr && m > -INFINITY) {                          // (few threads: their entries are read again, from L1)
        const uint2* e = my_ent;
#pragma unroll 1
        for (int s = half; s < nseg; s += THREADS / 16, e += next_ent) {
            const int count = p.cnt[slot0 + (size_t)s * kRows];
#pragma unroll 1
            for (int i = hl; i < count; i += 16) {
                const Cand x = load_cand(e + (i - hl));
                if (x.v >= thr && x.v > -INFINITY) {
                    const int at = atomicAdd(&s_count, 1);
                    if (at < kKeep) keep[at] = x;
                }
            }
        }
    }
    __syncthreads();
    int n = s_count;
    if (__builtin_expect(n > kKeep, 0)) {
        n = collect_equals<THREADS>(p.cnt + slot0 + (size_t)half * kRows, my_ent, next_ent, nseg, p.k, thr, reinterpret_cast<int*>(maxima), keep,
                           &s_count, &s_last);
    }
    if (n <= kKeep) {
        for (int i = threadIdx.x; i < n; i += THREADS) {
            const Cand e = keep[i];
            int rank = 0;
            for (int j = 0; j < n; ++j) {
                const Cand o = keep[j];
                rank += (o.v > e.v) | ((o.v == e.v) & (o.id < e.id));
            }
            if (rank < p.k) buf[rank] = e;
        }
        __syncthreads();
    }
    if (warp == 0) {
        Cand best = lane < p.k ? buf[lane] : no_cand();
        if (n > kKeep) {
            // more near the top than the buffer holds (many equal logits): over all of them
            const int most = p.cap;
            best = warp_topk<1>(nseg * most, p.k, [&](int f) {
                const int s = f / most, i = f - s * most;
                const size_t slot = slot0 + (size_t)s * kRows;
                return i < p.cnt[slot] ? load_cand(p.ent + slot * p.cap + i) : no_cand();
            }, buf, lane);
        }
        m2 = smz[0].x;
        z = smz[0].y;
        if (p.mz)
            for (int w = 1; w < kWarps; ++w) join_mz(m2, z, smz[w].x, smz[w].y);
        put_token(p, tok, best, m2, z, lane);
    }
}

// ================================================================================================ host side
constexpr int kSweepSmem = (228 * 1024 - 2 * 1024) / 2;     // two CTAs per SM

// Raise a kernel's dynamic shared-memory limit once per device; guarded by the API mutex.
template <class K>
bool allow_smem(K kern, int bytes, unsigned long long* done, bool wide_cluster = false)
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (*done >> (dev & 63) & 1ull) return true;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    if (wide_cluster && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    *done |= 1ull << (dev & 63);
    return true;
}

using SweepFn = void (*)(const CUtensorMap, const CUtensorMap, const SweepParams);

template <int KCAP, bool LSE, bool SHORT>
SweepFn sweep_ready()
{
    static unsigned long long done = 0;
    SweepFn f = sweep_kernel<KCAP, LSE, SHORT>;
    return allow_smem(f, kSweepSmem, &done) ? f : nullptr;
}
template <bool SHORT>
SweepFn sweep_fn(int k, bool lse)
{
    if (k <= 8) return lse ? sweep_ready<8, true, SHORT>() : sweep_ready<8, false, SHORT>();
    return lse ? sweep_ready<16, true, SHORT>() : sweep_ready<16, false, SHORT>();
}

template <class... Args>
cudaError_t launch(void (*kern)(Args...), int grid, int block, int smem, cudaStream_t st, bool dependent, int cluster, Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (dependent) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = (unsigned)cluster;
        at[n].val.clusterDim.y = at[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = at;
    cfg.numAttrs = (unsigned)n;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Eight threads per token rank up to two short lists by counting everything against everything; where there is
// more, the threshold of a warp's selection saves more than its 32 lanes per token cost (k = 16: T = 17000,
// M = 8192 121 -> 88 us, T = 32768, M = 4096 174 -> 114; k = 8 with two lists each, T = 17000, M = 4096 54 -> 51).
// A warp goes through many lists one after the other: from about 128 candidates on that are sure, a CTA per token
// is quicker, of 512 threads while all of them fit on the chip in about one go, of 128 for up to five times as many tokens
// as there are candidates.  (h = 512, r = 32; warp, 128, 512 threads: T = 256, M = 8192, k = 8 26.6, 19.3, 17.4 us,
// k = 16 33.6, 23.3, 20.5; T = 512, M = 4096, k = 8 20.7, 18.0, 20.7; T = 1024, M = 8192, k = 16 39.3, 32.4, 40.3,
// k = 4 21.2, 21.9, 30.1; T = 2048, M = 8192, k = 8 28.3, 31.9.  On 500 shapes drawn from T = 1 ... 12 k, M = 256 ... 32 k, k = 1 ... 16 the
// rule costs 0.4 % on average against the best of the four for each, more than 5 % at 1.6 % of them and 13 % at most; the best one
// for all, a warp with the candidates in registers, 3.6 %.)
cudaError_t finish(const FinishParams& fp, int tokens, int maxseg, bool few, int sms, cudaStream_t st)
{
    const int sure = maxseg * fp.k;
    if (few) return launch(finish_few_kernel, (tokens + 31) / 32, 256, 0, st, true, 1, fp);
    if (maxseg > kWarpSegs || (tokens <= 2 * sms && maxseg >= 16 && sure >= 128))
        return launch(finish_many_kernel<kManyThreads>, tokens, kManyThreads, 0, st, true, 1, fp);
    if (sure >= 128 && tokens <= 5 * sure) return launch(finish_many_kernel<kSomeThreads>, tokens, kSomeThreads, 0, st, true, 1, fp);
    if (sure >= kLongSure) return launch(finish_warp_kernel<true>, (tokens + 7) / 8, 256, 0, st, true, 1, fp);
    return launch(finish_warp_kernel<false>, (tokens + 7) / 8, 256, 0, st, true, 1, fp);
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

constexpr int kChunkTokens = 131072;               // tokens per pass: bounds the scratch, whatever T is
long long resident_ctas(int sm_count) { return 2 * sm_count < kManySegs - 2 ? 2 * sm_count : kManySegs - 2; }

struct Layout {
    size_t z, list, ent, cnt, mz, total;
};
int list_areas(const Plan& p) { return (p.parts - 1 >> p.list_shift) + 1; }

// The largest there is (T >= 131072, k = 16, r > 32): 32 MiB of z, 297 MiB of lists, 130 MiB of candidates and counts.
Layout layout_of(const RouteArgs& a, const Plan& p, bool lse)
{
    Layout L{};
    const size_t tokens = (size_t)(a.T < kChunkTokens ? a.T : kChunkTokens);
    const size_t blocks = (tokens + kRows - 1) / kRows, lists = (size_t)p.sweep_blocks * p.maxseg;
    size_t off = 0;
    L.z = off; off += align_up(blocks * kRows * (a.r <= 32 ? 128 : 256), 1024);
    L.ent = off; off += align_up(lists * (size_t)(4 * a.k) * kRows * 8, 1024);
    L.cnt = off; off += lists * kRows * 4;
    L.mz = off;
    if (lse) off += align_up(lists * kRows * 8, 1024);
    // (last: the finishing kernels' reads then lie at the same addresses however long the lists are; T = 40, M = 6424 26.4 us
    // with the lists in front and 25.1 behind)
    // (one area more than there are, mostly in front of them: lists_at)
    L.list = off; off += (size_t)(list_areas(p) + 1) * p.list_cap * kEntry;
    L.total = off;
    return L;
}

// Where the lists of a scratch at `base` begin.  They end where the scratch does, so that whatever is written behind them meets the
// guard there.  Only where an area would have a multiple of 2^32 bytes between its first and its last byte does it end there
// instead, and all the others move with it: a list's end is advanced by adds to its low word.
uint64_t lists_at(uint64_t base, const Layout& L, const Plan& p)
{
    const uint64_t area = (uint64_t)p.list_cap * kEntry, end = base + L.total, first = end - list_areas(p) * area;
    const uint64_t multiple = ((first >> 32) + 1) << 32;
    return multiple < end ? first - (area - (multiple - first) % area) % area : first;
}

}  // namespace

// Launch plan.  The unit of work is 128 tokens x 128 experts.  Two CTAs per SM get contiguous parts of the line of units,
// either equal ones wherever these begin (stretches of several token blocks are then cut into segments), or an equal share
// of one block each.  The second leaves some SMs idle but every CTA with one segment; what a segment costs on its own (its
// first MMAs, the threshold to start with, the pass through the lists at its end) is worth about eight units.  A forced
// split of s CTAs per token block is the second with that s, in as many launches as it takes for no launch to have more
// CTAs than are resident at once: each has lists of its own, up to 1 MiB (T = 131072, s = 64 in one launch: 64 GiB).
void plan_chain(int T, int M, int msplit, int sm_count, Plan* p)
{
    const long long blocks = ((T < kChunkTokens ? T : kChunkTokens) + kRows - 1) / kRows;
    const long long nsteps = (M + W - 1) / W, total = blocks * nsteps;
    const long long slots = resident_ctas(sm_count);
    const double kSegment = 8.0;
    long long g = total < slots ? total : slots, share = 0, sweep_blocks = blocks;
    if (msplit > 0) {
        share = msplit < nsteps ? msplit : nsteps;
    } else if (blocks <= slots) {
        const long long s = slots / blocks < nsteps ? slots / blocks : nsteps;
        const double whole = (double)((nsteps + s - 1) / s) + kSegment;
        const double cut = (double)total / g + kSegment * (double)((total / g) / nsteps + 2);
        if (blocks == 1 || whole <= cut) share = s;
    }
    if (share > 0) {
        if (blocks * share > slots) sweep_blocks = slots / share > 1 ? slots / share : 1;
        g = sweep_blocks * share;
        p->maxseg = (int)share;
    } else {
        p->maxseg = (int)(g / blocks) + 2;
    }
    p->parts = (int)g;
    p->sweep_blocks = (int)sweep_blocks;
    p->list_shift = T <= 32 ? 2 : (T <= 64 ? 1 : 0);
    // A unit adds at most kCols / 4 entries to a list (a later, shorter chunk may have longer segments).  One place more than
    // those, so that the end of a full list is still a place of it (append4).
    const long long units = share > 0 ? (nsteps + share - 1) / share : (total + g - 1) / g, most = units * (kCols / 4);
    p->list_cap = T <= kChunkTokens && most < kListCap ? (int)most + 1 : kListCap;
    p->ctas = (int)(share > 0 ? blocks * share : g);
    p->msplit = (int)(p->ctas / blocks > 1 ? p->ctas / blocks : 1);      // (whole ones; a part that begins anywhere can reach into two blocks)
    p->share = (int)share;
    p->chain = true;
    p->block_tokens = kRows;
    p->tg = p->es = 1;
}

size_t chain_scratch_bytes(const RouteArgs& a, const Plan& p)
{
    return layout_of(a, p, a.gate_mode == MORE_GATE_FULL_SOFTMAX || a.out_lse != nullptr).total;
}

void chain_lists(const RouteArgs& a, const Plan& p, unsigned long long scratch, unsigned long long* out4)
{
    const Layout L = layout_of(a, p, a.gate_mode == MORE_GATE_FULL_SOFTMAX || a.out_lse != nullptr);
    out4[0] = lists_at(scratch, L, p);
    out4[1] = (unsigned long long)list_areas(p);
    out4[2] = (unsigned long long)p.list_cap;
    out4[3] = kEntry;
}

int launch_finish(const RouteArgs& a, DeviceCtx& ctx, int segments, int cap, const uint2* ent, const int* cnt, const float2* mz)
{
    static_assert(kFinishTokens == kRows && kFinishMaxSegments <= kManySegs, "what the header promises");
    FinishParams fp{};
    fp.T = a.T; fp.M = a.M; fp.k = a.k; fp.gate_mode = a.gate_mode;
    fp.share = fp.maxseg = segments; fp.cap = cap;
    fp.ent = ent; fp.cnt = cnt; fp.mz = mz;
    fp.out_idx = a.out_idx; fp.out_gate = a.out_gate; fp.out_counts = a.out_counts;
    fp.out_topval = a.out_topval; fp.out_lse = a.out_lse;
    if (finish(fp, a.T, segments, false, ctx.sm_count, a.stream) != cudaSuccess) return MORE_ERR_CUDA;
    count_launch(1);
    return MORE_OK;
}

int launch_chain(const RouteArgs& a, DeviceCtx& ctx, const Plan& plan, void* scratch)
{
    const bool lse = a.gate_mode == MORE_GATE_FULL_SOFTMAX || a.out_lse != nullptr;
    const Layout L = layout_of(a, plan, lse);
    char* base = static_cast<char*>(scratch);
    const int n16 = (a.r + 15) / 16 * 16, zc = a.r <= 32 ? 64 : 128;

    SweepParams sp{};
    const int nsteps = (a.M + W - 1) / W;
    sp.M = a.M; sp.k = a.k; sp.ks = n16 / 16; sp.rk = n16; sp.wide = a.r > 32;
    sp.maxseg = plan.maxseg; sp.cap = 4 * a.k;
    sp.st_bytes = W * n16 * 2;
    sp.z_bytes = kRows * zc * 2;
    const int nb = a.k <= 8 ? 4 : 8;
    const int pub = 4 * kRows * nb * 4 + kRows * 8 + 3 * kRows * 8, ctl = 512;
    const int room = kSweepSmem - 1024 - pub - ctl;
    sp.zbufs = zc == 64 ? 2 : 1;
    sp.nst = (room - sp.zbufs * sp.z_bytes) / sp.st_bytes;
    if (sp.nst > kMaxStages) sp.nst = kMaxStages;
    if (sp.nst < 2) return MORE_ERR_SHAPE;
    sp.off_r2 = sp.zbufs * sp.z_bytes;
    sp.off_pub = sp.off_r2 + sp.nst * sp.st_bytes;
    sp.off_ctl = sp.off_pub + pub;
    const int smem = sp.off_ctl + ctl + 1024;
    sp.list = reinterpret_cast<uint8_t*>(lists_at(reinterpret_cast<uint64_t>(base), L, plan));
    sp.list_cap = plan.list_cap; sp.list_shift = plan.list_shift;
    sp.ent = reinterpret_cast<uint2*>(base + L.ent);
    sp.cnt = reinterpret_cast<int*>(base + L.cnt);
    sp.mz = lse ? reinterpret_cast<float2*>(base + L.mz) : nullptr;
    sp.status = ctx.status;

    // (plan.parts CTAs have even parts of the blocks of one launch)
    const long long units = plan.share > 0 ? (nsteps + plan.share - 1) / plan.share
                                           : ((long long)plan.sweep_blocks * nsteps + plan.parts - 1) / plan.parts;
    const bool few = a.T <= kChunkTokens && units <= kShortUnits;
    SweepFn sweep = few ? sweep_fn<true>(a.k, lse) : sweep_fn<false>(a.k, lse);
    static unsigned long long project_done = 0;
    const int psmem_max = kPStages * kPStageBytes + kPCtl + kPExchange + 1024;
    if (!sweep || !allow_smem(project_kernel, psmem_max, &project_done)) return MORE_ERR_CUDA;

    const int sms = ctx.sm_count > 0 ? ctx.sm_count : 148;
    CUtensorMap mr1, mr2;
    int rc = get_tensor_map(a.R1, a.h, a.r, 64, 64, &mr1);
    if (rc == MORE_OK) rc = get_tensor_map(a.R2, a.r, a.M, n16, 64, &mr2);
    if (rc != MORE_OK) return rc;
    for (int t0 = 0; t0 < a.T; t0 += kChunkTokens) {
        const int T = a.T - t0 < kChunkTokens ? a.T - t0 : kChunkTokens;
        const int blocks = (T + kRows - 1) / kRows;
        CUtensorMap mx, mz;
        rc = get_tensor_map(a.X + (size_t)t0 * a.h, T, a.h, kRows, 64, &mx);
        if (rc == MORE_OK) rc = get_tensor_map(base + L.z, blocks * kRows, zc, kRows, 64, &mz);
        if (rc != MORE_OK) return rc;

        ProjectParams pp{};
        pp.T = T; pp.h = a.h; pp.n = n16; pp.zc = zc;
        pp.z = reinterpret_cast<uint32_t*>(base + L.z);
        pp.counts = t0 == 0 ? a.out_counts : nullptr;
        pp.M = a.M;
        pp.status = ctx.status;
        pp.cs = 1;
        const int nkt = (a.h + 63) / 64;
        while (pp.cs < 8 && 2 * pp.cs * blocks <= sms && nkt >= 4 * pp.cs) { pp.cs *= 2; ++pp.cs_bits; }
        const int psmem = psmem_max - (pp.cs == 1 ? kPExchange : 0);
        if (launch(project_kernel, blocks * pp.cs, kPThreads, psmem, a.stream, true, pp.cs, mx, mr1, pp) != cudaSuccess)
            return MORE_ERR_CUDA;
        count_launch(1);

        const int step = plan.share > 0 && plan.sweep_blocks < blocks ? plan.sweep_blocks : blocks;      // blocks per sweep
        for (int b0 = 0; b0 < blocks; b0 += step) {
            const int nblk = blocks - b0 < step ? blocks - b0 : step, first = t0 + b0 * kRows;
            const int tokens = T - b0 * kRows < nblk * kRows ? T - b0 * kRows : nblk * kRows;
            if (b0 > 0) rc = get_tensor_map(base + L.z + (size_t)b0 * kRows * zc * 2, nblk * kRows, zc, kRows, 64, &mz);
            if (rc != MORE_OK) return rc;
            sp.T = tokens;
            const long long total = (long long)nblk * nsteps;
            int g = plan.share > 0 ? nblk * plan.share : plan.parts;
            if (plan.share == 0 && a.T > kChunkTokens) {     // (the last chunk of a long call may be shorter)
                const long long most = (long long)(plan.maxseg - 1) * blocks - 1;  // floor(g / blocks) + 2 <= maxseg
                if (g > total) g = (int)total;
                if (g > most) g = (int)(most > 1 ? most : 1);
            }
            sp.cut = make_cut(total, nsteps, g);
            if (launch(sweep, g, kSThreads, smem, a.stream, true, 1, mz, mr2, sp) != cudaSuccess) return MORE_ERR_CUDA;

            FinishParams fp{};
            fp.T = tokens; fp.M = a.M; fp.k = a.k; fp.gate_mode = a.gate_mode;
            fp.share = plan.share; fp.maxseg = plan.maxseg; fp.cap = sp.cap; fp.cut = sp.cut;
            fp.ent = sp.ent; fp.cnt = sp.cnt; fp.mz = sp.mz;
            const size_t ro = (size_t)first * a.k;
            fp.out_idx = a.out_idx + ro; fp.out_gate = a.out_gate + ro; fp.out_counts = a.out_counts;
            fp.out_topval = a.out_topval ? a.out_topval + ro : nullptr;
            fp.out_lse = a.out_lse ? a.out_lse + first : nullptr;
            if (finish(fp, tokens, plan.maxseg, a.k <= 8 && plan.maxseg <= (plan.share > 0 ? 1 : kFewSegs), sms, a.stream) != cudaSuccess)
                return MORE_ERR_CUDA;
            count_launch(2);
        }
    }
    return MORE_OK;
}

}  // namespace more
