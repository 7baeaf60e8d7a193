// Small selections of the library's second steps (merging candidate lists of one token): a warp keeps the k best of n
// (logit, expert id) pairs.  Internal; every translation unit gets its own copy.
#pragma once

#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

namespace more {

namespace {

struct Cand {
    float v;
    int id;
};

// full order of the result: larger logit first, equal logits by smaller id
__device__ __forceinline__ bool ahead(Cand a, Cand b) { return a.v > b.v || (a.v == b.v && a.id < b.id); }
__device__ __forceinline__ Cand no_cand() { return Cand{-INFINITY, INT_MAX}; }

// one float per lane, sorted over the warp, largest in lane 0
__device__ __forceinline__ float warp_sort_down(float x, int lane)
{
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const float o = __shfl_xor_sync(0xffffffffu, x, stride);
            x = (((lane & size) == 0) == ((lane & stride) == 0)) ? fmaxf(x, o) : fminf(x, o);
        }
    return x;
}

// The k <= 32 best of the candidates get(0) .. get(n - 1) (a logit of -inf is no candidate); lane i returns the i-th best.
// The k-th largest of the 32 lanes' own maxima is reached by at least k candidates, so only what reaches it (about 1.4 k)
// is ranked, by counting.  Up to 32 R candidates are held in registers, more are read twice.  buf: 64 entries of the
// warp's own in shared memory.  All 32 lanes call this together with the same n and k.
template <int R, class Get>
__device__ __forceinline__ Cand warp_topk(int n, int k, Get get, Cand* buf, int lane)
{
    constexpr unsigned kAll = 0xffffffffu;
    Cand c[R];
    float m = -INFINITY;
    const bool held = n <= 32 * R;
    if (held) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            c[r] = no_cand();
            if (32 * r < n && lane + 32 * r < n) c[r] = get(lane + 32 * r);
            m = fmaxf(m, c[r].v);
        }
    } else {
        for (int f = lane; f < n; f += 32) m = fmaxf(m, get(f).v);
    }
    const float thr = __shfl_sync(kAll, warp_sort_down(m, lane), k - 1);
    int count = 0;
    auto take = [&](Cand x, bool in) {
        const unsigned who = __ballot_sync(kAll, in);
        const int at = count + __popc(who & ((1u << lane) - 1u));
        if (in && at < 64) buf[at] = x;
        count += __popc(who);
    };
    if (held) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (32 * r < n) take(c[r], c[r].v >= thr && c[r].v > -INFINITY);
    } else {
        for (int f = lane; f - lane < n; f += 32) {
            const Cand x = f < n ? get(f) : no_cand();
            take(x, x.v >= thr && x.v > -INFINITY);
        }
    }
    if (__builtin_expect(count > 64, 0)) {
        // More than the buffer holds: many logits that equal thr, of which those with the smallest ids count.  The k-th
        // smallest of the 32 lanes' smallest ids bounds the k-th smallest of them; collected again with that.
        float least = -INFINITY;
#pragma unroll 1
        for (int f = lane; f < n; f += 32) {
            const Cand x = get(f);
            if (x.v == thr) least = fmaxf(least, -(float)x.id);
        }
        const float last = -__shfl_sync(kAll, warp_sort_down(least, lane), k - 1);
        __syncwarp();
        count = 0;
#pragma unroll 1
        for (int f = lane; f - lane < n; f += 32) {
            const Cand x = f < n ? get(f) : no_cand();
            take(x, x.v > thr || (x.v == thr && x.v > -INFINITY && (float)x.id <= last));
        }
    }
    __syncwarp();
    Cand best = no_cand();
    if (__builtin_expect(count <= 64, 1)) {
        // Ranks by the logits alone, and by the ids as well only if the ranks' sum shows that two logits were equal.
        Cand mine[2];
        int rank[2], sum = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int pos = lane + 32 * h;
            rank[h] = INT_MAX;
            if (32 * h < count) {
                mine[h] = pos < count ? buf[pos] : no_cand();
                int q = 0;
#pragma unroll 8
                for (int j = 0; j < count; ++j) q += buf[j].v > mine[h].v ? 1 : 0;
                if (pos < count) { rank[h] = q; sum += q; }
            }
        }
        if (__reduce_add_sync(kAll, sum) != count * (count - 1) / 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int pos = lane + 32 * h;
                if (pos < count)
                    for (int j = 0; j < count; ++j) {
                        const Cand o = buf[j];
                        rank[h] += (o.v == mine[h].v && (o.id < mine[h].id || (o.id == mine[h].id && j < pos))) ? 1 : 0;
                    }
            }
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (rank[h] < k) buf[rank[h]] = mine[h];
        __syncwarp();
        if (lane < k && lane < count) best = buf[lane];
    } else {
        // more near the top than the buffer holds (many equal logits): k rounds of a maximum
        Cand before{INFINITY, -1};
#pragma unroll 1
        for (int r = 0; r < k; ++r) {
            Cand top = no_cand();
#pragma unroll 1
            for (int f = lane; f < n; f += 32) {
                const Cand x = get(f);
                if (x.v > -INFINITY && ahead(before, x) && ahead(x, top)) top = x;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const Cand x{__shfl_xor_sync(kAll, top.v, o), __shfl_xor_sync(kAll, top.id, o)};
                if (ahead(x, top)) top = x;
            }
            if (lane == r) best = top;
            before = top;
        }
    }
    __syncwarp();
    return best;
}

}  // namespace

}  // namespace more
