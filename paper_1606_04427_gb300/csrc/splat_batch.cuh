// Batches of tile records, shared by the additive splat (k_splat.cu) and the depth-ordered
// splat (k_ordered.cu).
//
// A warp renders a region of up to 16 x 16 pixels from a tile's record list.  It gathers the
// records that meet the region into a batch in shared memory (batch_fill), finds for each the
// 4 x 4-pixel squares its box meets (batch_words) and lists, per square, the batch positions
// of its records in list order (batch_lists).  The squares are then evaluated by pairs of
// lanes, 2 x 4 pixels per lane, in passes over the squares sorted by list length
// (sort_squares): 16 squares per pass, or fewer with 2^a lane pairs each (choose_split), so
// that the pairs of a warp, which run in step, have lists of like length.
#pragma once

#include "splotch_internal.cuh"

namespace spl {

constexpr int kRegion = 16;  // edge of the region a warp owns, in pixels
constexpr int kAhead = 3;    // 32-record loads in flight

template <int B> struct __align__(16) Batch {
    static_assert(B < 256 && B % 32 == 0, "8-bit list entries; entry B covers nothing");
    static constexpr int kRounds = B / 32;             // records per lane of a full batch
    static constexpr int kWords = (kRounds + 1) / 2;   // 32-record words per lane (two lanes share a square's)
    float4 pa[B + 1];  // raw record, then (-X, -Y, R^2, Gaussian scale); the last entry covers nothing
    float4 pb[B + 1];  // what the record adds
    // per square: batch positions of the records that meet it (a word of padding per square
    // keeps equal places of the 16 lists in different banks)
    unsigned char list[16][B + 4];
    float4 ring[kAhead][32];  // records on their way from the list
};

// 16 bytes from global to shared memory, asynchronously (LDGSTS)
__device__ __forceinline__ void copy16_async(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4_async(void *dst, const void *src) {  // 4 bytes
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() {  // all but the newest N groups done
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void copy_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ uint32_t leading_zeros(uint32_t v) {  // v != 0
    uint32_t z;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(z) : "r"(v));
    return z;
}

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// Region of tw x th pixels at (px0, py0) and its geometry in squares.
struct Region {
    int px0, py0, tw, th;
    float xc, yc, half;     // centre of the pixel centres' box, half its larger extent
    float cx, cy, widen;    // pixel -> square coordinates
    uint32_t ex, ey;        // square columns and rows
};

__device__ __forceinline__ Region make_region(int px0, int py0, int tw, int th) {
    Region g;
    g.px0 = px0, g.py0 = py0, g.tw = tw, g.th = th;
    // A support that covers a pixel centre of the region lies within R of its centres' box:
    // max(|X - xc|, |Y - yc|) < R + half; the widening exceeds the FP32 rounding at any
    // position, so no covered pixel is left out
    const float hx = 0.5f * (float)(tw - 1), hy = 0.5f * (float)(th - 1);
    g.xc = (float)px0 + 0.5f + hx, g.yc = (float)py0 + 0.5f + hy;
    g.half = fmaxf(hx, hy) + 1e-3f + 4e-6f * (g.xc + g.yc);
    g.widen = 2.5e-4f + 1e-6f * (g.xc + g.yc);  // the same in squares
    g.ex = (tw + 3) >> 2, g.ey = (th + 3) >> 2;
    g.cx = -0.25f * ((float)px0 + 0.5f), g.cy = -0.25f * ((float)py0 + 0.5f);
    return g;
}

// Start the first kAhead copies of a list; a lane reads what it copied itself, so waiting for
// its own copies is enough.
template <int B> __device__ __forceinline__ void batch_start(Batch<B> *ws, const float4 *recs, int nrec) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int g = 0; g < kAhead; ++g) {
        if (g * 32 + lane < nrec) copy16_async(&ws->ring[g][lane], recs + g * 32 + lane);
        copy_commit();
    }
}

// Append records base, base + 32, ... that meet the region until the batch is full or the
// list ends; returns the batch's records.  `row` is the ring row of record `base`.
template <bool kEmit, int B>
__device__ __forceinline__ int batch_fill(Batch<B> *ws, const Region &g, const float4 *recs, int nrec, int &base,
                                          int &row, const float4 *emit) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
    int nbuf = 0;
    __syncwarp();
    while (base < nrec && nbuf <= B - 32) {
        copy_wait<kAhead - 1>();
        const float4 rec = ws->ring[row][lane];
        const bool live = base + lane < nrec && fmaxf(fabsf(rec.x - g.xc), fabsf(rec.y - g.yc)) <
                                                    fmaf(rec.z, 1.000004f, g.half);
        const uint32_t bal = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int j = nbuf + __popc(bal & lt_mask);
            ws->pa[j] = rec;
            if constexpr (kEmit)  // the record's last word is the particle index
                copy16_async(&ws->pb[j], &emit[__float_as_uint(rec.w)]);
        }
        nbuf += __popc(bal);
        // the ballot has consumed these records: their row takes the next copy
        const int nx = base + 32 * kAhead + lane;
        if (nx < nrec) copy16_async(&ws->ring[row][lane], recs + nx);
        copy_commit();
        row = row + 1 == kAhead ? 0 : row + 1;
        base += 32;
    }
    __syncwarp();
    return nbuf;
}

// Squares each record's box meets, as one word of 32 records per square and round: lanes s and
// 16 + s share the words of square s.  kOrdered: lane s keeps the first half of the rounds, so
// that the two lanes' parts of the list follow one another in record order; else it keeps the
// even rounds, which shares a batch that is not full more evenly (5.73 against 5.98 ms on the
// 100 M-particle frame, 119 against 150 us on 1 M particles at 637 x 483).  Returns the records
// of the lane's words.
//
// Pixel p of the region (centre p0 + p + 0.5) lies in square p / 4, so the support
// [X - R, X + R] meets squares ceil((X - p0 - 0.5) / 4 - 3 / 4 - R / 4) up to
// floor((X - p0 - 0.5) / 4 + R / 4).  (A record that meets no column or row of the region gets
// an empty or a meaningless mask; its pixels are tested one by one, so it adds nothing either
// way.)
template <bool kOrdered, int W> __device__ __forceinline__ constexpr int round_of(int half, int k) {
    return kOrdered ? half * W + k : 2 * k + half;  // round of word k of a half-warp
}

template <bool kOrdered, int B>
__device__ __forceinline__ int batch_words(const float4 (&rec)[Batch<B>::kRounds], int nbuf, const Region &g,
                                           uint32_t (&word)[Batch<B>::kWords]) {
    constexpr int kRounds = Batch<B>::kRounds, kWords = Batch<B>::kWords;
    const int lane = threadIdx.x & 31;
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < kWords; ++k) word[k] = 0;
#pragma unroll
    for (int k = 0; k < kRounds; ++k) {
        const float rq = fmaf(rec[k].z, 0.250001f, g.widen);
        const float qx = fmaf(rec[k].x, 0.25f, g.cx), qy = fmaf(rec[k].y, 0.25f, g.cy);
        // first square and one past the last (conversions below 0 give 0)
        const uint32_t x0 = __float2uint_ru(qx - (rq + 0.75f)), y0 = __float2uint_ru(qy - (rq + 0.75f));
        const uint32_t x1 = min(g.ex, __float2uint_rd(qx + (rq + 1.0f)));
        const uint32_t y1 = min(g.ey, __float2uint_rd(qy + (rq + 1.0f)));
        const uint32_t m = k * 32 + lane < nbuf ? ((1u << x1) - (1u << x0)) + (((1u << y1) - (1u << y0)) << 4) : 0u;
        uint32_t b[8];  // records of each column (0..3) and row (4..7)
#pragma unroll
        for (int q = 0; q < 8; ++q) b[q] = __ballot_sync(0xffffffffu, m & (1u << q));
        const uint32_t c = (lane & 2) ? ((lane & 1) ? b[3] : b[2]) : ((lane & 1) ? b[1] : b[0]);
        const uint32_t r = (lane & 8) ? ((lane & 4) ? b[7] : b[6]) : ((lane & 4) ? b[5] : b[4]);
        if ((lane >> 4) == (kOrdered ? k / kWords : k & 1)) {
            word[kOrdered ? k % kWords : k >> 1] = c & r;
            cnt += __popc(c & r);
        }
    }
    return cnt;
}

// Per square, the batch positions of its records (kOrdered: in ascending order).  Returns the
// square's (lane & 15) list length.
template <bool kOrdered, int B>
__device__ __forceinline__ int batch_lists(Batch<B> *ws, const uint32_t (&word)[Batch<B>::kWords], int cnt) {
    constexpr int kWords = Batch<B>::kWords;
    const int lane = threadIdx.x & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int other = __shfl_xor_sync(0xffffffffu, cnt, 16);
    const int dst = lane < 16 ? 0 : other;
    // a lane with more than twice the mean is unpacked by the whole warp, a word at a time, so
    // that a dense square does not hold up the others
    const int all = __reduce_add_sync(0xffffffffu, cnt);
    const bool heavy = cnt > max(8, all >> 4);
    for (uint32_t todo = __ballot_sync(0xffffffffu, heavy); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        int at = __shfl_sync(0xffffffffu, dst, src);
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const uint32_t w = __shfl_sync(0xffffffffu, word[k], src);
            if ((w >> lane) & 1u)
                ws->list[src & 15][at + __popc(w & lt_mask)] = (unsigned char)(round_of<kOrdered, kWords>(src >> 4, k) * 32 + lane);
            at += __popc(w);
        }
    }
    if (!heavy) {  // from the last record back
        unsigned char *p = ws->list[lane & 15] + dst + cnt;
#pragma unroll
        for (int k = kWords - 1; k >= 0; --k) {
            const int top = round_of<kOrdered, kWords>(lane >> 4, k) * 32 + 31;
            uint32_t w = word[k];
            while (w) {
                const uint32_t z = leading_zeros(w);
                *--p = (unsigned char)(top - z);
                w ^= 0x80000000u >> z;
            }
        }
    }
    __syncwarp();
    return cnt + other;
}

// Squares sorted by list length, longest first: lane k (and 16 + k) gets place k's key
// (length << 4 | square) and the records before it; total = all records.
__device__ __forceinline__ uint32_t sort_squares(int n, int &before, int &total) {
    const int lane = threadIdx.x & 31;
    uint32_t key = ((uint32_t)n << 4) | (uint32_t)(lane & 15);
#pragma unroll
    for (int size = 2; size <= 16; size <<= 1)
#pragma unroll
        for (int d = size >> 1; d; d >>= 1) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, key, d);
            const bool first = (lane & d) == 0, down = (lane & size & 15) == 0;
            key = (first == down) ? max(key, o) : min(key, o);
        }
    before = (int)(key >> 4);
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, before, d, 16);
        if ((lane & 15) >= d) before += u;
    }
    total = __shfl_sync(0xffffffffu, before, 15);
    before -= (int)(key >> 4);
    return key;
}

// Lane split of the pass that starts at place i, whose square has `lead` records: 2^a pairs
// per square, 16 >> a squares; the a with the most records per instruction (a step of the
// pass loop, the merge of two pairs' sums and a pass cost about kStep, kMerge and kPass).
// Lane a weighs option a.
template <int kStep, int kMerge, int kPass>
__device__ __forceinline__ int choose_split(int i, int lead, int before, int total) {
    const int a = min((int)(threadIdx.x & 31), 4);
    const int end = i + (16 >> a);
    const int upto = __shfl_sync(0xffffffffu, before, min(end, 15));
    const int from = __shfl_sync(0xffffffffu, before, i);
    const int covered = (end > 15 ? total : upto) - from;
    const int steps = (lead + (1 << a) - 1) >> a;
    const float gain = __fdividef((float)covered, (float)(kStep * steps + kMerge * a + kPass));
    return (int)(__reduce_max_sync(0xffffffffu, (__float_as_uint(gain) & ~7u) | (uint32_t)a) & 7u);
}

// Emission of the batch's records from the colormaps, one record per lane and round; the loads
// of all rounds go out together, stage by stage.
template <int R>
__device__ __forceinline__ void batch_colours(const float4 (&rec)[R], const float4 *lut, const int *lut_len,
                                              const int *lut_off, float3 (&e)[R]) {
    int len[R], off[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int type = (int)(__float_as_uint(rec[k].w) >> 24);
        len[k] = __ldg(&lut_len[type]);
        off[k] = __ldg(&lut_off[type]);
    }
    float4 c0[R], c1[R];
    float tau[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const uint32_t code = __float_as_uint(rec[k].w);
        const float It = fminf((float)(code & kCodeMax) * (1.0f / (float)kCodeMax), 1.0f);
        const float f = It * (float)(len[k] - 1);
        const int kk = min((int)f, len[k] - 2);
        tau[k] = f - (float)kk;
        c0[k] = __ldg(&lut[off[k] + kk]);
        c1[k] = __ldg(&lut[off[k] + kk + 1]);
    }
#pragma unroll
    for (int k = 0; k < R; ++k)
        e[k] = make_float3((1.0f - tau[k]) * c0[k].x + tau[k] * c1[k].x, (1.0f - tau[k]) * c0[k].y + tau[k] * c1[k].y,
                           (1.0f - tau[k]) * c0[k].z + tau[k] * c1[k].z);
}

// Gaussian scale of a record: the weight is 2^(distance^2 x scale).  Kept finite and nonzero,
// so that the product is never NaN (R^2 may underflow to 0 or overflow; the comparison with R^2
// decides what is covered).
__device__ __forceinline__ float gauss_scale(float kexp, float R2) {
    return fminf(fmaxf(__fdividef(kexp, R2), -1e30f), -1.2e-38f);
}

}  // namespace spl
