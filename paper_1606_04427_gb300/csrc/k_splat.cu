// Per-tile Gaussian splat and final transform for the Splotch hot path.
//
// Section 3.1: each tile's particle list is rendered by one worker that owns the
// tile's pixels, so pixel updates never race with another tile.  Section 3.2.2: a
// draw adds particle colour x scalar weight to the pixel.  Section 2.1: the weight is
// a Gaussian of the distance to the particle centre over the radius-dependent area.
//
// GB300 layout: persistent warps pull work items from a queue.  A work item is a region of
// up to 16 x 16 pixels (a tile, or one of the split x split regions of a tile above 16 px)
// and a tile list, or a K-record slice of a crowded tile's list; slices of a split tile add
// their partial sums into an exact scratch tile and the last one to finish writes the
// result.  In frames of few records teams of 2, 4 or 8 warps of a CTA take the long items
// together (team_of): each warp renders a consecutive part of the list and the parts' sums are
// added in order, so a frame of 256 tiles occupies 2048 warps instead of 256.  The items come
// longest first; at the first short one a team parts and its warps go on alone.  How an item's sums
// are formed depends on the item and the frame alone, never on which team or warp meets it.  Teams
// never wait on one another.
//
// What a warp does with an item.  The kernel is bound by instruction issue and the latency
// between its phases (the records are read once, DRAM is nearly idle), so the layout is
// chosen for few instructions per covered pixel and per record:
//   1. fill: records are read 32 at a time from the list (kAhead copies ahead, through a ring
//      in shared memory); those whose support meets the region are appended to a batch;
//   2. decode, one record per lane: the 4 x 4-pixel squares (16 of them) its box meets, its
//      colour (colormap, or the particle's emission) and Gaussian scale.  Ballots give every
//      square a word of records per 32;
//   3. lists: per square, the batch positions of its records, unpacked from the words by two
//      lanes per square;
//   4. passes: a square is evaluated by a pair of lanes, 2 x 4 pixels each in packed FP32x2
//      arithmetic, so 16 records are in flight per warp instruction.  The squares are taken
//      longest list first, 16 at a time, or fewer with 2^a lane pairs each where the lists are
//      unequal (the pairs of a square then split its list and their sums are added by
//      shuffles).  Sums stay in registers for a pass and are added to the region's accumulator
//      in shared memory.
// Squares of a pass are distinct and passes are in order, so no pixel is ever updated by two
// lanes at once and the summation order depends only on the list's order.
//
// Why 4 x 4 squares and two lanes each: a particle of the two-species benchmark set covers 50
// pixels in 6.7 such squares (107 lane evaluations, against 142 in 8 x 4 blocks with a warp per
// record), a step of the pass loop serves 16 records instead of one, and the small records,
// most of a list, no longer cost a whole warp each.  The 10 M-particle frame at 2048^2 takes
// 500 M warp instructions (792 M with a warp per record), the 100 M-particle frame 5.5 ms
// (7.35), 10 M close particles at 4096^2 4.4 ms (5.1), 1 M at 637 x 483 67 us (196), 100 k at
// 256^2 21 us (107).  Batches of 192: 128 balance worse (6.2 ms), 224 leave 14 warps per SM
// instead of 16 (6.7 ms); scalar instead of packed arithmetic: 18 more instructions per step
// (6.5 ms against 6.1 before the loop was unrolled); unrolling by 3 drops the copies of the
// prefetched record (6.1 -> 5.75 ms).
#include "splat_batch.cuh"

namespace spl {

// Output of a pixel's accumulation a: mode 0 gives 1 - exp(-a) (final transform), 1 gives a,
// 2 adds a to what the pixel held (several renders summed in one image).
__device__ __forceinline__ float pixel(float held, float a, int mode) {
    return mode == 2 ? held + a : (mode ? a : -expm1f(-a));
}

constexpr int kWarps = 8;    // per CTA: the largest team
constexpr int kBatch = 192;  // records per batch
// Records up to which an item that one warp renders takes render_few; the part of a warp in an
// item that its team shares: half of that.  (Whether the warp's team is still together does not
// count: which team meets an item changes from run to run, the sums must not.)  Times the regions
// per tile edge, a region keeping a part of its tile's list: 1 M single-pixel particles at 8192^2
// (tiles of 64) take 0.47 ms, 0.56 with 64 for every tile and blank regions summed as others.
constexpr int kFew = 64;

// Warps per team, from the frame's `records` (times the regions per tile edge: a region reads its
// tile's whole list and keeps a part of it), items of at most K records and `warps` warps.  A warp alone has the least overhead per
// item, but a frame with fewer records than `warps` full items ends with its longest ones.
// Measured on 2432 warps, us with teams of 1 / 2 / 4 / 8 (kernel and k_item_order; 50 k to 8 M
// clustered particles at 256^2, 1024^2 and 2048^2):
//   records / (warps K)
//   0.01 - 0.02   99 / 64 / 44 / 35     109 / 78 / 52 / 47     107 / 72 / 52 / 50
//   0.08 - 0.14   134 / 83 / 54 / 42    135 / 89 / 70 / 60     154 / 97 / 76 / 81
//   0.25 - 0.47   140 / 88 / 91 / 91    166 / 107 / 99 / 116   191 / 150 / 142 / 154
//   0.8 - 1.4     224 / 154 / 140 / 164    271 / 199 / 205 / 248    342 / 300 / 314 / 369
//   2.0 - 3.8     283 / 283 / 302 / 380    428 / 459 / 478 / 590    654 / 707 / 750 / 908
__device__ __forceinline__ int team_of(int64_t records, int64_t K, int64_t warps) {
    const float r = __fdividef((float)records, (float)(warps * K));
    return r < 0.2f ? 8 : r < 0.5f ? 4 : r < 1.5f ? 2 : 1;
}

// Size bin from which a team shares an item: an eighth of K, 256 records (from a quarter, 50 k
// particles at 256^2 take 48 us instead of 35), for teams of 2 a quarter (from an eighth, 1 M uniform
// particles at 2048^2 take 167 us against 151).  Twice that where a region is a part of its tile and
// keeps a part of the list: 1 M single-pixel particles at 2501^2 (tiles of 24) take 122 us instead of
// 218, and tiles of 64 at 256^2 lose what sharing gives 50 k clustered ones if it is four times.
__device__ __forceinline__ int shared_from(int team, int split) {
    return (team > 2 ? kOrderBins / 8 : kOrderBins / 4) * min(split, 2);
}

// Barrier of one team's warps (`team` of them, a power of two).
__device__ __forceinline__ void team_sync(int team) {
    __syncwarp();
    if (team > 1)
        asm volatile("barrier.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x >> 5) / team), "r"(team * 32) : "memory");
}

// What the epilogue of an item needs, kept in shared memory over the item's passes: its view,
// its tile and region (pixels), the tile's scratch slot (-1: not split) and the items that
// add into it.
struct __align__(16) Place {
    int v, tx0, ty0, qx, qy, tw, th, slot, arrivals;
};

// What a warp knows of the frame and its team, in shared memory as well: image size, tiles per
// row and the size of the team.
struct __align__(16) Known {
    int W, H, ntx, team;
};

struct __align__(16) WarpSmem {
    Batch<kBatch> batch;             // pb: emission r, g, b
    float acc[3][kRegion][kRegion];  // the region's accumulator
};

// End of an item: the final transform of the region's pixels, or the merge of a split tile.
// kAlone: the item was a lone warp's; else its whole team takes part.
template <bool kAlone>
__device__ __forceinline__ void finish_item(const FrameDev &fr, float *out, int out_accum, WarpSmem *ws,
                                            const Place &at, const Known &kn, int *s_last, bool blank) {
    const int team = kAlone ? 1 : kn.team, unit = 32 * team, me = (int)threadIdx.x & (unit - 1);
    float *acc = &ws->acc[0][0][0];
    if (!kAlone) {  // the warps' sums, in warp order, into the first one's accumulator
        team_sync(team);
        WarpSmem *first = ws - (me >> 5);
        acc = &first->acc[0][0][0];
        for (int k = me; k < 3 * kRegion * kRegion; k += unit) {
            float sum = acc[k];
            for (int w = 1; w < team; ++w) sum += (&first[w].acc[0][0][0])[k];
            acc[k] = sum;
        }
        team_sync(team);
    }
    const float(*sums)[kRegion][kRegion] = reinterpret_cast<const float(*)[kRegion][kRegion]>(acc);
    const int W = kn.W, H = kn.H, px0 = at.tx0 + at.qx, py0 = at.ty0 + at.qy, tw = at.tw, th = at.th, slot = at.slot;
    const bool vec_rows = (W & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;  // 16-byte rows of 4 pixels
    float *o = out + (int64_t)at.v * H * W * 3;
    if (slot < 0) {
        float *reg = o + ((int64_t)py0 * W + px0) * 3;
        // rows of 48 floats, four at a time where they are aligned
        const bool wide = tw == kRegion && vec_rows && (px0 & 3) == 0;
        // What the pixels held comes through the batch's space, all of a lane's values in flight
        // together (read one by one, a warp's 24 trips to memory: 485 instead of 338 us for 400 k
        // clustered particles added to an image of 3958 x 4096).
        const int lane = threadIdx.x & 31;
        if (kAlone && blank) {  // a = 0
            if (out_accum == 2) return;
            if (wide) {
                for (int k = lane; k < th * 12; k += 32) {
                    const int r = k / 12;
                    *reinterpret_cast<float4 *>(reg + (int64_t)r * W * 3 + 4 * (k - 12 * r)) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
            } else {
#pragma unroll 1
                for (int j = 0; j < 3; ++j) {
                    const int odd = 32 * j + lane >= 3 * kRegion, c = 32 * j + lane - 3 * kRegion * odd;
                    float *to = reg + (int64_t)odd * W * 3 + c;
                    if (c / 3 < tw)
                        for (int p = 0; 2 * p + odd < th; ++p) to[(int64_t)p * 6 * W] = 0.0f;
                }
            }
            return;
        }
        float *held = reinterpret_cast<float *>(ws->batch.pa) + (wide ? 4 : 1) * lane;
        static_assert(sizeof(ws->batch.pa) >= 3 * kRegion * kRegion * sizeof(float), "a region's values");
        if (out_accum == 2) {
            if (wide) {
                for (int k = me, i = 0; k < th * 12; k += unit, i += 128)
                    copy16_async(held + i, reg + (int64_t)(k / 12) * W * 3 + 4 * (k % 12));
            } else {
#pragma unroll 1
                for (int j = 0; j < 3; ++j) {
                    const int odd = 32 * j + lane >= 3 * kRegion, c = 32 * j + lane - 3 * kRegion * odd;
                    if (c / 3 < tw)
                        for (int p = me >> 5; 2 * p + odd < th; p += team)
                            copy4_async(held + 32 * (kRegion / 2 * j + p), reg + (int64_t)(2 * p + odd) * W * 3 + c);
                }
            }
            copy_wait_all();
        }
        if (wide) {
            for (int k = me, i = 0; k < th * 12; k += unit, i += 128) {
                const int r = k / 12, c = 4 * (k - 12 * r);
                float4 u = *reinterpret_cast<float4 *>(held + i);
                u.x = pixel(u.x, sums[(c + 0) % 3][r][(c + 0) / 3], out_accum);
                u.y = pixel(u.y, sums[(c + 1) % 3][r][(c + 1) / 3], out_accum);
                u.z = pixel(u.z, sums[(c + 2) % 3][r][(c + 2) / 3], out_accum);
                u.w = pixel(u.w, sums[(c + 3) % 3][r][(c + 3) / 3], out_accum);
                *reinterpret_cast<float4 *>(reg + (int64_t)r * W * 3 + c) = u;
            }
        } else {
            // Rows that are not aligned: two rows of 48 values are three rounds of a warp, and a lane's
            // places in them are the same in every pair of rows (dividing for every value took 0.70
            // instead of 0.42 ms on 100 k particles at 8191^2).
#pragma unroll 1
            for (int j = 0; j < 3; ++j) {
                const int odd = 32 * j + lane >= 3 * kRegion, c = 32 * j + lane - 3 * kRegion * odd, col = c / 3;
                if (col >= tw) continue;
                const float *from = &sums[c - 3 * col][odd][col];
                float *to = reg + (int64_t)odd * W * 3 + c;
#pragma unroll 4
                for (int p = me >> 5; 2 * p + odd < th; p += team)
                    to[(int64_t)p * 6 * W] = pixel(held[32 * (kRegion / 2 * j + p)], from[2 * kRegion * p], out_accum);
            }
        }
    } else {
        const int T = fr.T;
        unsigned long long *scr = fr.scratch + (int64_t)slot * 6 * T * T;
        // 8 values per thread at a time, so that their atomics are in flight together
#pragma unroll 1
        for (int k0 = me; k0 < 3 * kRegion * kRegion; k0 += 8 * unit) {
            float val[8];
            unsigned long long *dst[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const int k = k0 + unit * g;
                const int ch = k / (kRegion * kRegion), r = (k / kRegion) % kRegion, col = k % kRegion;
                val[g] = k < 3 * kRegion * kRegion && r < th && col < tw ? acc[k] : 0.0f;
                dst[g] = &scr[2 * (ch * T * T + (at.qy + r) * T + at.qx + col)];
            }
            fix_add_n<8>(dst, val);
        }
        __threadfence();
        int last = 0;
        team_sync(team);
        if (!kAlone) {
            if (me == 0) s_last[threadIdx.x / unit] = (atomicAdd(&fr.tickets[slot], 1) == at.arrivals - 1);
            team_sync(team);
            last = s_last[threadIdx.x / unit];
        } else {
            if (me == 0) last = (atomicAdd(&fr.tickets[slot], 1) == at.arrivals - 1);
            last = __shfl_sync(0xffffffffu, last, 0);
        }
        if (last) {
            // the whole tile, from the scratch every region of every slice added into
            __threadfence();
            const int TW = min(T, W - at.tx0), TH = min(T, H - at.ty0);
            const int rl = 3 * TW;
            float *ot = o + ((int64_t)at.ty0 * W + at.tx0) * 3;
            for (int k0 = me; k0 < TH * rl; k0 += 4 * unit) {
                float a[4];
                int64_t pos[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const int k = min(k0 + unit * g, TH * rl - 1);
                    const int rr = k / rl, c3 = k - rr * rl;
                    const int col = c3 / 3, ch = c3 - col * 3;
                    a[g] = fix_value(&scr[2 * (ch * T * T + rr * T + col)]);
                    pos[g] = (int64_t)rr * W * 3 + c3;
                }
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    if (k0 + unit * g < TH * rl) ot[pos[g]] = pixel(ot[pos[g]], a[g], out_accum);
            }
            team_sync(team);
            for (int k = me; k < 6 * T * T; k += unit) scr[k] = 0ull;
            if (me == 0) fr.tickets[slot] = 0;
        }
    }
}

// Adds a record (pa: -X, -Y, R^2, Gaussian scale; pb: its emission) to 2 x 4 pixels with
// centres at columns fx0, fx1 and rows fy.
__device__ __forceinline__ void add_record(float4 pa, float4 pb, float2 fx0, float2 fx1, float2 fy,
                                           float2 (&s)[3][2][2]) {
    const float R2 = pa.z;
    const float2 dx0 = __fadd2_rn(fx0, f2(pa.x)), dx1 = __fadd2_rn(fx1, f2(pa.x));
    const float2 dy = __fadd2_rn(fy, f2(pa.y));
    const float2 qx0 = __fmul2_rn(dx0, dx0), qx1 = __fmul2_rn(dx1, dx1);
    const float2 qy = __fmul2_rn(dy, dy);
#pragma unroll
    for (int row = 0; row < 2; ++row) {
        const float2 qr = f2(row ? qy.y : qy.x);
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const float2 d2 = __fadd2_rn(cp ? qx1 : qx0, qr);
            const float2 g = __fmul2_rn(d2, f2(pa.w));
            const float2 w = make_float2(d2.x < R2 ? ex2_fast(g.x) : 0.0f, d2.y < R2 ? ex2_fast(g.y) : 0.0f);
            s[0][row][cp] = __ffma2_rn(f2(pb.x), w, s[0][row][cp]);
            s[1][row][cp] = __ffma2_rn(f2(pb.y), w, s[1][row][cp]);
            s[2][row][cp] = __ffma2_rn(f2(pb.z), w, s[2][row][cp]);
        }
    }
}

// Records of the batch whose emission is not finite (brightness, colour and view scale are, their
// product need not be) are added to the accumulator one by one, at the pixels they cover only:
// add_record adds emission x 0 where a record covers nothing, which would not be 0.  Their emission
// in the batch becomes 0.  Rare, so out of line and without regard to speed.
__device__ __noinline__ void add_wild(WarpSmem *ws, int nbuf, int px0, int py0) {
    const int lane = threadIdx.x & 31, x = lane & 15, y0 = 8 * (lane >> 4);
    const float fx = (float)(px0 + x) + 0.5f;
    for (int j = 0; j < nbuf; ++j) {
        const float4 pa = ws->batch.pa[j], pb = ws->batch.pb[j];
        if (isfinite(pb.x) && isfinite(pb.y) && isfinite(pb.z)) continue;
        const float dx = __fadd_rn(fx, pa.x);
        for (int y = y0; y < y0 + 8; ++y) {
            const float dy = __fadd_rn((float)(py0 + y) + 0.5f, pa.y);
            const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
            if (!(d2 < pa.z)) continue;
            const float w = ex2_fast(__fmul_rn(d2, pa.w));
            ws->acc[0][y][x] += pb.x * w;
            ws->acc[1][y][x] += pb.y * w;
            ws->acc[2][y][x] += pb.z * w;
        }
        __syncwarp();
        if (lane == 0) ws->batch.pb[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncwarp();
}

// Finite unless a component is not (or the sum leaves the range: add_wild looks again).
__device__ __forceinline__ float magnitude(float x, float y, float z) { return fabsf(x) + fabsf(y) + fabsf(z); }

// An item of few records, into the accumulator: 32 records at a time are decoded, one per lane,
// and evaluated one after another by the whole warp, 2 x 4 pixels per lane.  Batches, lists and
// sorted squares cost an item about 15 us of a warp's time whatever it holds, nearly all of it
// latency: 50 k particles at 4096^2 take 142 us instead of 213.  The limit: with 32 / 64 / 96
// records, 300 k clustered particles at 4096^2 take 253 / 232 / 232 us; 1 M at 256^2 (teams of 4)
// 76 / 85 / 85.
template <bool kViewScale, bool kEmit, bool kWild>
__device__ __forceinline__ bool render_few(const SceneDev &sc, const FrameDev &fr, WarpSmem *ws, const Region &rg,
                                           const float4 *recs, int nrec, int v, float kexp) {
    const int lane = threadIdx.x & 31, x = 4 * (lane & 3), y = 2 * (lane >> 2);
    Batch<kBatch> *bt = &ws->batch;
    const float fx = (float)(rg.px0 + x) + 0.5f, fy0 = (float)(rg.py0 + y) + 0.5f;
    const float2 fx0 = make_float2(fx, fx + 1.0f), fx1 = make_float2(fx + 2.0f, fx + 3.0f);
    const float2 fy = make_float2(fy0, fy0 + 1.0f);
    float2 s[3][2][2];  // channel, row, column pair
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[c][k >> 1][k & 1] = f2(0.0f);
    bool wild = false;  // add_wild has added to the accumulator
    bool drawn = false;
    float4 ahead = make_float4(0.0f, 0.0f, 0.0f, 0.0f);  // the next 32 records, on their way
    if (nrec > 0) ahead = __ldcg(&recs[min(lane, nrec - 1)]);
    for (int base = 0; base < nrec; base += 32) {
        const float4 rec[1] = {ahead};
        if (base + 32 < nrec) ahead = __ldcg(&recs[min(base + 32 + lane, nrec - 1)]);
        const bool live = base + lane < nrec && fmaxf(fabsf(rec[0].x - rg.xc), fabsf(rec[0].y - rg.yc)) <
                                                    fmaf(rec[0].z, 1.000004f, rg.half);
        const uint32_t bal = __ballot_sync(0xffffffffu, live);
        if (bal == 0) continue;
        drawn = true;
        float3 e[1];
        float vs = 1.0f;
        if constexpr (kEmit) {  // the record's last word is the particle index
            const float4 em = __ldg(&sc.emit[__float_as_uint(rec[0].w)]);
            e[0] = make_float3(em.x, em.y, em.z);
            if constexpr (kViewScale) vs = __ldg(&fr.vscale[v * sc.n_types + __float_as_int(em.w)]);
        } else {
            batch_colours<1>(rec, kViewScale ? fr.vlut : sc.lut, kViewScale ? fr.vlut_len + v * sc.n_types : sc.lut_len,
                             kViewScale ? fr.vlut_off + v * sc.n_types : sc.lut_off, e);
            if constexpr (kViewScale) vs = __ldg(&fr.vscale[v * sc.n_types + (__float_as_uint(rec[0].w) >> 24)]);
        }
        if (live) {
            const int j = __popc(bal & ((1u << lane) - 1u));
            const float R2 = __fmul_rn(rec[0].z, rec[0].z);
            bt->pa[j] = make_float4(-rec[0].x, -rec[0].y, R2, gauss_scale(kexp, R2));
            bt->pb[j] = make_float4(e[0].x * vs, e[0].y * vs, e[0].z * vs, 0.0f);
        }
        __syncwarp();
        const int n = __popc(bal);
        if (kWild && __any_sync(0xffffffffu, live && !isfinite(magnitude(e[0].x * vs, e[0].y * vs, e[0].z * vs)))) {
            if (!wild)
                for (int k = lane; k < 3 * kRegion * kRegion; k += 32) (&ws->acc[0][0][0])[k] = 0.0f;
            wild = true;
            __syncwarp();
            add_wild(ws, n, rg.px0, rg.py0);
        }
#pragma unroll 2
        for (int j = 0; j < n; ++j) {
            const float4 pa = bt->pa[j], pb = bt->pb[j];
            add_record(pa, pb, fx0, fx1, fy, s);
        }
        __syncwarp();
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int row = 0; row < 2; ++row) {
            float4 *p = reinterpret_cast<float4 *>(&ws->acc[c][y + row][x]);
            float4 u = make_float4(s[c][row][0].x, s[c][row][0].y, s[c][row][1].x, s[c][row][1].y);
            if (kWild && wild) u.x += p->x, u.y += p->y, u.z += p->z, u.w += p->w;
            *p = u;
        }
    return drawn;
}

// kViewScale: multiply every record's emission by a per-view, per-species scale (plans
// with a brightness sequence); a separate instance, so plain renders carry no extra code.
// kWild: an emission may not be finite (add_wild): scenes that say so, and all plans, whose scales
// change between replays.  The branch cost plain frames 0.4 to 0.8 % when they had it as well.
template <bool kViewScale, bool kEmit, bool kWild>
__global__ void __launch_bounds__(kWarps * 32, 2)
    k_splat(SceneDev sc, FrameDev fr, int *queue, float *out, int out_accum, int split) {
    if (fr.status[kStatOverflow]) return;  // no complete tile lists
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ int s_item[kWarps], s_last[kWarps];  // per team
    __shared__ Known s_known[kWarps];
    __shared__ Place s_place[kWarps];
    WarpSmem *ws = reinterpret_cast<WarpSmem *>(s_raw) + (threadIdx.x >> 5);
    const int total_items = (int)fr.sizes[kSizeItems] * split * split;
    Batch<kBatch> *bt = &ws->batch;
    constexpr int kRounds = Batch<kBatch>::kRounds;
    const int lane = threadIdx.x & 31;
    const int nt = fr.n_tiles;
    const int S2 = split * split;
    const int64_t K = fr.sizes[kSizeK];
    const int pair = lane >> 1;  // lane pair: the unit that evaluates a square
    if (lane == 0) {
        bt->pa[kBatch] = make_float4(0.0f, 0.0f, -1.0f, -1.0f);
        bt->pb[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }

    // What a warp knows of the frame, its team and its item is read from shared memory before
    // and after the item's passes: they leave no registers for it.
    if (lane == 0)
        s_known[threadIdx.x >> 5] = {fr.views[0].W, fr.views[0].H, fr.views[0].ntx,
                                     team_of(fr.sizes[kSizePairs] * split, K, (int)gridDim.x * kWarps)};
    __syncwarp();

    // the next item is taken from the queue while the current one is rendered
    int next = 0;
    if ((threadIdx.x & (32 * s_known[threadIdx.x >> 5].team - 1)) == 0) next = atomicAdd(queue, 1);
    for (;;) {
        const Known kn = s_known[threadIdx.x >> 5];
        const int me = (int)threadIdx.x & (32 * kn.team - 1);  // of the team's threads
        int item;
        if (kn.team > 1) {
            int *box = &s_item[threadIdx.x / (32 * kn.team)];
            if (me == 0) *box = next;
            team_sync(kn.team);
            item = *box;
        } else {
            item = __shfl_sync(0xffffffffu, next, 0);
        }
        if (item >= total_items) break;
        if (me == 0) next = atomicAdd(queue, 1);

        // item = (slice of a tile list, region of the tile); the regions of a slice are
        // consecutive items, so they run at once and share the slice's records in L2
        const int qs = item / S2, q = item - qs * S2;
        const int2 ord = __ldg(&fr.order[qs]);
        const int gt = ord.x, chunk = ord.y;  // the slice's tile and its place in the tile's list
        const int v = gt / nt, t = gt - v * nt;
        const float kexp = fr.views[v].kexp;
        Region rg;
        int nrec;
        {
            const int T = fr.T, sub = (T + split - 1) / split;  // edge of the region a team owns
            Place p;
            p.v = v;
            p.tx0 = t % kn.ntx * T, p.ty0 = t / kn.ntx * T;
            p.qx = (q % split) * sub, p.qy = (q / split) * sub;
            p.tw = max(0, min(min(sub, T - p.qx), kn.W - p.tx0 - p.qx));
            p.th = max(0, min(min(sub, T - p.qy), kn.H - p.ty0 - p.qy));
            p.slot = fr.split_slot[gt];
            p.arrivals = (fr.item_off[gt + 1] - fr.item_off[gt]) * S2;
            if (lane == 0) s_place[threadIdx.x >> 5] = p;
            rg = make_region(p.tx0 + p.qx, p.ty0 + p.qy, p.tw, p.th);
            nrec = p.tw > 0 && p.th > 0;
        }
        const int64_t seg1 = fr.offsets[gt + 1];
        const int64_t e0 = fr.offsets[gt] + (int64_t)chunk * K;
        const int len = (int)(min(seg1, e0 + K) - e0);
        if (nrec) nrec = len;
        if (nrec == 0 && out_accum == 2 && kn.team == 1 && fr.split_slot[gt] < 0) continue;  // adds nothing
        const float4 *recs = fr.lists + e0;
        int few = kFew * split;
        bool blank = false;  // no record meets the region
        if (kn.team > 1) {
            // by the slice's length: that of the order, also where the region has no pixel
            if (order_bin(len, (int)K) >= shared_from(kn.team, split)) {
                // this warp's consecutive part of the slice
                const int part = ((nrec + kn.team - 1) / kn.team + 31) & ~31;
                const int first = min(nrec, (me >> 5) * part);
                recs += first;
                nrec = min(part, nrec - first);
                few = kFew / 2 * split;
            } else {  // the first warp's alone, and so are all later items: the team parts
                if (lane == 0) s_known[threadIdx.x >> 5].team = 1;
                __syncwarp();
                if (me >= 32) {
                    if (lane == 0) next = atomicAdd(queue, 1);
                    continue;
                }
            }
        }

        if (nrec <= few) {
            blank = !render_few<kViewScale, kEmit, kWild>(sc, fr, ws, rg, recs, nrec, v, kexp);
            nrec = 0;
        } else {
            float *acc = &ws->acc[0][0][0];
#pragma unroll
            for (int k = 0; k < 3 * kRegion * kRegion / 128; ++k)
                reinterpret_cast<float4 *>(acc)[k * 32 + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            batch_start(bt, recs, nrec);
        }
        int base = 0, row = 0;
        while (base < nrec) {
            // ---- 1. fill the batch with records that meet the region
            const int nbuf = batch_fill<kEmit>(bt, rg, recs, nrec, base, row, sc.emit);
            if (nbuf == 0) continue;

            // ---- 2. squares, colour and Gaussian scale, one record per lane; lanes past the end
            // repeat the last record
            uint32_t word[Batch<kBatch>::kWords];
            int cnt;
            float most = 0.0f;  // finite if the lane's emissions are
            {
                float4 rec[kRounds];
#pragma unroll
                for (int g = 0; g < kRounds; ++g) rec[g] = bt->pa[min(g * 32 + lane, nbuf - 1)];
                cnt = batch_words<false, kBatch>(rec, nbuf, rg, word);
                float3 e[kRounds];
                float vs[kRounds];
                if constexpr (kEmit) {
                    copy_wait_all();
                    __syncwarp();
                    if constexpr (kViewScale)
#pragma unroll
                        for (int g = 0; g < kRounds; ++g) {
                            const float4 em = bt->pb[min(g * 32 + lane, nbuf - 1)];
                            e[g] = make_float3(em.x, em.y, em.z);
                            vs[g] = __ldg(&fr.vscale[v * sc.n_types + __float_as_int(em.w)]);
                        }
                } else {
                    // the view's colormap in a plan with per-view sequences, else the scene's
                    const float4 *lut = kViewScale ? fr.vlut : sc.lut;
                    const int *lut_len = kViewScale ? fr.vlut_len + v * sc.n_types : sc.lut_len;
                    const int *lut_off = kViewScale ? fr.vlut_off + v * sc.n_types : sc.lut_off;
                    batch_colours<kRounds>(rec, lut, lut_len, lut_off, e);
#pragma unroll
                    for (int g = 0; g < kRounds; ++g)
                        vs[g] = kViewScale ? __ldg(&fr.vscale[v * sc.n_types + (__float_as_uint(rec[g].w) >> 24)]) : 1.0f;
                }
                __syncwarp();
#pragma unroll
                for (int g = 0; g < kRounds; ++g) {
                    const int j = g * 32 + lane;
                    if (j >= nbuf) break;
                    const float R2 = __fmul_rn(rec[g].z, rec[g].z);
                    bt->pa[j] = make_float4(-rec[g].x, -rec[g].y, R2, gauss_scale(kexp, R2));
                    if constexpr (kViewScale || !kEmit)
                        bt->pb[j] = make_float4(e[g].x * vs[g], e[g].y * vs[g], e[g].z * vs[g], 0.0f);
                    if constexpr (kWild && kViewScale)
                        most += magnitude(e[g].x * vs[g], e[g].y * vs[g], e[g].z * vs[g]);
                }
            }
            if (kWild && (!kViewScale || __any_sync(0xffffffffu, !isfinite(most)))) {
                __syncwarp();
                add_wild(ws, nbuf, rg.px0, rg.py0);
            }

            // ---- 3. per square, the batch positions of its records; squares longest list first
            int before, total;
            const uint32_t key = sort_squares(batch_lists<false>(bt, word, cnt), before, total);

            // ---- 4. passes over the squares
            for (int i = 0; i < 16;) {
                const int lead = (int)(__shfl_sync(0xffffffffu, key, i) >> 4);
                if (lead == 0) break;
                const int a = choose_split<64, 36, 60>(i, lead, before, total);
                const int place = i + (pair >> a), r = pair & ((1 << a) - 1);
                const uint32_t kp = __shfl_sync(0xffffffffu, key, place & 15);
                const int sq = (int)(kp & 15u);
                const int n = place < 16 ? (int)(kp >> 4) : 0;
                const int mine = (n - r + (1 << a) - 1) >> a;  // list entries r, r + 2^a, ...
                const int steps = (lead + (1 << a) - 1) >> a;
                const unsigned char *lp = bt->list[sq] + r;
                // this lane's pixels: rows y, y + 1 and columns x .. x + 3 of the region
                const int x = 4 * (sq & 3), y = 4 * (sq >> 2) + 2 * (lane & 1);
                const float fx = (float)(rg.px0 + x) + 0.5f, fy0 = (float)(rg.py0 + y) + 0.5f;
                const float2 fx0 = make_float2(fx, fx + 1.0f), fx1 = make_float2(fx + 2.0f, fx + 3.0f);
                const float2 fy = make_float2(fy0, fy0 + 1.0f);
                float2 s[3][2][2];  // channel, row, column pair
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int k = 0; k < 4; ++k) s[c][k >> 1][k & 1] = f2(0.0f);
                // the records of the next step load while this one is evaluated; a pair past
                // the end of its list takes the record that covers nothing
                int idx = mine > 0 ? *lp : kBatch;
                float4 na = bt->pa[idx], nb = bt->pb[idx];
                lp += 1 << a;
                idx = mine > 1 ? *lp : kBatch;
#pragma unroll 3
                for (int k = 2; k < steps + 2; ++k) {
                    const float4 pa = na, pb = nb;
                    na = bt->pa[idx];
                    nb = bt->pb[idx];
                    lp += 1 << a;
                    idx = k < mine ? *lp : kBatch;
                    add_record(pa, pb, fx0, fx1, fy, s);
                }
                for (int d = 2; d < (2 << a); d <<= 1) {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float2 &u = s[c][k >> 1][k & 1];
                            u = __fadd2_rn(u, make_float2(__shfl_xor_sync(0xffffffffu, u.x, d),
                                                          __shfl_xor_sync(0xffffffffu, u.y, d)));
                        }
                }
                if (r == 0 && n > 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int row = 0; row < 2; ++row) {
                            float4 *p = reinterpret_cast<float4 *>(&ws->acc[c][y + row][x]);
                            float4 u = *p;
                            u.x += s[c][row][0].x, u.y += s[c][row][0].y;
                            u.z += s[c][row][1].x, u.w += s[c][row][1].y;
                            *p = u;
                        }
                }
                __syncwarp();
                i += 16 >> a;
            }
        }
        __syncwarp();
        const Known end = s_known[threadIdx.x >> 5];
        const Place at = s_place[threadIdx.x >> 5];
        if (end.team == 1)
            finish_item<true>(fr, out, out_accum, ws, at, end, s_last, blank);
        else
            finish_item<false>(fr, out, out_accum, ws, at, end, s_last, false);
        __syncwarp();
    }
}

typedef void (*SplatFn)(SceneDev, FrameDev, int *, float *, int, int);

// Regions per tile edge.  Each reads its tile's whole list and keeps a part of it.  At tiles of 32 /
// 40 / 48 / 64 pixels (10 M particles at 2048^2) the splat takes 0.85 / 1.03 / 1.02 / 1.30 ms, where a
// CTA per tile above 32 pixels that read the list once took 3.80 / 4.52 / 4.91; 20 M at 8192^2 (64
// pixels) 8.75 against 32.3 ms, 200 k at 5000^2 (40 pixels) 0.27 against 0.43.
int splat_split(int T) { return (T + kRegion - 1) / kRegion; }

static SplatFn splat_fn(bool scaled, bool emit, bool wild) {
    if (scaled) return emit ? k_splat<true, true, true> : k_splat<true, false, true>;
    if (wild) return emit ? k_splat<false, true, true> : k_splat<false, false, true>;
    return emit ? k_splat<false, true, false> : k_splat<false, false, false>;
}

static size_t splat_smem() { return sizeof(WarpSmem) * kWarps; }

int splat_blocks_per_sm() {
    const void *fn = (const void *)splat_fn(false, false, false);
    if (ensure_smem_limit(fn, splat_smem()) != cudaSuccess) return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kWarps * 32, splat_smem()) != cudaSuccess) return 0;
    return nb;
}

int splat_workers_per_sm() { return splat_blocks_per_sm() * kWarps; }

// k_item_order: the splat's work items (tile-list slices) ordered by record count, largest
// first, so that the items taken last by the workers are the short ones and the kernel does
// not end waiting for a few long slices started late.  Slices fall into kOrderBins bins of
// equal width up to K (the slice length of a split tile), whose sizes k_scan has counted;
// within a bin the order is that of the atomic cursors.  Each item writes its own tile, or adds
// into the exact accumulators of a split tile, and its sums do not depend on who renders it, so
// images do not depend on the order.  One tile
// per thread: 8 us for 16384 tiles and 5 us for 65536 that are hardly split (33 and 84 us with
// one CTA for all).
__global__ void __launch_bounds__(1024) k_item_order(FrameDev fr) {
    __shared__ int s_cnt[kOrderBins], s_all[kOrderBins], s_pos[kOrderBins];
    if (fr.status[kStatOverflow]) return;
    const int N = fr.V * fr.n_tiles, lane = threadIdx.x & 31;
    const int K = (int)fr.sizes[kSizeK];
    if (threadIdx.x < kOrderBins) s_cnt[threadIdx.x] = 0, s_all[threadIdx.x] = fr.bins[threadIdx.x];
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    // every slice of a split tile holds K records but the last; tiles of a warp whose last slices
    // share a bin are counted and placed together
    int n = 0, last_bin = kOrderBins;
    if (t < N) {
        n = fr.item_off[t + 1] - fr.item_off[t];
        last_bin = order_bin(fr.counts[t] - K * (n - 1), K);
    }
    const uint32_t peers = warp_peers<7>((uint32_t)last_bin);
    const int leader = __ffs(peers) - 1;
    if (t < N && lane == leader) atomicAdd(&s_cnt[last_bin], __popc(peers));
    if (n > 1) atomicAdd(&s_cnt[order_bin(K, K)], n - 1);
    __syncthreads();
    // this CTA's place in each bin: the bins before it (the largest first), then the CTAs that
    // came earlier
    if (threadIdx.x < kOrderBins) {
        int start = 0;
        for (int b = kOrderBins - 1; b > (int)threadIdx.x; --b) start += s_all[b];
        const int c = s_cnt[threadIdx.x];
        s_pos[threadIdx.x] = start + (c ? atomicAdd(&fr.bins[kOrderBins + threadIdx.x], c) : 0);
    }
    __syncthreads();
    int at = 0;
    if (t < N && lane == leader) at = atomicAdd(&s_pos[last_bin], __popc(peers));
    at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
    if (t < N) fr.order[at] = make_int2(t, n - 1);
    // the full slices of a split tile, by its warp
    for (uint32_t todo = __ballot_sync(0xffffffffu, n > 1); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const int m = __shfl_sync(0xffffffffu, n, src) - 1, tt = __shfl_sync(0xffffffffu, t, src);
        int p = 0;
        if (lane == 0) p = atomicAdd(&s_pos[order_bin(K, K)], m);
        p = __shfl_sync(0xffffffffu, p, 0);
        for (int k = lane; k < m; k += 32) fr.order[p + k] = make_int2(tt, k);
    }
}

cudaError_t launch_item_order(const FrameDev &fr, cudaStream_t st) {
    const int64_t N = (int64_t)fr.V * fr.n_tiles;
    k_item_order<<<(int)((N + 1023) / 1024), 1024, 0, st>>>(fr);
    return cudaGetLastError();
}

cudaError_t launch_splat(const SceneDev &sc, const FrameDev &fr, float *out, int out_accum, int grid,
                         cudaStream_t st) {
    cudaError_t e = launch_item_order(fr, st);
    if (e != cudaSuccess) return e;
    const SplatFn fn = splat_fn(fr.vscale != nullptr, sc.emit != nullptr, sc.wild != 0);
    e = ensure_smem_limit((const void *)fn, splat_smem());
    if (e != cudaSuccess) return e;
    fn<<<grid, kWarps * 32, splat_smem(), st>>>(sc, fr, fr.queue, out, out_accum, splat_split(fr.T));
    return cudaGetLastError();
}

__global__ void k_final(float *a, int64_t count) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = -expm1f(-a[i]);
}

cudaError_t launch_final(float *a, int64_t count, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 8192) blocks = 8192;
    k_final<<<(int)blocks, 256, 0, st>>>(a, count);
    return cudaGetLastError();
}

// A CTA waits on an mbarrier that expects one arrival nobody makes: the bounded wait must
// give up and report, leaving the context usable.
__global__ void k_selftest_wait(long long limit, int *result) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    const bool ok = mbar_wait_bounded(&bar, 0, limit);
    if (threadIdx.x == 0) *result = ok ? 1 : 2;
}

cudaError_t launch_selftest_wait(long long limit, int *result, cudaStream_t st) {
    k_selftest_wait<<<1, 32, 0, st>>>(limit, result);
    return cudaGetLastError();
}

}  // namespace spl
