// Depth-ordered splat: radiative transfer with absorption different from emission.
//
// Section 2.1 renders by solving the radiative-transfer equation along each line of
// sight.  With absorption A equal to emission E every particle's update commutes and the
// image is 1 - exp(-a) of a plain sum; with A = s_t E for species t (s_t >= 0) it does
// not, and the particles must be applied in depth order, farthest first, from a black
// background:
//     I <- a I + b,   a = exp(-A w),   b = (E / A)(1 - a) = (1 - a) / s_t   (I + E w if s_t = 0)
// per pixel and channel, w the particle's Gaussian weight there.  The tile lists reach
// this kernel far to near, particles of exactly equal depth in index order: the particles
// are sorted by depth (stably, from index order), their records are written out in that
// order, and a stable sort by tile id groups them (depth-ordered binning).
//
// Layout as the additive splat (splat_batch.cuh): a warp takes a region of up to 16 x 16 pixels
// and batches of its records, lists them per 4 x 4-pixel square in list order, and evaluates a
// square by a pair of lanes, 2 x 4 pixels each.  Each lane keeps, per pixel and channel, the
// affine map of the records applied so far, I_out = alpha I_in + beta.  Where a square gets
// several lane pairs, each takes a consecutive part of the list and the maps are composed by
// shuffles; the map of a pass is composed onto the region's map in shared memory.  A tile that
// is not split writes beta; the slices of a split tile store their maps, which k_compose_slices
// composes far to near.
//
// What bounds it: the FP32 pipe (67 % of its cycles on the 10 M-particle two-species frame; a packed
// operation holds it two).  Hence the short polynomials (9, 10 or 12 packed operations per channel
// and two pixels, 15 with the exponential) and squares of 4 x 4 pixels: 6.7 squares, 107 pixel
// evaluations per particle, against 235 in the 8 x 8 units of a warp per record.  10 M particles at
// 2048^2: 3.33 ms with a warp per record, 1.66 and 0.05 for the composition now (1.52 with the
// cheaper and less accurate update named below); a frame of 1 M particles as maps at 1000 x 757:
// 1.24 -> 0.55 ms (0.55).  Batches of 192 (12 warps per SM): 128 on 16 warps took 2.47 ms where 192
// took 2.21.
#include "splat_batch.cuh"

namespace spl {

constexpr int kOWarps = 2;    // warps per CTA
constexpr int kOBatch = 192;  // records per batch

struct __align__(16) OWarpSmem {
    Batch<kOBatch> batch;            // pb: emission E per channel, and s
    float map[6][kRegion][kRegion];  // the region's map: alpha r, g, b, beta r, g, b
};

// Update of one record with e = E w, x = s e and phi(x) = (1 - exp(-x)) / x per pixel and channel:
//     alpha <- alpha - x phi alpha,   beta <- beta + phi (e - x beta),
// which needs no 1 / s: a species with s = 0 has x = 0, phi = 1, and a pixel of few records has as
// few roundings as e phi itself.  (With u = x phi and beta <- beta + u (1 / s - beta), an operation
// less and polynomials a degree shorter, the errors of u, 1 / s and phi reached beta: 1.0e-7 instead
// of 4e-8 RMS on pixels of one to three records, with a bias of 5e-8 to 9e-8; and 1 / s overflowed
// where s = 0 stood for 2^-40 / E.  Emulated against 64 bits for 1 to 200 records, x from 0.001 to 2,
// the present form is nowhere less accurate than a beta + b with a and b rounded apart.)
// phi is a polynomial whose degree follows the step's largest x (w <= 1, so a record's x is at most
// its s E): degree 3 up to kDeg3Max, 4 up to kDeg4Max and 6 up to kDeg6Max, minimax with phi(0) = 1
// (fitted here by iteratively reweighted least squares against expm1 in 64 bits; largest relative
// errors 8.0e-9, 3.0e-9 and 9.3e-9).  Beyond, and for negative emissions, the Taylor polynomial of
// degree 5 where |x| <= kDeg4Max (next term x^6 / 7! <= 5e-8) and the exponential itself elsewhere:
// alpha <- a alpha, beta <- a beta + (1 - a) / s, a = exp(-x).  (A degree 2 up to 0.015 as well: 10 M
// particles at 2048^2 in 3.15 instead of 3.11 ms, a step's 16 records are rarely all below.)
constexpr float kDeg3Max = 0.1f, kDeg4Max = 0.25f, kDeg6Max = 1.0f;

// phi as a polynomial in -x (all coefficients positive)
template <int kDeg> __device__ __forceinline__ float2 phi_of(float2 nx) {  // degree 3, 4, 6 or 5 (Taylor)
    float2 phi;
    if (kDeg == 5) {
        phi = __ffma2_rn(nx, f2(1.0f / 720.0f), f2(1.0f / 120.0f));
        phi = __ffma2_rn(nx, phi, f2(1.0f / 24.0f));
        phi = __ffma2_rn(nx, phi, f2(1.0f / 6.0f));
        phi = __ffma2_rn(nx, phi, f2(0.5f));
    } else if (kDeg == 6) {
        phi = __ffma2_rn(nx, f2(0.000129130945f), f2(0.00130112655f));
        phi = __ffma2_rn(nx, phi, f2(0.00827620924f));
        phi = __ffma2_rn(nx, phi, f2(0.0416474678f));
        phi = __ffma2_rn(nx, phi, f2(0.166663662f));
        phi = __ffma2_rn(nx, phi, f2(0.499999851f));
    } else if (kDeg == 4) {
        phi = __ffma2_rn(nx, f2(0.00753017422f), f2(0.0415001325f));
        phi = __ffma2_rn(nx, phi, f2(0.166652888f));
        phi = __ffma2_rn(nx, phi, f2(0.499999642f));
    } else {
        phi = __ffma2_rn(nx, f2(0.0400981233f), f2(0.166576117f));
        phi = __ffma2_rn(nx, phi, f2(0.49999851f));
    }
    return __ffma2_rn(nx, phi, f2(1.0f));
}

// One step of a pass: every lane applies its record (pb: E r, g, b and s) to its 2 x 4 pixels.
// kDeg 5: the exponential where x is beyond kDeg4Max.
template <int kDeg>
__device__ __forceinline__ void apply_record(const float4 &pa, const float4 &pb, const float2 (&fx)[2], const float2 &fy,
                                             float2 (&al)[3][2][2], float2 (&be)[3][2][2]) {
    const float E[3] = {pb.x, pb.y, pb.z};
    const float inv_s = kDeg == 5 ? 1.0f / pb.w : 0.0f;
    const float2 dx[2] = {__fadd2_rn(fx[0], f2(pa.x)), __fadd2_rn(fx[1], f2(pa.x))};
    const float2 dy = __fadd2_rn(fy, f2(pa.y));
    const float2 qx[2] = {__fmul2_rn(dx[0], dx[0]), __fmul2_rn(dx[1], dx[1])};
    const float2 qy = __fmul2_rn(dy, dy);
#pragma unroll
    for (int row = 0; row < 2; ++row) {
        const float2 qr = f2(row ? qy.y : qy.x);
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const float2 d2 = __fadd2_rn(qx[cp], qr);
            const float2 g = __fmul2_rn(d2, f2(pa.w));
            // uncovered: e = x = 0
            const float2 w = make_float2(d2.x < pa.z ? ex2_fast(g.x) : 0.0f, d2.y < pa.z ? ex2_fast(g.y) : 0.0f);
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                float2 &A = al[ch][row][cp], &B = be[ch][row][cp];
                const float2 e = __fmul2_rn(f2(E[ch]), w), nx = __fmul2_rn(f2(-pb.w), e), phi = phi_of<kDeg>(nx);
                float2 an = __ffma2_rn(__fmul2_rn(nx, phi), A, A);
                float2 bn = __ffma2_rn(phi, __ffma2_rn(nx, B, e), B);
                if (kDeg == 5) {
                    const float2 y = __fmul2_rn(nx, f2(kLog2e));
                    const float2 a = make_float2(ex2_fast(y.x), ex2_fast(y.y));
                    const float2 fa = __fmul2_rn(a, A);
                    const float2 fb = __ffma2_rn(a, B, __ffma2_rn(a, f2(-inv_s), f2(inv_s)));
                    if (fabsf(nx.x) > kDeg4Max) an.x = fa.x, bn.x = fb.x;
                    if (fabsf(nx.y) > kDeg4Max) an.y = fa.y, bn.y = fb.y;
                }
                A = an, B = bn;
            }
        }
    }
}

template <bool kEmit>
__global__ void __launch_bounds__(kOWarps * 32, 6)
    k_splat_ordered(SceneDev sc, FrameDev fr, int *queue, float *out, int split,
                    const float *__restrict__ absorb, float *ord_scratch, int map_out) {
    if (fr.status[kStatOverflow]) return;
    extern __shared__ __align__(16) unsigned char s_raw[];
    OWarpSmem *ws = reinterpret_cast<OWarpSmem *>(s_raw) + (threadIdx.x >> 5);
    Batch<kOBatch> *bt = &ws->batch;
    constexpr int kRounds = Batch<kOBatch>::kRounds;
    const int lane = threadIdx.x & 31;
    const int pair = lane >> 1;
    const int nt = fr.n_tiles;
    const int S2 = split * split;
    const int total_items = (int)fr.sizes[kSizeItems] * S2;
    const int64_t K = fr.sizes[kSizeK];
    const ViewParams g0 = fr.views[0];
    const int T = g0.T, W = g0.W, H = g0.H, ntx = g0.ntx;
    const int sub = (T + split - 1) / split;
    if (lane == 0) {  // covers nothing
        bt->pa[kOBatch] = make_float4(0.0f, 0.0f, -1.0f, -1.0f);
        bt->pb[kOBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }

    int next = 0;
    if (lane == 0) next = atomicAdd(queue, 1);
    for (;;) {
        const int item = __shfl_sync(0xffffffffu, next, 0);
        if (item >= total_items) break;
        if (lane == 0) next = atomicAdd(queue, 1);

        const int qs = item / S2, q = item - qs * S2;
        const int2 ord = __ldg(&fr.order[qs]);  // largest slices first
        const int gt = ord.x, chunk = ord.y, slice = fr.item_off[gt] + chunk;
        const int v = gt / nt, t = gt - v * nt;
        const int slot = fr.split_slot[gt];
        const float kexp = fr.views[v].kexp;
        const int tx = t % ntx, ty = t / ntx;
        const int qx = (q % split) * sub, qy = (q / split) * sub;
        const int px0 = tx * T + qx, py0 = ty * T + qy;
        const int tw = max(0, min(min(sub, T - qx), W - px0));
        const int th = max(0, min(min(sub, T - qy), H - py0));
        const int64_t seg1 = fr.offsets[gt + 1];
        const int64_t e0 = fr.offsets[gt] + (int64_t)chunk * K;
        const int nrec = (tw > 0 && th > 0) ? (int)(min(seg1, e0 + K) - e0) : 0;
        const float4 *recs = fr.lists + e0;

        float *map = &ws->map[0][0][0];
#pragma unroll
        for (int k = 0; k < 6 * kRegion * kRegion / 128; ++k) {
            const float id = k < 3 * kRegion * kRegion / 128 ? 1.0f : 0.0f;
            reinterpret_cast<float4 *>(map)[k * 32 + lane] = make_float4(id, id, id, id);
        }

        const Region rg = make_region(px0, py0, tw, th);
        batch_start(bt, recs, nrec);
        int base = 0, row = 0;
        while (base < nrec) {
            const int nbuf = batch_fill<kEmit>(bt, rg, recs, nrec, base, row, sc.emit);
            if (nbuf == 0) continue;

            // ---- decode, one record per lane
            uint32_t word[Batch<kOBatch>::kWords];
            int cnt;
            {
                float4 rec[kRounds];
#pragma unroll
                for (int g = 0; g < kRounds; ++g) rec[g] = bt->pa[min(g * 32 + lane, nbuf - 1)];
                cnt = batch_words<true, kOBatch>(rec, nbuf, rg, word);
                float3 e[kRounds];
                float s[kRounds];
                if constexpr (kEmit) {
                    copy_wait_all();
                    __syncwarp();
#pragma unroll
                    for (int g = 0; g < kRounds; ++g) {
                        const float4 em = bt->pb[min(g * 32 + lane, nbuf - 1)];
                        e[g] = make_float3(em.x, em.y, em.z);
                        s[g] = __ldg(&absorb[__float_as_int(em.w)]);
                    }
                } else {
                    batch_colours<kRounds>(rec, sc.lut, sc.lut_len, sc.lut_off, e);
#pragma unroll
                    for (int g = 0; g < kRounds; ++g) s[g] = __ldg(&absorb[__float_as_uint(rec[g].w) >> 24]);
                }
                __syncwarp();
#pragma unroll
                for (int g = 0; g < kRounds; ++g) {
                    const int j = g * 32 + lane;
                    if (j >= nbuf) break;
                    const float R2 = __fmul_rn(rec[g].z, rec[g].z);
                    bt->pa[j] = make_float4(-rec[g].x, -rec[g].y, R2, gauss_scale(kexp, R2));
                    bt->pb[j] = make_float4(e[g].x, e[g].y, e[g].z, s[g]);
                }
            }
            int before, total;
            const uint32_t key = sort_squares(batch_lists<true>(bt, word, cnt), before, total);

            // ---- passes over the squares
            for (int i = 0; i < 16;) {
                const int lead = (int)(__shfl_sync(0xffffffffu, key, i) >> 4);
                if (lead == 0) break;
                const int a = choose_split<160, 220, 150>(i, lead, before, total);
                const int place = i + (pair >> a), r = pair & ((1 << a) - 1);
                const uint32_t kp = __shfl_sync(0xffffffffu, key, place & 15);
                const int sq = (int)(kp & 15u);
                const int n = place < 16 ? (int)(kp >> 4) : 0;
                const int steps = (lead + (1 << a) - 1) >> a;
                // this pair's consecutive part of the list
                const int part = (n + (1 << a) - 1) >> a;
                const int mine = min(part, n - r * part);
                const unsigned char *lp = bt->list[sq] + r * part;
                const int x = 4 * (sq & 3), y = 4 * (sq >> 2) + 2 * (lane & 1);
                const float fx0 = (float)(px0 + x) + 0.5f, fy0 = (float)(py0 + y) + 0.5f;
                const float2 fx[2] = {make_float2(fx0, fx0 + 1.0f), make_float2(fx0 + 2.0f, fx0 + 3.0f)};
                const float2 fy = make_float2(fy0, fy0 + 1.0f);
                float2 al[3][2][2], be[3][2][2];  // channel, row, column pair
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int k = 0; k < 4; ++k) al[c][k >> 1][k & 1] = f2(1.0f), be[c][k >> 1][k & 1] = f2(0.0f);
                int idx = mine > 0 ? *lp : kOBatch;
#pragma unroll 1
                for (int k = 1; k <= steps; ++k) {
                    const float4 pa = bt->pa[idx];
                    const float4 pb = bt->pb[idx];
                    ++lp;
                    idx = k < mine ? *lp : kOBatch;
                    // the largest x; compared as unsigned integers, so that a negative one counts as
                    // the largest
                    const uint32_t emax = max(__float_as_uint(pb.x), max(__float_as_uint(pb.y), __float_as_uint(pb.z)));
                    const uint32_t xmax = __float_as_uint(__uint_as_float(emax) * pb.w);
                    const uint32_t most = __reduce_max_sync(0xffffffffu, xmax);
                    if (most <= __float_as_uint(kDeg3Max))
                        apply_record<3>(pa, pb, fx, fy, al, be);
                    else if (most <= __float_as_uint(kDeg4Max))
                        apply_record<4>(pa, pb, fx, fy, al, be);
                    else if (most <= __float_as_uint(kDeg6Max))
                        apply_record<6>(pa, pb, fx, fy, al, be);
                    else
                        apply_record<5>(pa, pb, fx, fy, al, be);
                }
                // compose the maps of a square's pairs, parts in list order
                for (int d = 2; d < (2 << a); d <<= 1) {
                    const bool near = (lane & d) != 0;  // this lane's part is applied after the other's
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float2 &A = al[c][k >> 1][k & 1], &B = be[c][k >> 1][k & 1];
                            const float2 oa = make_float2(__shfl_xor_sync(0xffffffffu, A.x, d),
                                                          __shfl_xor_sync(0xffffffffu, A.y, d));
                            const float2 ob = make_float2(__shfl_xor_sync(0xffffffffu, B.x, d),
                                                          __shfl_xor_sync(0xffffffffu, B.y, d));
                            B = __ffma2_rn(near ? A : oa, near ? ob : B, near ? B : ob);
                            A = __fmul2_rn(A, oa);
                        }
                }
                if (r == 0 && n > 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int rr = 0; rr < 2; ++rr) {
                            float4 *pA = reinterpret_cast<float4 *>(&ws->map[c][y + rr][x]);
                            float4 *pB = reinterpret_cast<float4 *>(&ws->map[3 + c][y + rr][x]);
                            const float2 a0 = al[c][rr][0], a1 = al[c][rr][1], b0 = be[c][rr][0], b1 = be[c][rr][1];
                            float4 A = *pA, B = *pB;
                            B.x = fmaf(a0.x, B.x, b0.x), B.y = fmaf(a0.y, B.y, b0.y);
                            B.z = fmaf(a1.x, B.z, b1.x), B.w = fmaf(a1.y, B.w, b1.y);
                            A.x *= a0.x, A.y *= a0.y, A.z *= a1.x, A.w *= a1.y;
                            *pA = A;
                            *pB = B;
                        }
                }
                __syncwarp();
                i += 16 >> a;
            }
        }
        __syncwarp();

        // epilogue: a whole tile writes I = beta (black background), or with map_out the
        // map (alpha rgb, beta rgb); a slice of a split tile stores its map
        const int oc = map_out ? 6 : 3;  // floats per pixel
        float *o = out + (int64_t)v * H * W * oc;
        if (slot < 0) {
            for (int k = lane; k < kRegion * kRegion * oc; k += 32) {
                const int p = k / oc, c = k - p * oc, r = p / kRegion, col = p % kRegion;
                if (r < th && col < tw)
                    o[((int64_t)(py0 + r) * W + px0 + col) * oc + c] = ws->map[map_out ? c : 3 + c][r][col];
            }
        } else {
            float *ms = ord_scratch + (int64_t)slice * 6 * T * T;  // [alpha r g b, beta r g b][T][T]
            if (((T | sub) & 3) == 0) {  // rows of the region in fours (past its width: another pixel of it)
                for (int k = lane; k < 6 * kRegion * kRegion / 4; k += 32) {
                    const int c = k / (kRegion * kRegion / 4), r = (k / (kRegion / 4)) % kRegion, col = 4 * (k % (kRegion / 4));
                    if (r < th && col < sub)
                        *reinterpret_cast<float4 *>(&ms[c * T * T + (qy + r) * T + qx + col]) =
                            reinterpret_cast<const float4 *>(map)[k];
                }
            } else {
                for (int k = lane; k < 6 * kRegion * kRegion; k += 32) {
                    const int c = k / (kRegion * kRegion), r = (k / kRegion) % kRegion, col = k % kRegion;
                    if (r < th && col < tw) ms[c * T * T + (qy + r) * T + qx + col] = map[k];
                }
            }
        }
        __syncwarp();
    }
}

// k_compose_slices: the maps of a split tile's slices, far to near, one thread per pixel and
// channel, the maps of several slices on their way together.  A CTA takes 256 pixels and channels
// of a tile at a time; it collects those of split tiles among every gridDim-th, so that
// neighbouring crowded tiles go to different CTAs.  Bound by the latency of the loads: 41 us on
// the 10 M-particle frame at 2048^2 (crowded tiles of some 350 slices), 109 with the loads left to
// the compiler.  The last warp to finish a tile used to compose it, which held the splat up: 1.90
// ms against 1.53 and these 41 us; 4 M particles at 1024^2: 0.89 ms against 0.40 + 0.09 (with the
// cheaper update).
constexpr int kComposeThreads = 256;
constexpr int kAtOnce = 16;  // slices loaded together

__global__ void __launch_bounds__(kComposeThreads) k_compose_slices(FrameDev fr, const float *__restrict__ slices,
                                                                    float *__restrict__ out, int map_out) {
    if (fr.status[kStatOverflow]) return;
    __shared__ int s_todo[kComposeThreads], s_n;
    const int T = fr.T, T2 = T * T, W = fr.views[0].W, H = fr.views[0].H, ntx = fr.views[0].ntx;
    const int oc = map_out ? 6 : 3, parts = (3 * T2 + kComposeThreads - 1) / kComposeThreads;
    const int count = fr.n_tiles * parts;  // at most 16384 tiles of 12 parts
    for (int i0 = blockIdx.x; i0 < count; i0 += gridDim.x * kComposeThreads) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const int mine = i0 + threadIdx.x * gridDim.x;
        if (mine < count && fr.split_slot[mine / parts] >= 0) s_todo[atomicAdd(&s_n, 1)] = mine;
        __syncthreads();
        for (int e = 0; e < s_n; ++e) {
            const int t = s_todo[e] / parts, part = s_todo[e] - t * parts, tx = t % ntx, ty = t / ntx;
            const int j = part * kComposeThreads + threadIdx.x;
            const int ch = j / T2, pix = j - ch * T2, r = pix / T, col = pix - r * T;
            if (ch >= 3 || ty * T + r >= H || tx * T + col >= W) continue;
            const int s0 = fr.item_off[t], s1 = fr.item_off[t + 1];
            const float *m = slices + (int64_t)s0 * 6 * T2 + j;
            float A = 1.0f, I = 0.0f;
            for (int k = s0; k < s1; k += kAtOnce, m += kAtOnce * 6 * T2) {
                float a[kAtOnce], b[kAtOnce];
#pragma unroll
                for (int g = 0; g < kAtOnce; ++g) {  // past the last slice: the map that changes nothing
                    a[g] = k + g < s1 ? __ldg(m + g * 6 * T2) : 1.0f;
                    b[g] = k + g < s1 ? __ldg(m + g * 6 * T2 + 3 * T2) : 0.0f;
                }
#pragma unroll
                for (int g = 0; g < kAtOnce; ++g) {
                    I = fmaf(a[g], I, b[g]);
                    A *= a[g];
                }
            }
            float *p = out + ((int64_t)(ty * T + r) * W + tx * T + col) * oc;
            if (map_out) p[ch] = A, p[3 + ch] = I;
            else p[ch] = I;
        }
        __syncthreads();
    }
}

__global__ void k_gather_records(const float4 *__restrict__ src, const uint32_t *__restrict__ idx, uint32_t last,
                                 int64_t n, float4 *dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[min(idx[i], last)];
}

static int grid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 32)); }

cudaError_t launch_gather_records(const float4 *src, const uint32_t *idx, uint32_t last, int64_t n, float4 *dst,
                                  cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_gather_records<<<grid_for(n), 256, 0, st>>>(src, idx, last, n, dst);
    return cudaGetLastError();
}

int ordered_split(int T) { return T > 16 ? 2 : 1; }

static size_t ordered_smem() { return sizeof(OWarpSmem) * kOWarps; }

int ordered_ctas_per_sm() {
    const void *fn = (const void *)k_splat_ordered<false>;
    if (ensure_smem_limit(fn, ordered_smem()) != cudaSuccess) return 1;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kOWarps * 32, ordered_smem()) != cudaSuccess) return 1;
    return std::max(1, nb);
}

int ordered_workers_per_sm() { return ordered_ctas_per_sm() * kOWarps; }

// Composition of depth-slab maps (Section 2.1: the transfer along a line of sight takes
// the farther material first; Section 4.2.2: tasks render their particles independently).
// maps: n arrays of `pixels` x 6 floats, farthest first, each pixel (alpha rgb, beta rgb)
// of I_out = alpha I_in + beta.  Composing far to near: beta <- alpha_k beta + beta_k,
// alpha <- alpha_k alpha.  One thread per (pixel, channel); the result's beta is the
// frame from a black background.
__global__ void k_compose_maps(const float *__restrict__ maps, int n, int64_t pixels, float *__restrict__ out) {
    const int64_t count = pixels * 3, stride = pixels * 6;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < count; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = j / 3;
        const int64_t ia = p * 6 + (j - p * 3), ib = ia + 3;
        float a = maps[ia], b = maps[ib];
        for (int k = 1; k < n; ++k) {
            const float ak = maps[k * stride + ia], bk = maps[k * stride + ib];
            b = __fmaf_rn(ak, b, bk);
            a = __fmul_rn(ak, a);
        }
        out[ia] = a;
        out[ib] = b;
    }
}

cudaError_t launch_compose_maps(const float *maps, int n, int64_t pixels, float *out, cudaStream_t st) {
    if (pixels <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((pixels * 3 + 255) / 256, 152 * 16);
    k_compose_maps<<<(int)blocks, 256, 0, st>>>(maps, n, pixels, out);
    return cudaGetLastError();
}

cudaError_t launch_splat_ordered(const SceneDev &sc, const FrameDev &fr, float *out, const float *absorb,
                                 float *ord_scratch, int map_out, int grid, int splits, cudaStream_t st) {
    auto fn = sc.emit ? k_splat_ordered<true> : k_splat_ordered<false>;
    cudaError_t err = ensure_smem_limit((const void *)fn, ordered_smem());
    if (err != cudaSuccess) return err;
    if ((err = launch_item_order(fr, st)) != cudaSuccess) return err;
    fn<<<grid, kOWarps * 32, ordered_smem(), st>>>(sc, fr, fr.queue, out, ordered_split(fr.T), absorb, ord_scratch, map_out);
    if (splits) {
        const int ctas = std::min(fr.n_tiles * ((3 * fr.T * fr.T + kComposeThreads - 1) / kComposeThreads), 152 * 6);
        k_compose_slices<<<ctas, kComposeThreads, 0, st>>>(fr, ord_scratch, out, map_out);
    }
    return cudaGetLastError();
}

}  // namespace spl
