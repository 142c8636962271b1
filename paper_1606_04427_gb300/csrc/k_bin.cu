// Scene preparation and tile binning (count / scan / scatter) for the Splotch hot path.
//
// Section 3.1 builds, per tile, the list of particles that affect it; Section 3.2.1
// gives the membership rule and notes that growing per-thread vectors stalled on
// allocation.  Here the lists are one flat array sized exactly from a counting pass:
//   k_count      streams the particles once (coalesced SoA loads), rasterises them
//                for a group of views, histograms tile memberships in shared memory and
//                writes each chunk's count of every tile;
//   k_chunk_scan scans every tile's counts over the chunks in chunk order: the base of
//                each chunk's slice of the tile segment, and the tile's total;
//   k_scan       turns the totals into tile segment offsets and the splat's work items;
//   k_scatter    streams the particles again and writes a 16-byte record per
//                (particle, tile) pair into its tile segment (each chunk's slice in the
//                order its warps reach the records); k_scatter_stable writes every slice
//                in ascending particle index, as Section 3.2.1 builds the lists by walking
//                the particles in order.
#include "splotch_internal.cuh"

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

namespace spl {

cudaError_t ensure_smem_limit(const void *kernel, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, size_t> set;
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    std::lock_guard<std::mutex> lk(mu);
    size_t &cur = set[std::make_pair(kernel, dev)];
    if (cur >= bytes) return cudaSuccess;
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    // the largest shared-memory carveout, so that the CTAs the occupancy allows all fit
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (err == cudaSuccess) cur = bytes;
    return err;
}

// largest tile histogram: G x n_tiles <= kMaxTiles counters
constexpr size_t kBinSmemMax = sizeof(int) * (size_t)kMaxTiles;

// ---------------------------------------------------------------------------------------
// Scene preparation (Section 2.1: ranging, normalisation, optional logarithm).

__device__ __forceinline__ unsigned order_key(float f) {
    unsigned b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Sort key of a depth z_c such that ascending keys run from the farthest particle to the
// nearest: the order-preserving unsigned image of the float, complemented.
__device__ __forceinline__ uint32_t depth_key(float zc) { return ~order_key(zc); }
constexpr uint32_t kInactiveKey = 0xFFFFFFFFu;  // no finite depth in front of the near plane maps here

__global__ void k_minmax(const float *__restrict__ I, int64_t begin, int64_t end, int i_log,
                         unsigned *keys) {
    unsigned lo = 0xFFFFFFFFu, hi = 0u;
    for (int64_t i = begin + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < end;
         i += (int64_t)gridDim.x * blockDim.x) {
        float v = I[i];
        if (i_log) v = logf(fmaxf(v, 1e-30f));
        if (!isfinite(v)) continue;
        unsigned k = order_key(v);
        lo = min(lo, k);
        hi = max(hi, k);
    }
    for (int o = 16; o; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&keys[0], lo);
        atomicMax(&keys[1], hi);
    }
}

cudaError_t launch_minmax(int, const float *I, int64_t begin, int64_t end, int i_log, unsigned *keys,
                          cudaStream_t st) {
    if (end <= begin) return cudaSuccess;
    int64_t blocks = (end - begin + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_minmax<<<(int)blocks, 256, 0, st>>>(I, begin, end, i_log, keys);
    return cudaGetLastError();
}

template <typename T> __device__ __forceinline__ T to_store(float v);
template <> __device__ __forceinline__ float to_store<float>(float v) { return v; }
template <> __device__ __forceinline__ __half to_store<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 to_store<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}

template <typename T>
__global__ void k_prepare(const float *__restrict__ x, const float *__restrict__ y,
                          const float *__restrict__ z, const float *__restrict__ h,
                          const float *__restrict__ I, int64_t n, int n_types,
                          const int64_t *__restrict__ tb, const float *__restrict__ lo,
                          const float *__restrict__ hi, const int *__restrict__ i_log, T *ox, T *oy,
                          T *oz, T *oh, T *oit, int *bad, int64_t first) {
    for (int64_t i = first + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int a = 0, b = n_types - 1;  // species: last t with tb[t] <= i
        while (a < b) {
            int mid = (a + b + 1) >> 1;
            if (tb[mid] <= i) a = mid; else b = mid - 1;
        }
        const float xv = x[i], yv = y[i], zv = z[i], hv = h[i], Iv = I[i];
        if (!(isfinite(xv) && isfinite(yv) && isfinite(zv) && isfinite(hv) && hv > 0.0f && isfinite(Iv)))
            atomicOr(bad, 1);
        float v = i_log[a] ? logf(fmaxf(Iv, 1e-30f)) : Iv;
        const float span = __fsub_rn(hi[a], lo[a]);
        float t = span > 0.0f ? __fdiv_rn(__fsub_rn(v, lo[a]), span) : 0.0f;
        t = fminf(fmaxf(t, 0.0f), 1.0f);
        ox[i] = to_store<T>(xv);
        oy[i] = to_store<T>(yv);
        oz[i] = to_store<T>(zv);
        oh[i] = to_store<T>(hv);
        oit[i] = to_store<T>(t);
    }
}

// Four consecutive particles per thread with 16-byte loads of every input array (inputs
// 16-byte aligned): a quarter of the memory requests, which matters when the inputs are
// read in place from page-locked host memory over the host link.
template <typename T>
__global__ void k_prepare4(const float4 *__restrict__ x, const float4 *__restrict__ y,
                           const float4 *__restrict__ z, const float4 *__restrict__ h,
                           const float4 *__restrict__ I, int64_t n4, int n_types,
                           const int64_t *__restrict__ tb, const float *__restrict__ lo,
                           const float *__restrict__ hi, const int *__restrict__ i_log, T *ox, T *oy,
                           T *oz, T *oh, T *oit, int *bad) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n4; q += (int64_t)gridDim.x * blockDim.x) {
        const float4 xv = x[q], yv = y[q], zv = z[q], hv = h[q], Iv = I[q];
        const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, ys[4] = {yv.x, yv.y, yv.z, yv.w};
        const float zs[4] = {zv.x, zv.y, zv.z, zv.w}, hs[4] = {hv.x, hv.y, hv.z, hv.w};
        const float is[4] = {Iv.x, Iv.y, Iv.z, Iv.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = 4 * q + k;
            int a = 0, b = n_types - 1;  // species: last t with tb[t] <= i
            while (a < b) {
                int mid = (a + b + 1) >> 1;
                if (tb[mid] <= i) a = mid; else b = mid - 1;
            }
            if (!(isfinite(xs[k]) && isfinite(ys[k]) && isfinite(zs[k]) && isfinite(hs[k]) && hs[k] > 0.0f &&
                  isfinite(is[k])))
                atomicOr(bad, 1);
            float v = i_log[a] ? logf(fmaxf(is[k], 1e-30f)) : is[k];
            const float span = __fsub_rn(hi[a], lo[a]);
            float t = span > 0.0f ? __fdiv_rn(__fsub_rn(v, lo[a]), span) : 0.0f;
            t = fminf(fmaxf(t, 0.0f), 1.0f);
            ox[i] = to_store<T>(xs[k]);
            oy[i] = to_store<T>(ys[k]);
            oz[i] = to_store<T>(zs[k]);
            oh[i] = to_store<T>(hs[k]);
            oit[i] = to_store<T>(t);
        }
    }
}

template <typename T>
static void prepare_launch(const float *x, const float *y, const float *z, const float *h, const float *I,
                           int64_t n, int n_types, const int64_t *tb, const float *lo, const float *hi,
                           const int *i_log, void *ox, void *oy, void *oz, void *oh, void *oit, int *bad,
                           cudaStream_t st) {
    auto aligned = [](const void *p) { return ((uintptr_t)p & 15u) == 0; };
    int64_t done = 0;
    if (aligned(x) && aligned(y) && aligned(z) && aligned(h) && aligned(I) && n >= 4) {
        const int64_t n4 = n / 4;
        int64_t blocks = (n4 + 255) / 256;
        if (blocks > 65536) blocks = 65536;
        k_prepare4<T><<<(int)blocks, 256, 0, st>>>((const float4 *)x, (const float4 *)y, (const float4 *)z,
                                                   (const float4 *)h, (const float4 *)I, n4, n_types, tb, lo, hi,
                                                   i_log, (T *)ox, (T *)oy, (T *)oz, (T *)oh, (T *)oit, bad);
        done = 4 * n4;
    }
    if (done < n) {
        // the remaining particles (or all, for unaligned inputs), one per thread; the
        // outputs are offset so indices stay global
        int64_t blocks = (n - done + 255) / 256;
        if (blocks > 65536) blocks = 65536;
        k_prepare<T><<<(int)blocks, 256, 0, st>>>(x, y, z, h, I, n, n_types, tb, lo, hi, i_log, (T *)ox, (T *)oy,
                                                  (T *)oz, (T *)oh, (T *)oit, bad, done);
    }
}

// Per-particle emission of a scene with vector-coloured species (Section 2.1: colour
// directly from a vector input field, or from a scalar through the colormap): for a
// vector species, C~ = clamp((C' - lo) / (hi - lo), 0, 1) per component (C' = ln(max(C,
// 1e-30)) with the log flag; 0 when hi <= lo) and e = brightness C~; for the others the
// colormap (premultiplied by brightness) interpolated at the stored normalised intensity.
// The species index rides in .w.  A non-finite colour component sets *bad.
template <int S>
__global__ void k_emission(SceneDev sc, const float *__restrict__ rgb, const int *__restrict__ vec,
                           const float *__restrict__ lo, const float *__restrict__ hi, const int *__restrict__ lg,
                           const float *__restrict__ beta, float4 *emit, int *bad) {
    __shared__ int64_t s_tb[kMaxTypes + 1];
    for (int k = threadIdx.x; k <= sc.n_types; k += blockDim.x) s_tb[k] = sc.type_begin[k];
    __syncthreads();
    int type = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < sc.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        while (type + 1 < sc.n_types && i >= s_tb[type + 1]) ++type;
        float e[3];
        if (vec[type]) {
            const float l = lo[type], span = hi[type] - l;
            for (int c = 0; c < 3; ++c) {
                float v = rgb[3 * i + c];
                if (!isfinite(v)) atomicExch(bad, 1);
                if (lg[type]) v = logf(fmaxf(v, 1e-30f));
                float t = span > 0.0f ? (v - l) / span : 0.0f;
                t = fminf(fmaxf(t, 0.0f), 1.0f);
                e[c] = beta[type] * t;
            }
        } else {
            const float It = load1<S>(sc.it, i);
            const int len = sc.lut_len[type];
            const float f = It * (float)(len - 1);
            const int kk = min((int)f, len - 2);
            const float tau = f - (float)kk;
            const float4 c0 = sc.lut[sc.lut_off[type] + kk], c1 = sc.lut[sc.lut_off[type] + kk + 1];
            e[0] = (1.0f - tau) * c0.x + tau * c1.x;
            e[1] = (1.0f - tau) * c0.y + tau * c1.y;
            e[2] = (1.0f - tau) * c0.z + tau * c1.z;
        }
        emit[i] = make_float4(e[0], e[1], e[2], __int_as_float(type));
    }
}

cudaError_t launch_emission(int storage, const SceneDev &sc, const float *rgb, const int *vec, const float *lo,
                            const float *hi, const int *lg, const float *beta, float4 *emit, int *bad,
                            cudaStream_t st) {
    if (sc.n <= 0) return cudaSuccess;
    int64_t blocks = (sc.n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (storage == 0) k_emission<0><<<(int)blocks, 256, 0, st>>>(sc, rgb, vec, lo, hi, lg, beta, emit, bad);
    else if (storage == 1) k_emission<1><<<(int)blocks, 256, 0, st>>>(sc, rgb, vec, lo, hi, lg, beta, emit, bad);
    else k_emission<2><<<(int)blocks, 256, 0, st>>>(sc, rgb, vec, lo, hi, lg, beta, emit, bad);
    return cudaGetLastError();
}

cudaError_t launch_prepare(const float *x, const float *y, const float *z, const float *h,
                           const float *I, int64_t n, int n_types, const int64_t *type_begin,
                           const float *lo, const float *hi, const int *i_log, int storage,
                           void *ox, void *oy, void *oz, void *oh, void *oit, int *bad,
                           cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    switch (storage) {
    case 0:
        prepare_launch<float>(x, y, z, h, I, n, n_types, type_begin, lo, hi, i_log, ox, oy, oz, oh, oit, bad, st);
        break;
    case 1:
        prepare_launch<__half>(x, y, z, h, I, n, n_types, type_begin, lo, hi, i_log, ox, oy, oz, oh, oit, bad, st);
        break;
    default:
        prepare_launch<__nv_bfloat16>(x, y, z, h, I, n, n_types, type_begin, lo, hi, i_log, ox, oy, oz, oh, oit,
                                      bad, st);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// k_count: raster a chunk of particles for up to G views and count tile memberships.
// Bound by instruction issue (raster, tile tests, histogram atomics).  On the 100 M-particle
// frame (FP16) 1.30 -> 1.20 ms with the shared squares of tile_mask2 and candidate blocks without
// divisions, 1.11 ms with the attributes kept as stored until they are used.

// Bin one particle for every view of the group: 2 x 2 candidate tiles or fewer by this
// lane, larger candidate boxes by the whole warp (one such particle at a time).  Called by
// all lanes of the warp together.
__device__ __forceinline__ void count_particle(bool valid, float x, float y, float z, float h,
                                               const ViewParams *s_view, int g_n, int *s_hist, int nt,
                                               int lane) {
    for (int g = 0; g < g_n; ++g) {
        const ViewParams &vp = s_view[g];
        int *hist = s_hist + g * nt;
        Raster r;
        int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
        if (valid && raster_one(vp, x, y, z, h, r)) {
            tx0 = tile_of(vp, r.i0), tx1 = tile_of(vp, r.i1);
            ty0 = tile_of(vp, r.j0), ty1 = tile_of(vp, r.j1);
        }
        const bool small = tx1 >= tx0 && tx1 - tx0 <= 1 && ty1 - ty0 <= 1;
        if (small) {
            const uint32_t m = tile_mask2(vp, r.X, r.Y, r.R, tx0, tx1, ty0, ty1);
            const int t00 = ty0 * vp.ntx + tx0;
            if (m & 1u) atomicAdd(&hist[t00], 1);
            if (m & 2u) atomicAdd(&hist[t00 + 1], 1);
            if (m & 4u) atomicAdd(&hist[t00 + vp.ntx], 1);
            if (m & 8u) atomicAdd(&hist[t00 + vp.ntx + 1], 1);
        }
        uint32_t big = __ballot_sync(0xffffffffu, tx1 >= tx0 && !small);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const float bX = __shfl_sync(0xffffffffu, r.X, src), bY = __shfl_sync(0xffffffffu, r.Y, src);
            const float bR = __shfl_sync(0xffffffffu, r.R, src);
            const int bx0 = __shfl_sync(0xffffffffu, tx0, src), bx1 = __shfl_sync(0xffffffffu, tx1, src);
            const int by0 = __shfl_sync(0xffffffffu, ty0, src), by1 = __shfl_sync(0xffffffffu, ty1, src);
            // blocks of 8 x 4 candidates, one per lane
            for (int ty = by0 + (lane >> 3); ty - (lane >> 3) <= by1; ty += 4)
                for (int tx = bx0 + (lane & 7); tx - (lane & 7) <= bx1; tx += 8)
                    if (tx <= bx1 && ty <= by1 && tile_member(vp, bX, bY, bR, tx, ty))
                        atomicAdd(&hist[ty * vp.ntx + tx], 1);
        }
    }
}

template <int S>
__global__ void __launch_bounds__(kThreads) k_count(SceneDev sc, FrameDev fr) {
    extern __shared__ int s_hist[];  // [g_n][n_tiles]
    __shared__ ViewParams s_view[kMaxGroup];
    const int b = blockIdx.x;
    const int v0 = blockIdx.y * fr.G;
    const int g_n = min(fr.G, fr.V - v0);
    const int nt = fr.n_tiles;
    for (int k = threadIdx.x; k < g_n * nt; k += blockDim.x) s_hist[k] = 0;
    if (threadIdx.x < g_n) s_view[threadIdx.x] = fr.views[v0 + threadIdx.x];
    // the frame's first kernel clears what the later ones count into (each of its launches does,
    // before any of those)
    if (b == 0 && blockIdx.y == 0) {
        for (int k = threadIdx.x; k < 2 * kOrderBins; k += blockDim.x) fr.bins[k] = 0;
        if (threadIdx.x < 4) fr.status[threadIdx.x] = 0, fr.queue[threadIdx.x] = 0;
    }
    __syncthreads();

    const int64_t s = (int64_t)b * fr.chunk;
    const int64_t e = min(sc.n, s + fr.chunk);
    // Two particles per thread per iteration, A and B, each in its own registers: A's next
    // attributes are loaded as soon as A is binned and stay in flight while B is binned
    // (and the other way round), hiding DRAM latency.  The loop runs warp-uniformly (a lane
    // past the chunk end idles) because large particles are binned by the whole warp.
    const int lane = threadIdx.x & 31;
    const int64_t stride = blockDim.x;
    int64_t i = s + threadIdx.x;
    typename Stored<S>::T ax{}, ay{}, az{}, ah{}, bx{}, by{}, bz{}, bh{};
    if (i < e) ax = load_stored<S>(sc.x, i), ay = load_stored<S>(sc.y, i), az = load_stored<S>(sc.z, i), ah = load_stored<S>(sc.h, i);
    if (i + stride < e)
        bx = load_stored<S>(sc.x, i + stride), by = load_stored<S>(sc.y, i + stride), bz = load_stored<S>(sc.z, i + stride),
        bh = load_stored<S>(sc.h, i + stride);
    for (; i - lane < e; i += 2 * stride) {
        count_particle(i < e, value_of(ax), value_of(ay), value_of(az), value_of(ah), s_view, g_n, s_hist, nt, lane);
        const int64_t ia = i + 2 * stride;
        if (ia < e) ax = load_stored<S>(sc.x, ia), ay = load_stored<S>(sc.y, ia), az = load_stored<S>(sc.z, ia), ah = load_stored<S>(sc.h, ia);
        if (i + stride - lane >= e) break;
        count_particle(i + stride < e, value_of(bx), value_of(by), value_of(bz), value_of(bh), s_view, g_n, s_hist, nt, lane);
        const int64_t ib = i + 3 * stride;
        if (ib < e) bx = load_stored<S>(sc.x, ib), by = load_stored<S>(sc.y, ib), bz = load_stored<S>(sc.z, ib), bh = load_stored<S>(sc.h, ib);
    }
    __syncthreads();
    // this chunk's count of every tile (zeros included): k_chunk_scan turns the column of
    // each tile into chunk bases in chunk order
    for (int k = threadIdx.x; k < g_n * nt; k += blockDim.x) {
        const int g = k / nt, t = k - g * nt;
        fr.rel[((int64_t)(v0 + g) * fr.n_chunks + b) * nt + t] = s_hist[k];
    }
}

// f on the frame's views, at most `most` at a time: a grid's second dimension, over views or groups
// of views, ends at 65535.
constexpr int64_t kGridY = 65535;
template <class F> static cudaError_t by_views(const FrameDev &fr, int64_t most, F f) {
    for (int64_t v0 = 0; v0 < fr.V; v0 += most) {
        FrameDev part = fr;
        part.V = (int)std::min<int64_t>(most, fr.V - v0);
        part.views = fr.views + v0;
        part.rel = fr.rel + v0 * fr.n_chunks * fr.n_tiles;
        part.counts = fr.counts + v0 * fr.n_tiles;
        part.offsets = fr.offsets + v0 * fr.n_tiles;
        f(part);
    }
    return cudaGetLastError();
}

template <int S> static cudaError_t count_impl(const SceneDev &sc, const FrameDev &fr, cudaStream_t st) {
    const size_t smem = (size_t)fr.G * fr.n_tiles * sizeof(int);
    cudaError_t err = ensure_smem_limit((const void *)k_count<S>, kBinSmemMax);
    if (err != cudaSuccess) return err;
    return by_views(fr, kGridY * fr.G, [&](const FrameDev &part) {
        k_count<S><<<dim3(part.n_chunks, (part.V + part.G - 1) / part.G), kThreads, smem, st>>>(sc, part);
    });
}

cudaError_t launch_count(int storage, const SceneDev &sc, const FrameDev &fr, cudaStream_t st) {
    if (storage == 0) return count_impl<0>(sc, fr, st);
    if (storage == 1) return count_impl<1>(sc, fr, st);
    return count_impl<2>(sc, fr, st);
}

// ---------------------------------------------------------------------------------------
// Scans of the tile counts.

template <typename T> __device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Exclusive block scan (1024 threads); returns the exclusive prefix, *total = block sum.
template <typename T> __device__ T block_excl_scan(T v, T *s_warp, T *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = warp_incl_scan(v);
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T w = s_warp[lane];
        T wi = warp_incl_scan(w);
        s_warp[lane] = wi - w;
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    T res = s_warp[warp] + incl - v;
    *total = s_warp[32];
    __syncthreads();
    return res;
}

// ---------------------------------------------------------------------------------------
// k_chunk_scan: per (view, tile), the exclusive scan of the chunks' counts in chunk order
// (rel becomes each chunk's base inside the tile segment) and the tile's total.  The
// bases depend only on the counts, so the lists' layout is the same on every run.
//
// A CTA takes 32 tiles of a view (a lane each, so rows of rel are read 128 bytes at a time);
// its kChunkSegs warps share the chunks, sum their parts, and write the bases in a second read.
// Bound by the latency of the column walk: with one thread per tile it took 87 us on the 100 M
// frame (582 chunks, 16384 tiles), now 15 us.

constexpr int kChunkScanUnroll = 8, kChunkSegs = 8;

__global__ void __launch_bounds__(32 * kChunkSegs) k_chunk_scan(FrameDev fr) {
    __shared__ long long s_sum[kChunkSegs][32];
    const int nt = fr.n_tiles, nch = fr.n_chunks;
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
    const int per = (nch + kChunkSegs - 1) / kChunkSegs;
    const int b0 = min(nch, seg * per), b1 = min(nch, b0 + per);
    const int v = blockIdx.y, t = blockIdx.x * 32 + lane;
    int *col = fr.rel + (int64_t)v * nch * nt + t;
    long long sum = 0;
    if (t < nt) {
        int b = b0;
        for (; b + kChunkScanUnroll <= b1; b += kChunkScanUnroll) {
            int c[kChunkScanUnroll];
#pragma unroll
            for (int q = 0; q < kChunkScanUnroll; ++q) c[q] = col[(int64_t)(b + q) * nt];
#pragma unroll
            for (int q = 0; q < kChunkScanUnroll; ++q) sum += c[q];
        }
        for (; b < b1; ++b) sum += col[(int64_t)b * nt];
    }
    s_sum[seg][lane] = sum;
    __syncthreads();
    if (t >= nt) return;
    long long run = 0, total = 0;
#pragma unroll
    for (int k = 0; k < kChunkSegs; ++k) {
        if (k == seg) run = total;
        total += s_sum[k][lane];
    }
    int b = b0;
    for (; b + kChunkScanUnroll <= b1; b += kChunkScanUnroll) {
        int c[kChunkScanUnroll];
#pragma unroll
        for (int q = 0; q < kChunkScanUnroll; ++q) c[q] = col[(int64_t)(b + q) * nt];
#pragma unroll
        for (int q = 0; q < kChunkScanUnroll; ++q) {
            col[(int64_t)(b + q) * nt] = (int)run;
            run += c[q];
        }
    }
    for (; b < b1; ++b) {
        const int c = col[(int64_t)b * nt];
        col[(int64_t)b * nt] = (int)run;
        run += c;
    }
    if (seg == 0) {
        // a tile holding 2^31 pairs or more cannot be indexed by the 32-bit cursors
        if (total > (long long)INT32_MAX) {
            atomicExch(&fr.status[kStatOverflow], 1);
            total = INT32_MAX;
        }
        fr.counts[(int64_t)v * nt + t] = (int)total;
    }
}

// ---------------------------------------------------------------------------------------
// k_scan: tile segment offsets (int64), work items (a tile with more than K pairs is split
// into ceil(count / K) items), scratch slots of split tiles, and the items' size histogram
// for k_item_order.  A CTA scans kScanTiles tiles, or several times as many one after another, and
// sums those before it itself (their counts are in L2), so the CTAs need no order among them: 14 us
// for 16384 tiles and 22 us for 65536 (30 and 113 us with one CTA for all).  At most kScanCtas of
// them, or the sums would grow with the square of the tiles: 16 M tiles take 3.8 ms with the chunk
// scan, 46 with a CTA for each 4096 tiles, 31 with one for all.

constexpr int kScanItems = 4, kScanTiles = 1024 * kScanItems, kScanCtas = 152;

// Sum of two values over a 1024-thread CTA, for every thread.
__device__ __forceinline__ void block_sum2(long long &a, long long &b, long long (*s_w)[33]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    __syncthreads();
    if (lane == 0) s_w[0][warp] = a, s_w[1][warp] = b;
    __syncthreads();
    a = s_w[0][lane], b = s_w[1][lane];
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
}

// rounds: scans of kScanTiles tiles per CTA
__global__ void __launch_bounds__(1024) k_scan(FrameDev fr, int target_items, int kmin, int rounds) {
    __shared__ long long s_w[2][33];
    __shared__ int s_hist[kOrderBins];
    const int N = fr.V * fr.n_tiles;
    const int base = blockIdx.x * rounds * kScanTiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < kOrderBins) s_hist[threadIdx.x] = 0;
    // total pairs (counts is padded to a whole int4; entries past N are not added)
    long long tot = 0, none = 0;
#pragma unroll 4
    for (int k = 4 * threadIdx.x; k < N; k += 4 * blockDim.x) {
        const int4 c = *reinterpret_cast<const int4 *>(fr.counts + k);
        tot += (long long)c.x + (k + 1 < N ? c.y : 0) + (k + 2 < N ? c.z : 0) + (k + 3 < N ? c.w : 0);
    }
    block_sum2(tot, none, s_w);
    long long K64 = (tot + target_items - 1) / (target_items > 0 ? target_items : 1);
    if (K64 < kmin) K64 = kmin;
    if (K64 > (1LL << 30)) K64 = (1LL << 30);
    const int K = (int)K64;
    auto items_of = [&](int c) -> int { return c <= K ? 1 : (int)(((uint32_t)c + (uint32_t)K - 1u) / (uint32_t)K); };

    // pairs, and items and split tiles (two 32-bit halves), before this CTA's tiles
    long long pre_p = 0, pre_is = 0;
#pragma unroll 4
    for (int k = 4 * threadIdx.x; k < base; k += 4 * blockDim.x) {
        const int4 c = *reinterpret_cast<const int4 *>(fr.counts + k);
        pre_p += (long long)c.x + c.y + c.z + c.w;
        pre_is += ((long long)(items_of(c.x) + items_of(c.y) + items_of(c.z) + items_of(c.w)) << 32) +
                  (c.x > K) + (c.y > K) + (c.z > K) + (c.w > K);
    }
    if (base > 0) block_sum2(pre_p, pre_is, s_w);

    for (int round = 0; round < rounds; ++round) {
        const int64_t k0 = base + (int64_t)round * kScanTiles + threadIdx.x * kScanItems;
        int c[kScanItems], it[kScanItems];
        long long lp = 0, lis = 0;
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) {
            const bool in = k0 + q < N;
            c[q] = in ? fr.counts[k0 + q] : 0;
            it[q] = in ? items_of(c[q]) : 0;
            lp += c[q];
            lis += ((long long)it[q] << 32) + (c[q] > K);
            // the tile's last slice, counted once per warp and bin, and its full ones
            const int bin = in ? order_bin(c[q] - K * (it[q] - 1), K) : kOrderBins;
            const uint32_t peers = warp_peers<7>((uint32_t)bin);
            if (in && lane == __ffs(peers) - 1) atomicAdd(&s_hist[bin], __popc(peers));
            if (it[q] > 1) atomicAdd(&s_hist[order_bin(K, K)], it[q] - 1);
        }
        // exclusive scan of both over the CTA
        const long long wp = warp_incl_scan(lp), wis = warp_incl_scan(lis);
        __syncthreads();
        if (lane == 31) s_w[0][warp] = wp, s_w[1][warp] = wis;
        __syncthreads();
        const long long p_w = s_w[0][lane], is_w = s_w[1][lane];
        const long long p_i = warp_incl_scan(p_w), is_i = warp_incl_scan(is_w);
        long long ep = pre_p + wp - lp + __shfl_sync(0xffffffffu, p_i - p_w, warp);
        long long eis = pre_is + wis - lis + __shfl_sync(0xffffffffu, is_i - is_w, warp);
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) {
            if (k0 + q < N) {
                fr.offsets[k0 + q] = ep;
                fr.item_off[k0 + q] = (int)(eis >> 32);
                fr.split_slot[k0 + q] = c[q] > K ? (int)(eis & 0xffffffffll) : -1;
            }
            ep += c[q];
            eis += ((long long)it[q] << 32) + (c[q] > K);
        }
        pre_p += __shfl_sync(0xffffffffu, p_i, 31), pre_is += __shfl_sync(0xffffffffu, is_i, 31);
    }
    if (threadIdx.x < kOrderBins && s_hist[threadIdx.x]) atomicAdd(&fr.bins[threadIdx.x], s_hist[threadIdx.x]);
    if (blockIdx.x != gridDim.x - 1) return;
    // the scatter's cursors are 32-bit within a view
    int big = 0;
    if (tot > (long long)INT32_MAX)
        for (int v = warp; v < fr.V; v += 32) {
            long long sum = 0;
            for (int t = lane; t < fr.n_tiles; t += 32) sum += fr.counts[(int64_t)v * fr.n_tiles + t];
            for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            big |= sum > (long long)INT32_MAX;
        }
    big = __syncthreads_or(big);
    if (threadIdx.x == 0) {
        const int items = (int)(pre_is >> 32), splits = (int)(pre_is & 0xffffffffll);
        fr.offsets[N] = tot;
        fr.item_off[N] = items;
        fr.sizes[kSizePairs] = tot;
        fr.sizes[kSizeItems] = items;
        fr.sizes[kSizeSplits] = splits;
        fr.sizes[kSizeK] = K;
        const bool over = tot > fr.pair_cap || items > fr.item_cap || splits > fr.split_cap || big ||
                          fr.status[kStatOverflow];
        fr.status[kStatOverflow] = over ? 1 : 0;
    }
}

cudaError_t launch_scan(const FrameDev &fr, int target_items, int kmin, cudaStream_t st) {
    const int64_t N = (int64_t)fr.V * fr.n_tiles;
    const cudaError_t err = by_views(fr, kGridY, [&](const FrameDev &part) {
        k_chunk_scan<<<dim3((part.n_tiles + 31) / 32, part.V), 32 * kChunkSegs, 0, st>>>(part);
    });
    if (err != cudaSuccess) return err;
    const int blocks = (int)((N + kScanTiles - 1) / kScanTiles), rounds = (blocks + kScanCtas - 1) / kScanCtas;
    k_scan<<<(blocks + rounds - 1) / rounds, 1024, 0, st>>>(fr, target_items, kmin, rounds);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// k_scatter: same chunks as k_count; every (particle, tile) pair becomes a record
// {X, Y, R, type << 24 | 24-bit normalised intensity} in its tile segment (in scenes with
// a per-particle emission the last word is the particle index).  Each chunk fills its
// slice of a tile segment (slices in chunk order, k_chunk_scan) through a shared-memory
// cursor per tile: the slice holds exactly the chunk's members of the tile, in the order
// the CTA's warps reached them.  k_scatter_stable (below) orders them by particle index.

// Write the records of one particle for every view of the group (same split between
// lane and warp as count_particle).  Called by all lanes of the warp together.
__device__ __forceinline__ void scatter_particle(bool valid, int64_t i, float x, float y, float z, float h,
                                                 float code, const ViewParams *s_view, const int64_t *s_vbase,
                                                 int g_n, int *s_cur, int nt, const FrameDev &fr, int lane) {
    for (int g = 0; g < g_n; ++g) {
        const ViewParams &vp = s_view[g];
        int *cur = s_cur + g * nt;
        float4 *lists = fr.lists + s_vbase[g];
        int *pids = fr.pids ? fr.pids + s_vbase[g] : nullptr;
        Raster r;
        int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
        if (valid && raster_one(vp, x, y, z, h, r)) {
            tx0 = tile_of(vp, r.i0), tx1 = tile_of(vp, r.i1);
            ty0 = tile_of(vp, r.j0), ty1 = tile_of(vp, r.j1);
        }
        const bool small = tx1 >= tx0 && tx1 - tx0 <= 1 && ty1 - ty0 <= 1;
        if (small) {
            // all cursor reservations first, then the stores: one atomic latency per
            // particle instead of one per tile
            const float4 rec = make_float4(r.X, r.Y, r.R, code);
            const int t00 = ty0 * vp.ntx + tx0;
            const uint32_t m = tile_mask2(vp, r.X, r.Y, r.R, tx0, tx1, ty0, ty1);
            const bool m00 = m & 1u, m10 = m & 2u, m01 = m & 4u, m11 = m & 8u;
            const int p00 = m00 ? atomicAdd(&cur[t00], 1) : 0;
            const int p10 = m10 ? atomicAdd(&cur[t00 + 1], 1) : 0;
            const int p01 = m01 ? atomicAdd(&cur[t00 + vp.ntx], 1) : 0;
            const int p11 = m11 ? atomicAdd(&cur[t00 + vp.ntx + 1], 1) : 0;
            if (m00) lists[p00] = rec;
            if (m10) lists[p10] = rec;
            if (m01) lists[p01] = rec;
            if (m11) lists[p11] = rec;
            if (pids) {
                if (m00) pids[p00] = (int)i;
                if (m10) pids[p10] = (int)i;
                if (m01) pids[p01] = (int)i;
                if (m11) pids[p11] = (int)i;
            }
        }
        uint32_t big = __ballot_sync(0xffffffffu, tx1 >= tx0 && !small);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const float bX = __shfl_sync(0xffffffffu, r.X, src), bY = __shfl_sync(0xffffffffu, r.Y, src);
            const float bR = __shfl_sync(0xffffffffu, r.R, src);
            const float bcode = __shfl_sync(0xffffffffu, code, src);
            const int bid = __shfl_sync(0xffffffffu, (int)i, src);
            const int bx0 = __shfl_sync(0xffffffffu, tx0, src), bx1 = __shfl_sync(0xffffffffu, tx1, src);
            const int by0 = __shfl_sync(0xffffffffu, ty0, src), by1 = __shfl_sync(0xffffffffu, ty1, src);
            const float4 rec = make_float4(bX, bY, bR, bcode);
            for (int ty = by0 + (lane >> 3); ty - (lane >> 3) <= by1; ty += 4)
                for (int tx = bx0 + (lane & 7); tx - (lane & 7) <= bx1; tx += 8)
                    if (tx <= bx1 && ty <= by1 && tile_member(vp, bX, bY, bR, tx, ty)) {
                        const int pos = atomicAdd(&cur[ty * vp.ntx + tx], 1);
                        lists[pos] = rec;
                        if (pids) pids[pos] = bid;
                    }
        }
    }
}

// Record code of a particle: species in the top 8 bits, normalised intensity in 24 bits.
__device__ __forceinline__ float record_code(int type, float itn) {
    uint32_t q = __float2uint_rn(__fmul_rn(itn, (float)kCodeMax));
    q = min(q, kCodeMax);
    return __uint_as_float(((uint32_t)type << 24) | q);
}

template <int S>
__global__ void __launch_bounds__(kThreads) k_scatter(SceneDev sc, FrameDev fr) {
    if (fr.status[kStatOverflow]) return;
    // cursor of this chunk's slice of every tile segment, relative to the start of the
    // view's segments (a view holds fewer than 2^31 pairs: the scan checks it)
    extern __shared__ int s_cur[];  // [g_n][n_tiles]
    __shared__ ViewParams s_view[kMaxGroup];
    __shared__ int64_t s_vbase[kMaxGroup];
    __shared__ int64_t s_tb[kMaxTypes + 1];
    const int b = blockIdx.x;
    const int v0 = blockIdx.y * fr.G;
    const int g_n = min(fr.G, fr.V - v0);
    const int nt = fr.n_tiles;
    for (int k = threadIdx.x; k < g_n * nt; k += blockDim.x) {
        const int g = k / nt, t = k - g * nt;
        const int64_t *seg = fr.offsets + (int64_t)(v0 + g) * nt;
        s_cur[k] = (int)(seg[t] - seg[0]) + fr.rel[((int64_t)(v0 + g) * fr.n_chunks + b) * nt + t];
    }
    if (threadIdx.x < g_n) {
        s_view[threadIdx.x] = fr.views[v0 + threadIdx.x];
        s_vbase[threadIdx.x] = fr.offsets[(int64_t)(v0 + threadIdx.x) * nt];
    }
    for (int k = threadIdx.x; k <= sc.n_types; k += blockDim.x) s_tb[k] = sc.type_begin[k];
    __syncthreads();

    const int64_t s = (int64_t)b * fr.chunk;
    const int64_t e = min(sc.n, s + fr.chunk);
    // two particles per thread per iteration in separate registers (see k_count)
    const int lane = threadIdx.x & 31;
    const int64_t stride = blockDim.x;
    int type = 0;
    int64_t i = s + threadIdx.x;
    typename Stored<S>::T ax{}, ay{}, az{}, ah{}, ai{}, bx{}, by{}, bz{}, bh{}, bi{};
    if (i < e)
        ax = load_stored<S>(sc.x, i), ay = load_stored<S>(sc.y, i), az = load_stored<S>(sc.z, i), ah = load_stored<S>(sc.h, i),
        ai = load_stored<S>(sc.it, i);
    if (i + stride < e)
        bx = load_stored<S>(sc.x, i + stride), by = load_stored<S>(sc.y, i + stride), bz = load_stored<S>(sc.z, i + stride),
        bh = load_stored<S>(sc.h, i + stride), bi = load_stored<S>(sc.it, i + stride);
    for (; i - lane < e; i += 2 * stride) {
        if (i < e)
            while (type + 1 < sc.n_types && i >= s_tb[type + 1]) ++type;
        scatter_particle(i < e, i, value_of(ax), value_of(ay), value_of(az), value_of(ah),
                         sc.emit ? __uint_as_float((uint32_t)i) : record_code(type, value_of(ai)),
                         s_view, s_vbase, g_n, s_cur, nt, fr, lane);
        const int64_t ia = i + 2 * stride;
        if (ia < e)
            ax = load_stored<S>(sc.x, ia), ay = load_stored<S>(sc.y, ia), az = load_stored<S>(sc.z, ia), ah = load_stored<S>(sc.h, ia),
            ai = load_stored<S>(sc.it, ia);
        const int64_t j = i + stride;
        if (j - lane >= e) break;
        if (j < e)
            while (type + 1 < sc.n_types && j >= s_tb[type + 1]) ++type;
        scatter_particle(j < e, j, value_of(bx), value_of(by), value_of(bz), value_of(bh),
                         sc.emit ? __uint_as_float((uint32_t)j) : record_code(type, value_of(bi)),
                         s_view, s_vbase, g_n, s_cur, nt, fr, lane);
        const int64_t ib = i + 3 * stride;
        if (ib < e)
            bx = load_stored<S>(sc.x, ib), by = load_stored<S>(sc.y, ib), bz = load_stored<S>(sc.z, ib), bh = load_stored<S>(sc.h, ib),
            bi = load_stored<S>(sc.it, ib);
    }
}

template <int S> static cudaError_t scatter_impl(const SceneDev &sc, const FrameDev &fr, cudaStream_t st) {
    const size_t smem = (size_t)fr.G * fr.n_tiles * sizeof(int);
    cudaError_t err =
        ensure_smem_limit((const void *)k_scatter<S>, kBinSmemMax);
    if (err != cudaSuccess) return err;
    return by_views(fr, kGridY * fr.G, [&](const FrameDev &part) {
        k_scatter<S><<<dim3(part.n_chunks, (part.V + part.G - 1) / part.G), kThreads, smem, st>>>(sc, part);
    });
}


// ---------------------------------------------------------------------------------------
// k_scatter_stable: the same slices, each in ascending particle index (as the per-thread
// index vectors of Section 3.2.1 are filled by walking each thread's particle range in
// order).  A CTA takes its chunk in rounds of kThreads consecutive particles (thread k
// holds particle round + k).  Per round and view
//   1. every thread rasterises its particle and counts its member tiles (a particle with
//      more than 2 x 2 candidate tiles is counted by its whole warp, one candidate per
//      lane);
//   2. a block scan of the counts places every pair in the round's pair list, which is
//      therefore in particle order; the pairs are staged in shared memory as (tile,
//      particle slot), kStableStage at a time;
//   3. the staged pairs are sorted by tile, stably, with a radix sort of 7 bits per pass in
//      shared memory (one pass up to 128 tiles per view, else two);
//   4. a tile's pairs are then consecutive: the first sets the tile's cursor relative to its
//      place, all threads store the records at cursor + place (consecutive slots for a run),
//      and the last moves the cursor past the run.
// With the chunk bases in chunk order, every tile list is in ascending particle index
// whatever the order in which CTAs and warps run, so images do not depend on it.  Renders ask
// for it with SPLOTCH_STABLE.  Bound by instruction issue and barriers; 20.7 M pairs of the
// 10 M-particle frame in 1.35 ms (1.83 ms when one warp took the slots of all 32-pair slices in
// turn), the scatter in arrival order 0.34 ms.

constexpr int kStableStage = 4096;  // staged pairs per window
constexpr int kSlotBits = 10;       // particle slot in a staged pair (kThreads of them), tile above
static_assert(kThreads == 1 << kSlotBits && kMaxTiles <= 1 << 14, "staged pair: 14-bit tile, 10-bit slot");
constexpr int kDigitBits = 7, kDigits = 1 << kDigitBits, kBinWarps = kThreads / 32;
constexpr int kSortRows = kStableStage / kThreads;  // staged pairs per lane
// shared memory beyond the cursors: round records, two buffers of staged pairs, and the sort's
// counters (digit-major, one per warp, padded against bank conflicts)
constexpr size_t kStableExtra =
    sizeof(float4) * kThreads + sizeof(uint32_t) * (2 * kStableStage + kDigits * (kBinWarps + 1));

// One stable counting-sort pass of src[0, m) by 7 bits into dst, by the whole CTA: warps own
// consecutive parts and rank their pairs in order, and the exclusive scan of the counters in
// (digit, warp) order is where each warp's pairs of a digit go.
__device__ __forceinline__ void sort_pairs_pass(const uint32_t *src, uint32_t *dst, int m, int shift, uint32_t *cnt,
                                                int *s_scan) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    for (int k = tid; k < kDigits * (kBinWarps + 1); k += kThreads) cnt[k] = 0;
    __syncthreads();
    const int rows = (m + kThreads - 1) / kThreads;  // 32-pair rows per warp
    const int first = warp * rows * 32 + lane;
    uint32_t key[kSortRows];
    int rank[kSortRows];
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
        if (r >= rows) break;
        const int j = first + r * 32;
        key[r] = j < m ? src[j] : 0u;
        const uint32_t d = j < m ? (key[r] >> shift) & (kDigits - 1) : kDigits;
        const uint32_t peers = warp_peers<kDigitBits + 1>(d);
        const int leader = __ffs(peers) - 1;
        int before = 0;
        if (j < m && lane == leader) {
            before = (int)cnt[d * (kBinWarps + 1) + warp];
            cnt[d * (kBinWarps + 1) + warp] = before + __popc(peers);
        }
        rank[r] = __shfl_sync(0xffffffffu, before, leader) + __popc(peers & lt);
        __syncwarp();
    }
    __syncthreads();
    // thread t scans counters 4 t .. 4 t + 3 of the (digit, warp) sequence
    static_assert(kDigits * kBinWarps == 4 * kThreads, "four counters per thread");
    uint32_t *c = cnt + (tid >> 3) * (kBinWarps + 1) + 4 * (tid & 7);
    const int c0 = (int)c[0], c1 = (int)c[1], c2 = (int)c[2], c3 = (int)c[3];
    int all;
    const int base = block_excl_scan<int>(c0 + c1 + c2 + c3, s_scan, &all);
    c[0] = base, c[1] = base + c0, c[2] = base + c0 + c1, c[3] = base + c0 + c1 + c2;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
        if (r >= rows) break;
        if (first + r * 32 < m)
            dst[cnt[((key[r] >> shift) & (kDigits - 1)) * (kBinWarps + 1) + warp] + rank[r]] = key[r];
    }
    __syncthreads();
}

// Member tiles of a particle whose candidate box is large, tested by the whole warp (one
// candidate per lane, candidates in row-major order).  With kStage false, returns the
// member count; with kStage true, stages the members of the window [w0, w0 + m) at pair
// indices off, off + 1, ... (off: the particle's first pair).
template <bool kStage>
__device__ __forceinline__ int big_members(const ViewParams &vp, float X, float Y, float R, int bx0, int bx1,
                                           int by0, int by1, int off, int w0, int m, int slot, uint32_t *s_pair,
                                           int lane) {
    const int bw = bx1 - bx0 + 1, bh = by1 - by0 + 1;
    const uint32_t lt = (1u << lane) - 1u;
    int run = off - w0;
    for (int dy = 0; dy < bh; ++dy) {
        for (int dx0 = 0; dx0 < bw; dx0 += 32) {
            const int tx = bx0 + dx0 + lane, ty = by0 + dy;
            const bool mem = dx0 + lane < bw && tile_member(vp, X, Y, R, tx, ty);
            const uint32_t bal = __ballot_sync(0xffffffffu, mem);
            if (kStage) {
                const int j = run + __popc(bal & lt);
                if (mem && (unsigned)j < (unsigned)m)
                    s_pair[j] = (uint32_t)(ty * vp.ntx + tx) << kSlotBits | (uint32_t)slot;
            }
            run += __popc(bal);
        }
    }
    return run - (off - w0);
}

template <int S>
__global__ void __launch_bounds__(kThreads) k_scatter_stable(SceneDev sc, FrameDev fr) {
    if (fr.status[kStatOverflow]) return;
    extern __shared__ __align__(16) unsigned char s_raw[];
    float4 *s_rec = reinterpret_cast<float4 *>(s_raw);                     // [kThreads]
    uint32_t *s_pair = reinterpret_cast<uint32_t *>(s_rec + kThreads);     // [kStableStage]
    uint32_t *s_alt = s_pair + kStableStage;                               // [kStableStage]
    uint32_t *s_cnt = s_alt + kStableStage;                                // [kDigits][kBinWarps + 1]
    // cursor of this chunk's slice of every tile segment, relative to the start of the
    // view's segments (a view holds fewer than 2^31 pairs: the scan checks it)
    int *s_cur = reinterpret_cast<int *>(s_cnt + kDigits * (kBinWarps + 1));  // [g_n][n_tiles]
    __shared__ ViewParams s_view[kMaxGroup];
    __shared__ int64_t s_vbase[kMaxGroup];
    __shared__ int64_t s_tb[kMaxTypes + 1];
    __shared__ int s_scan[33];
    const int b = blockIdx.x;
    const int v0 = blockIdx.y * fr.G;
    const int g_n = min(fr.G, fr.V - v0);
    const int nt = fr.n_tiles;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k < g_n * nt; k += blockDim.x) {
        const int g = k / nt, t = k - g * nt;
        const int64_t *seg = fr.offsets + (int64_t)(v0 + g) * nt;
        s_cur[k] = (int)(seg[t] - seg[0]) + fr.rel[((int64_t)(v0 + g) * fr.n_chunks + b) * nt + t];
    }
    if (tid < g_n) {
        s_view[tid] = fr.views[v0 + tid];
        s_vbase[tid] = fr.offsets[(int64_t)(v0 + tid) * nt];
    }
    for (int k = tid; k <= sc.n_types; k += blockDim.x) s_tb[k] = sc.type_begin[k];
    __syncthreads();

    const int64_t s = (int64_t)b * fr.chunk;
    const int64_t e = min(sc.n, s + fr.chunk);
    int type = 0;
    int64_t i = s + tid;
    typename Stored<S>::T cx{}, cy{}, cz{}, ch{}, ci{};
    if (i < e)
        cx = load_stored<S>(sc.x, i), cy = load_stored<S>(sc.y, i), cz = load_stored<S>(sc.z, i), ch = load_stored<S>(sc.h, i),
        ci = load_stored<S>(sc.it, i);
    for (int64_t r0 = s; r0 < e; r0 += kThreads, i += kThreads) {
        const bool valid = i < e;
        // the next round's attributes load while this round is binned
        typename Stored<S>::T nx{}, ny{}, nz{}, nh{}, ni{};
        const int64_t in = i + kThreads;
        if (in < e)
            nx = load_stored<S>(sc.x, in), ny = load_stored<S>(sc.y, in), nz = load_stored<S>(sc.z, in), nh = load_stored<S>(sc.h, in),
            ni = load_stored<S>(sc.it, in);
        if (valid)
            while (type + 1 < sc.n_types && i >= s_tb[type + 1]) ++type;
        const float code = sc.emit ? __uint_as_float((uint32_t)i) : record_code(type, value_of(ci));
        for (int g = 0; g < g_n; ++g) {
            const ViewParams &vp = s_view[g];
            Raster r;
            r.X = r.Y = r.R = 0.0f;
            int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
            if (valid && raster_one(vp, value_of(cx), value_of(cy), value_of(cz), value_of(ch), r)) {
                tx0 = tile_of(vp, r.i0), tx1 = tile_of(vp, r.i1);
                ty0 = tile_of(vp, r.j0), ty1 = tile_of(vp, r.j1);
            }
            const bool small = tx1 >= tx0 && tx1 - tx0 <= 1 && ty1 - ty0 <= 1;
            // member bits of a small particle: (tx0, ty0), (tx1, ty0), (tx0, ty1), (tx1, ty1)
            uint32_t mask = 0;
            if (small) {
                mask = tile_mask2(vp, r.X, r.Y, r.R, tx0, tx1, ty0, ty1);
            }
            int cnt = __popc(mask);
            const uint32_t big = __ballot_sync(0xffffffffu, tx1 >= tx0 && !small);
            for (uint32_t bb = big; bb; bb &= bb - 1) {
                const int src = __ffs(bb) - 1;
                const int n = big_members<false>(
                    vp, __shfl_sync(0xffffffffu, r.X, src), __shfl_sync(0xffffffffu, r.Y, src),
                    __shfl_sync(0xffffffffu, r.R, src), __shfl_sync(0xffffffffu, tx0, src),
                    __shfl_sync(0xffffffffu, tx1, src), __shfl_sync(0xffffffffu, ty0, src),
                    __shfl_sync(0xffffffffu, ty1, src), 0, 0, 0, 0, nullptr, lane);
                if (lane == src) cnt = n;
            }
            int M = 0;
            const int off = block_excl_scan<int>(cnt, s_scan, &M);
            s_rec[tid] = make_float4(r.X, r.Y, r.R, code);
            float4 *lists = fr.lists + s_vbase[g];
            int *pids = fr.pids ? fr.pids + s_vbase[g] : nullptr;
            int *cur = s_cur + g * nt;
            for (int w0 = 0; w0 < M; w0 += kStableStage) {
                const int m = min(kStableStage, M - w0);
                // ---- 2. stage this window's pairs, in particle order
                if (mask) {
                    const int t00 = ty0 * vp.ntx + tx0;
                    int j = off - w0;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (!((mask >> q) & 1u)) continue;
                        if ((unsigned)j < (unsigned)m)
                            s_pair[j] = (uint32_t)(t00 + (q & 1) + ((q >> 1) ? vp.ntx : 0)) << kSlotBits | (uint32_t)tid;
                        ++j;
                    }
                }
                for (uint32_t bb = big; bb; bb &= bb - 1) {
                    const int src = __ffs(bb) - 1;
                    big_members<true>(vp, __shfl_sync(0xffffffffu, r.X, src), __shfl_sync(0xffffffffu, r.Y, src),
                                      __shfl_sync(0xffffffffu, r.R, src), __shfl_sync(0xffffffffu, tx0, src),
                                      __shfl_sync(0xffffffffu, tx1, src), __shfl_sync(0xffffffffu, ty0, src),
                                      __shfl_sync(0xffffffffu, ty1, src), __shfl_sync(0xffffffffu, off, src), w0, m,
                                      warp * 32 + src, s_pair, lane);
                }
                __syncthreads();
                // ---- 3. sort by tile, keeping particle order within a tile
                sort_pairs_pass(s_pair, s_alt, m, kSlotBits, s_cnt, s_scan);
                const uint32_t *sorted = s_alt;
                if (nt > kDigits) {
                    sort_pairs_pass(s_alt, s_pair, m, kSlotBits + kDigitBits, s_cnt, s_scan);
                    sorted = s_pair;
                }
                // ---- 4. records to their slots; a run's cursor is relative to its first place
                for (int j = tid; j < m; j += kThreads) {
                    const uint32_t t = sorted[j] >> kSlotBits;
                    if (j == 0 || sorted[j - 1] >> kSlotBits != t) cur[t] -= j;
                }
                __syncthreads();
                for (int j = tid; j < m; j += kThreads) {
                    const uint32_t p = sorted[j], sl = p & (kThreads - 1);
                    const int pos = cur[p >> kSlotBits] + j;
                    lists[pos] = s_rec[sl];
                    if (pids) pids[pos] = (int)(r0 + sl);
                }
                __syncthreads();
                for (int j = tid; j < m; j += kThreads) {
                    const uint32_t t = sorted[j] >> kSlotBits;
                    if (j + 1 == m || sorted[j + 1] >> kSlotBits != t) cur[t] += j + 1;
                }
                __syncthreads();
            }
        }
        cx = nx, cy = ny, cz = nz, ch = nh, ci = ni;
    }
}

template <int S> static cudaError_t scatter_stable_impl(const SceneDev &sc, const FrameDev &fr, cudaStream_t st) {
    const size_t smem = (size_t)fr.G * fr.n_tiles * sizeof(int) + kStableExtra;
    cudaError_t err = ensure_smem_limit((const void *)k_scatter_stable<S>, kBinSmemMax + kStableExtra);
    if (err != cudaSuccess) return err;
    return by_views(fr, kGridY * fr.G, [&](const FrameDev &part) {
        k_scatter_stable<S><<<dim3(part.n_chunks, (part.V + part.G - 1) / part.G), kThreads, smem, st>>>(sc, part);
    });
}

cudaError_t launch_scatter(int storage, const SceneDev &sc, const FrameDev &fr, bool stable, cudaStream_t st) {
    if (stable) {
        if (storage == 0) return scatter_stable_impl<0>(sc, fr, st);
        if (storage == 1) return scatter_stable_impl<1>(sc, fr, st);
        return scatter_stable_impl<2>(sc, fr, st);
    }
    if (storage == 0) return scatter_impl<0>(sc, fr, st);
    if (storage == 1) return scatter_impl<1>(sc, fr, st);
    return scatter_impl<2>(sc, fr, st);
}

// Resident CTAs per SM of the binning kernels with a histogram of `smem` bytes (the
// smaller of count and scatter, so both run their chunks in whole waves).
template <int S> static int bin_occupancy(size_t smem) {
    int a = 0, b = 0;
    if (ensure_smem_limit((const void *)k_count<S>, kBinSmemMax) != cudaSuccess ||
        ensure_smem_limit((const void *)k_scatter<S>, kBinSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_count<S>, kThreads, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_scatter<S>, kThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return std::max(1, std::min(a, b));
}

int bin_ctas_per_sm(int storage, size_t smem) {
    if (storage == 0) return bin_occupancy<0>(smem);
    if (storage == 1) return bin_occupancy<1>(smem);
    return bin_occupancy<2>(smem);
}

// ---------------------------------------------------------------------------------------
// Debug raster: X, Y, R, zc, colour (brightness x colormap of the stored normalised
// intensity), active, for one view.

template <int S>
__global__ void k_debug_raster(SceneDev sc, const ViewParams *__restrict__ view, float *out8) {
    const ViewParams vp = *view;
    constexpr int VEC = Store<S>::VEC;
    const int64_t n = sc.n;
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * VEC; i < n;
         i += (int64_t)gridDim.x * blockDim.x * VEC) {
        float x[VEC], y[VEC], z[VEC], h[VEC], it[VEC];
        Store<S>::load(sc.x, i, x);
        Store<S>::load(sc.y, i, y);
        Store<S>::load(sc.z, i, z);
        Store<S>::load(sc.h, i, h);
        Store<S>::load(sc.it, i, it);
        for (int k = 0; k < VEC; ++k) {
            const int64_t p = i + k;
            if (p >= n) break;
            Raster r;
            r.X = r.Y = r.R = 0.0f;
            const bool act = raster_one(vp, x[k], y[k], z[k], h[k], r);
            int t = 0;
            while (t + 1 < sc.n_types && p >= sc.type_begin[t + 1]) ++t;
            const int len = sc.lut_len[t];
            const float f = it[k] * (float)(len - 1);
            const int kk = min((int)floorf(f), len - 2);
            const float tau = f - (float)kk;
            const float4 c0 = sc.lut[sc.lut_off[t] + kk], c1 = sc.lut[sc.lut_off[t] + kk + 1];
            out8[0 * n + p] = r.X;
            out8[1 * n + p] = r.Y;
            out8[2 * n + p] = r.R;
            out8[3 * n + p] = r.zc;
            out8[4 * n + p] = (1.0f - tau) * c0.x + tau * c1.x;
            out8[5 * n + p] = (1.0f - tau) * c0.y + tau * c1.y;
            out8[6 * n + p] = (1.0f - tau) * c0.z + tau * c1.z;
            out8[7 * n + p] = act ? 1.0f : 0.0f;
        }
    }
}

cudaError_t launch_debug_raster(int storage, const SceneDev &sc, const ViewParams *view, float *out8,
                                cudaStream_t st) {
    if (sc.n <= 0) return cudaSuccess;
    int64_t blocks = (sc.n + 255 * 8) / (256 * 8) + 1;
    if (blocks > 4096) blocks = 4096;
    if (storage == 0) k_debug_raster<0><<<(int)blocks, 256, 0, st>>>(sc, view, out8);
    else if (storage == 1) k_debug_raster<1><<<(int)blocks, 256, 0, st>>>(sc, view, out8);
    else k_debug_raster<2><<<(int)blocks, 256, 0, st>>>(sc, view, out8);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Depth-ordered binning (one view), for the transfer with absorption different from
// emission, where every tile list must run from the farthest particle to the nearest.
//   k_depth_records  per particle: record {X, Y, R, code}, depth key (all ones when the
//                    particle is not active) and its index;
//   (stable radix sort of the depth keys with the indices: equal depths keep index order)
//   k_sorted_counts  in that order: the gathered record and the number of tiles it belongs
//                    to (plus a zero past the end, so the exclusive scan ends with the total);
//   (exclusive scan of the counts: each particle's first output slot)
//   k_expand         each particle's place in the depth order, at its slots, keyed by tile id;
//   (stable radix sort by tile id: each tile's records stay in depth order; its last pass
//   writes the records of the places)
// All three stream over the particles and are bound by the latency of their loads, so the next
// particle's loads are issued before the current one is worked on.
// 10 M particles, 20.7 M pairs (FP16 storage): k_depth_records 135 -> 72 us, k_sorted_counts
// 204 -> 168, k_expand 202 -> 117 (places instead of 16-byte records), the last pass of the sort
// by tile 317 -> 238 (the records of 10 M places instead of 20.7 M pairs).

// krange: {min, max} of the active particles' depth keys (atomicMin / atomicMax; the
// caller sets {all ones, 0} first), so that the sort covers only the bits they span.
template <int S>
__global__ void __launch_bounds__(256) k_depth_records(SceneDev sc, const ViewParams *__restrict__ views,
                                                       float4 *prec, uint32_t *dkey, uint32_t *pid,
                                                       uint32_t *krange) {
    __shared__ ViewParams s_v;
    __shared__ int64_t s_tb[kMaxTypes + 1];
    if (threadIdx.x == 0) s_v = views[0];
    for (int k = threadIdx.x; k <= sc.n_types; k += blockDim.x) s_tb[k] = sc.type_begin[k];
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int type = 0;
    uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
    typename Stored<S>::T nx{}, ny{}, nz{}, nh{}, ni{};
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < sc.n)
        nx = load_stored<S>(sc.x, i), ny = load_stored<S>(sc.y, i), nz = load_stored<S>(sc.z, i),
        nh = load_stored<S>(sc.h, i), ni = load_stored<S>(sc.it, i);
    for (; i < sc.n; i += stride) {
        const float x = value_of(nx), y = value_of(ny), z = value_of(nz), h = value_of(nh), it = value_of(ni);
        if (i + stride < sc.n)
            nx = load_stored<S>(sc.x, i + stride), ny = load_stored<S>(sc.y, i + stride),
            nz = load_stored<S>(sc.z, i + stride), nh = load_stored<S>(sc.h, i + stride),
            ni = load_stored<S>(sc.it, i + stride);
        while (type + 1 < sc.n_types && i >= s_tb[type + 1]) ++type;
        Raster r;
        const bool act = raster_one(s_v, x, y, z, h, r);
        prec[i] = make_float4(r.X, r.Y, r.R, sc.emit ? __uint_as_float((uint32_t)i) : record_code(type, it));
        const uint32_t k = act ? depth_key(r.zc) : kInactiveKey;
        dkey[i] = k;
        pid[i] = (uint32_t)i;
        if (act) kmin = min(kmin, k), kmax = max(kmax, k);
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if ((threadIdx.x & 31) == 0 && kmin <= kmax) {
        atomicMin(&krange[0], kmin);
        atomicMax(&krange[1], kmax);
    }
}

// Candidate tiles of a rasterised particle (up to 2 x 2 are tested by one lane, more by the whole
// warp).
__device__ __forceinline__ void tile_box(const ViewParams &v, float X, float Y, float R, int &tx0, int &tx1,
                                         int &ty0, int &ty1) {
    int i0, i1, j0, j1;
    pixel_box(v, X, Y, R, i0, i1, j0, j1);
    tx0 = tile_of(v, i0), tx1 = tile_of(v, i1), ty0 = tile_of(v, j0), ty1 = tile_of(v, j1);
}

__global__ void __launch_bounds__(256) k_sorted_counts(const ViewParams *__restrict__ views,
                                                       const float4 *__restrict__ prec,
                                                       const uint32_t *__restrict__ skey,
                                                       const uint32_t *__restrict__ spid, int64_t n,
                                                       uint32_t inactive, float4 *srec, uint32_t *cnt,
                                                       uint32_t *arrivals) {
    __shared__ ViewParams s_v;
    if (threadIdx.x == 0) s_v = views[0];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t wstride = (int64_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) cnt[n] = 0, *arrivals = 0;
    const int64_t base0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
    // ahead: the next particle's record, and the key and index of the one after it
    float4 nrec = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    bool nact = false;
    uint32_t key = inactive, pid = 0;
    if (base0 + lane < n) {
        nact = skey[base0 + lane] != inactive;
        if (nact) nrec = prec[spid[base0 + lane]];
    }
    if (base0 + lane + wstride < n) key = skey[base0 + lane + wstride], pid = spid[base0 + lane + wstride];
    for (int64_t base = base0; base < n; base += wstride) {
        const int64_t q = base + lane;
        const float4 rec = nrec;
        const bool act = nact;
        nrec = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        nact = key != inactive;
        if (nact) nrec = prec[pid];
        key = inactive;
        if (q + 2 * wstride < n) key = skey[q + 2 * wstride], pid = spid[q + 2 * wstride];
        int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
        if (act) tile_box(s_v, rec.x, rec.y, rec.z, tx0, tx1, ty0, ty1);
        const bool small = tx1 >= tx0 && tx1 - tx0 <= 1 && ty1 - ty0 <= 1;
        uint32_t c = 0;
        if (small) c = __popc(tile_mask2(s_v, rec.x, rec.y, rec.z, tx0, tx1, ty0, ty1));
        uint32_t big = __ballot_sync(0xffffffffu, tx1 >= tx0 && !small);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const float bX = __shfl_sync(0xffffffffu, rec.x, src), bY = __shfl_sync(0xffffffffu, rec.y, src);
            const float bR = __shfl_sync(0xffffffffu, rec.z, src);
            const int bx0 = __shfl_sync(0xffffffffu, tx0, src), bx1 = __shfl_sync(0xffffffffu, tx1, src);
            const int by0 = __shfl_sync(0xffffffffu, ty0, src), by1 = __shfl_sync(0xffffffffu, ty1, src);
            uint32_t mine = 0;
            for (int ty = by0 + (lane >> 3); ty <= by1; ty += 4)
                for (int tx = bx0 + (lane & 7); tx <= bx1; tx += 8)
                    mine += tile_member(s_v, bX, bY, bR, tx, ty) ? 1u : 0u;
            const uint32_t tot = __reduce_add_sync(0xffffffffu, mine);
            if (lane == src) c = tot;
        }
        if (q < n) {
            srec[q] = rec;
            cnt[q] = c;
        }
    }
}

__global__ void __launch_bounds__(256) k_expand(const ViewParams *__restrict__ views,
                                                const float4 *__restrict__ srec, const uint32_t *__restrict__ poff,
                                                const uint32_t *__restrict__ sums, int64_t n, int64_t P,
                                                uint32_t *__restrict__ tkey, uint32_t *__restrict__ tval,
                                                int *status) {
    __shared__ ViewParams s_v;
    if (threadIdx.x == 0) s_v = views[0];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t wstride = (int64_t)gridDim.x * blockDim.x;
    const int64_t base0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
    float4 nrec = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    uint32_t n0 = 0, n1 = 0;  // first slot of the next particle and of the one after it
    auto ahead = [&](int64_t q) {
        n0 = n1 = 0;
        if (q < n) {
            nrec = srec[q];
            n0 = poff[q] + sums[q / kScanChunk];
            n1 = poff[q + 1] + sums[(q + 1) / kScanChunk];
        }
    };
    // every slot of the P has to be written: the counts add up to them
    if (blockIdx.x == 0 && threadIdx.x == 0 && (int64_t)poff[n] + sums[n / kScanChunk] != P)
        atomicExch(&status[kStatOverflow], 1);
    ahead(base0 + lane);
    for (int64_t base = base0; base < n; base += wstride) {
        const int64_t q = base + lane;
        const float4 rec = nrec;
        const uint32_t o0 = n0, c = n1 - n0;
        ahead(q + wstride);
        int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
        if (c) tile_box(s_v, rec.x, rec.y, rec.z, tx0, tx1, ty0, ty1);
        const bool small = c && tx1 >= tx0 && tx1 - tx0 <= 1 && ty1 - ty0 <= 1;
        if (c && (tx1 < tx0 || ty1 < ty0)) atomicExch(&status[kStatOverflow], 1);
        if (small) {
            const uint32_t m = tile_mask2(s_v, rec.x, rec.y, rec.z, tx0, tx1, ty0, ty1);
            const uint32_t t00 = (uint32_t)(ty0 * s_v.ntx + tx0);
            uint32_t pos = o0;
            if ((uint32_t)__popc(m) != c || (int64_t)o0 + c > P) {
                atomicExch(&status[kStatOverflow], 1);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (m & (1u << k)) {
                        tkey[pos] = t00 + (k & 1 ? 1u : 0u) + (k & 2 ? (uint32_t)s_v.ntx : 0u);
                        tval[pos++] = (uint32_t)q;
                    }
            }
        }
        uint32_t big = __ballot_sync(0xffffffffu, c && tx1 >= tx0 && !small);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const float bX = __shfl_sync(0xffffffffu, rec.x, src), bY = __shfl_sync(0xffffffffu, rec.y, src);
            const float bR = __shfl_sync(0xffffffffu, rec.z, src);
            const uint32_t bo = __shfl_sync(0xffffffffu, o0, src), bc = __shfl_sync(0xffffffffu, c, src);
            const int bx0 = __shfl_sync(0xffffffffu, tx0, src), bx1 = __shfl_sync(0xffffffffu, tx1, src);
            const int by0 = __shfl_sync(0xffffffffu, ty0, src), by1 = __shfl_sync(0xffffffffu, ty1, src);
            uint32_t k = 0;
            // blocks of 8 x 4 candidates, one per lane
            for (int y = by0; y <= by1; y += 4)
                for (int x = bx0; x <= bx1; x += 8) {
                    const int tx = x + (lane & 7), ty = y + (lane >> 3);
                    const bool m = tx <= bx1 && ty <= by1 && tile_member(s_v, bX, bY, bR, tx, ty);
                    const uint32_t bal = __ballot_sync(0xffffffffu, m);
                    if (m) {
                        const uint32_t kk = k + (uint32_t)__popc(bal & lt);
                        const uint32_t pos = bo + kk;
                        if (kk >= bc || (int64_t)pos >= P) {
                            atomicExch(&status[kStatOverflow], 1);
                        } else {
                            tkey[pos] = (uint32_t)(ty * s_v.ntx + tx);
                            tval[pos] = (uint32_t)(base + src);
                        }
                    }
                    k += (uint32_t)__popc(bal);
                }
            if (lane == 0 && k != bc) atomicExch(&status[kStatOverflow], 1);
        }
    }
}

static int stream_grid(int64_t n, int threads) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * (2048 / threads)));
}

cudaError_t launch_depth_records(int storage, const SceneDev &sc, const ViewParams *views, float4 *prec,
                                 uint32_t *dkey, uint32_t *pid, uint32_t *krange, cudaStream_t st) {
    if (sc.n <= 0) return cudaSuccess;
    const int g = stream_grid(sc.n, 256);
    if (storage == 0) k_depth_records<0><<<g, 256, 0, st>>>(sc, views, prec, dkey, pid, krange);
    else if (storage == 1) k_depth_records<1><<<g, 256, 0, st>>>(sc, views, prec, dkey, pid, krange);
    else k_depth_records<2><<<g, 256, 0, st>>>(sc, views, prec, dkey, pid, krange);
    return cudaGetLastError();
}

cudaError_t launch_sorted_counts(const ViewParams *views, const float4 *prec, const uint32_t *skey,
                                 const uint32_t *spid, int64_t n, uint32_t inactive, float4 *srec, uint32_t *cnt,
                                 uint32_t *arrivals, cudaStream_t st) {
    k_sorted_counts<<<stream_grid(std::max<int64_t>(1, n), 256), 256, 0, st>>>(views, prec, skey, spid, n, inactive,
                                                                               srec, cnt, arrivals);
    return cudaGetLastError();
}

cudaError_t launch_expand(const ViewParams *views, const float4 *srec, const uint32_t *poff, const uint32_t *sums,
                          int64_t n, int64_t P, uint32_t *tkey, uint32_t *tval, int *status, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_expand<<<stream_grid(n, 256), 256, 0, st>>>(views, srec, poff, sums, n, P, tkey, tval, status);
    return cudaGetLastError();
}

}  // namespace spl
