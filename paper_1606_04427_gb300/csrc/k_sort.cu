// Stable LSD radix sort of (32- or 64-bit key, 32-bit value) pairs on the device.
//
// The depth-ordered render (Section 2.1: with absorption different from emission the
// transfer equation must be applied along each line of sight in order) needs every tile
// list in depth order.  It sorts the particles by a 32-bit depth key, from index order (so
// equal depths keep it), and then their (tile, place in depth order) pairs by tile: each pass
// is stable, so the lists are tile-major and far to near.
//
// One pass over 8 key bits:
//   k_digit_hist   each CTA counts the digits of its 4096 elements (shared counters per warp),
//                  written digit-major: hist[digit * n_blocks + block];
//   k_scan_chunks  exclusive scan of hist within chunks of 4096 entries; the last CTA to finish
//                  scans the chunks' totals.  hist[d * n_blocks + b] plus its chunk's total is
//                  where block b's elements of digit d start in the output;
//   k_digit_scatter each CTA re-reads its elements and writes them to their slots: an
//                  element's rank among equal digits follows input order (warps own
//                  consecutive ranges, lanes rank in order), so every pass is stable.
// The element loops are bound by latency: a thread's 8 keys are loaded before any is used, and the
// values while the keys are written (loaded one by one between the barriers of the ranking, a pass
// over 10 to 21 M pairs took 57 + 108 us in k_digit_hist and k_digit_scatter; now 19 + 90).  CTAs of
// 512 threads: with 16 elements per thread in registers only two CTAs of 256 fit on an SM
// (k_digit_scatter 132 us).
#include "splotch_internal.cuh"

namespace spl {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortPerWarp = 256;                       // consecutive elements per warp
constexpr int kSortTile = kSortWarps * kSortPerWarp;    // elements per CTA
constexpr int kSortRounds = kSortPerWarp / 32;

template <typename K> __device__ __forceinline__ uint32_t digit_of(K k, int shift) {
    return (uint32_t)(k >> shift) & 255u;
}

// Key as the first pass of a sort reads it: 32-bit keys up to base + span relative to base, the
// all-ones key just past them.  KeyRange{} changes nothing.
__device__ __forceinline__ uint64_t rebased(uint64_t k, KeyRange) { return k; }
__device__ __forceinline__ uint32_t rebased(uint32_t k, KeyRange r) { return k == 0xFFFFFFFFu ? r.span + 1u : k - r.base; }

template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_digit_hist(const K *__restrict__ keys, int64_t n, int shift,
                                                            KeyRange range, int n_blocks, uint32_t *hist,
                                                            uint32_t *arrivals) {
    __shared__ uint32_t s_cnt[kSortWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) *arrivals = 0;
    for (int k = threadIdx.x; k < kSortWarps * 256; k += kSortThreads) (&s_cnt[0][0])[k] = 0;
    const int64_t base = (int64_t)blockIdx.x * kSortTile + (int64_t)warp * kSortPerWarp + lane;
    K key[kSortRounds];
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) key[r] = keys[min(base + r * 32, n - 1)];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r)
        if (base + r * 32 < n) atomicAdd(&s_cnt[warp][digit_of(rebased(key[r], range), shift)], 1u);
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t sum = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) sum += s_cnt[w][threadIdx.x];
        hist[(int64_t)threadIdx.x * n_blocks + blockIdx.x] = sum;
    }
}

// Exclusive scan: every chunk by a CTA, the chunks' totals by the last CTA that finishes.
__device__ __forceinline__ uint32_t warp_scan_incl_u(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Exclusive scan of one value per thread over a 1024-thread CTA; *total gets the sum.
__device__ uint32_t block_scan_excl_u(uint32_t v, uint32_t *s_warp, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t incl = warp_scan_incl_u(v);
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0u;
        const uint32_t wi = warp_scan_incl_u(w);
        s_warp[lane] = wi - w;
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    const uint32_t res = s_warp[warp] + incl - v;
    *total = s_warp[32];
    __syncthreads();
    return res;
}

// *arrivals is 0 before and the number of CTAs after.
__global__ void __launch_bounds__(1024) k_scan_chunks(uint32_t *a, int64_t n, uint32_t *sums, uint32_t *arrivals) {
    __shared__ uint32_t s_warp[33];
    __shared__ bool s_last;
    const int64_t c0 = (int64_t)blockIdx.x * kScanChunk;
    uint32_t v[kScanChunk / 1024];
    uint32_t local = 0;
#pragma unroll
    for (int q = 0; q < kScanChunk / 1024; ++q) {
        const int64_t i = c0 + (int64_t)threadIdx.x * (kScanChunk / 1024) + q;
        v[q] = i < n ? a[i] : 0u;
        local += v[q];
    }
    uint32_t total;
    uint32_t run = block_scan_excl_u(local, s_warp, &total);
#pragma unroll
    for (int q = 0; q < kScanChunk / 1024; ++q) {
        const int64_t i = c0 + (int64_t)threadIdx.x * (kScanChunk / 1024) + q;
        if (i < n) a[i] = run;
        run += v[q];
    }
    if (threadIdx.x == 0) {
        sums[blockIdx.x] = total;
        __threadfence();
        s_last = atomicAdd(arrivals, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    uint32_t carry = 0;
    for (int b = 0; b < (int)gridDim.x; b += 1024) {
        const int i = b + threadIdx.x;
        const uint32_t w = i < (int)gridDim.x ? __ldcg(&sums[i]) : 0u;
        const uint32_t ex = block_scan_excl_u(w, s_warp, &total);
        if (i < (int)gridDim.x) sums[i] = carry + ex;
        carry += total;
    }
}

// kGather: the last pass of a sort whose values index a payload: instead of the keys and
// values, write payload[value] to each element's slot (payload_out).  A value past payload_last
// reads that one.
template <typename K, bool kGather>
__global__ void __launch_bounds__(kSortThreads, 3) k_digit_scatter(const K *__restrict__ keys,
                                                               const uint32_t *__restrict__ vals, int64_t n,
                                                               int shift, KeyRange range, int n_blocks,
                                                               const uint32_t *__restrict__ offs,
                                                               const uint32_t *__restrict__ sums,
                                                               K *__restrict__ keys_out,
                                                               uint32_t *__restrict__ vals_out,
                                                               const float4 *__restrict__ payload,
                                                               uint32_t payload_last,
                                                               float4 *__restrict__ payload_out) {
    __shared__ uint32_t s_wc[kSortWarps][256];  // per warp: running count, then warp base
    __shared__ uint32_t s_off[256];             // output start of this CTA's digit d
    __shared__ uint32_t s_loc[256];             // start of digit d in the CTA's staged tile
    __shared__ uint32_t s_scan[33];
    __shared__ __align__(16) K s_key[kSortTile];  // staged keys, then staged values
    __shared__ uint8_t s_dig[kSortTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < kSortWarps * 256; k += kSortThreads) (&s_wc[0][0])[k] = 0;
    const int64_t tile0 = (int64_t)blockIdx.x * kSortTile;
    const int cnt = (int)min((int64_t)kSortTile, n - tile0);
    const int64_t base = tile0 + (int64_t)warp * kSortPerWarp;
    K k_r[kSortRounds];
    uint32_t rank[kSortRounds];
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) k_r[r] = rebased(keys[min(base + r * 32 + lane, n - 1)], range);
    if (threadIdx.x < 256) {
        const int64_t at = (int64_t)threadIdx.x * n_blocks + blockIdx.x;
        s_off[threadIdx.x] = offs[at] + sums[at / kScanChunk];
    }
    __syncthreads();
    // rank of each element among the equal digits of its warp's range, in input order
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        const int64_t i = base + r * 32 + lane;
        const bool ok = i < n;
        const uint32_t d = ok ? digit_of(k_r[r], shift) : 256u;
        const uint32_t peers = warp_peers<9>(d);  // digits 0..255, 256 past the end
        const int leader = __ffs(peers) - 1;
        uint32_t before = 0;
        if (ok && lane == leader) {
            before = s_wc[warp][d];
            s_wc[warp][d] = before + (uint32_t)__popc(peers);
        }
        before = __shfl_sync(0xffffffffu, before, leader);
        rank[r] = before + (uint32_t)__popc(peers & lt);
        __syncwarp();  // this round's counter updates before the next round reads them
    }
    __syncthreads();
    // warp bases (elements of earlier warps with the same digit come first), the CTA's
    // digit totals, and their exclusive scan: where each digit starts in the staged tile
    {
        const int d = threadIdx.x & 255;  // a digit per thread, by the first 256
        uint32_t run = 0;
        if (threadIdx.x < 256)
            for (int w = 0; w < kSortWarps; ++w) {
                const uint32_t c = s_wc[w][d];
                s_wc[w][d] = run;
                run += c;
            }
        const uint32_t incl = warp_scan_incl_u(run);
        if (lane == 31) s_scan[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const uint32_t wv = lane < 8 ? s_scan[lane] : 0u;
            const uint32_t wi = warp_scan_incl_u(wv);
            if (lane < 8) s_scan[lane] = wi - wv;
        }
        __syncthreads();
        if (threadIdx.x < 256) s_loc[d] = s_scan[warp] + incl - run;
    }
    __syncthreads();
    // stage the keys in digit order, then write each digit's run to consecutive slots
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        const int64_t i = base + r * 32 + lane;
        if (i >= n) continue;
        const uint32_t d = digit_of(k_r[r], shift);
        rank[r] += s_loc[d] + s_wc[warp][d];  // now the place in the staged tile
        if (!kGather) s_key[rank[r]] = k_r[r];
        s_dig[rank[r]] = (uint8_t)d;
    }
    // the values are on their way while the keys are written
    uint32_t v_r[kSortRounds];
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) v_r[r] = vals[min(base + r * 32 + lane, n - 1)];
    __syncthreads();
    if (!kGather) {
#pragma unroll 4
        for (int l = threadIdx.x; l < cnt; l += kSortThreads) {
            const uint32_t d = s_dig[l];
            keys_out[s_off[d] + (uint32_t)l - s_loc[d]] = s_key[l];
        }
    }
    __syncthreads();
    uint32_t *s_val = reinterpret_cast<uint32_t *>(s_key);
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        const int64_t i = base + r * 32 + lane;
        if (i < n) s_val[rank[r]] = v_r[r];
    }
    __syncthreads();
#pragma unroll 4
    for (int l = threadIdx.x; l < cnt; l += kSortThreads) {
        const uint32_t d = s_dig[l];
        const uint32_t g = s_off[d] + (uint32_t)l - s_loc[d];
        if (kGather)
            payload_out[g] = payload[min(s_val[l], payload_last)];
        else
            vals_out[g] = s_val[l];
    }
}

static int sort_blocks(int64_t n) { return (int)((n + kSortTile - 1) / kSortTile); }

size_t sort_temp_bytes(int64_t n) {
    const int64_t h = (int64_t)256 * std::max(1, sort_blocks(n));
    const int64_t chunks = (h + kScanChunk - 1) / kScanChunk;
    return sizeof(uint32_t) * (size_t)(h + chunks) + 256;
}

// Sorts keys[0, n) with their values by key bits [bit_lo, bit_hi), stably, ping-ponging
// with the alternate buffers; *in_alt tells which pair of buffers holds the result.
template <typename K>
static cudaError_t sort_impl(K *keys, K *keys_alt, uint32_t *vals, uint32_t *vals_alt, int64_t n, int bit_lo,
                             int bit_hi, void *temp, cudaStream_t st, bool *in_alt, KeyRange range,
                             const float4 *payload = nullptr, uint32_t payload_last = 0,
                             float4 *payload_out = nullptr) {
    *in_alt = false;
    if (n <= 1 || bit_lo >= bit_hi) {
        if (payload && n > 0) return launch_gather_records(payload, vals, payload_last, n, payload_out, st);
        return cudaSuccess;
    }
    const int nb = sort_blocks(n);
    const int64_t h = (int64_t)256 * nb;
    const int chunks = (int)((h + kScanChunk - 1) / kScanChunk);
    uint32_t *hist = (uint32_t *)temp;
    uint32_t *sums = hist + h, *arrivals = sums + chunks;
    K *ka = keys, *kb = keys_alt;
    uint32_t *va = vals, *vb = vals_alt;
    for (int shift = bit_lo; shift < bit_hi; shift += 8) {
        k_digit_hist<K><<<nb, kSortThreads, 0, st>>>(ka, n, shift, range, nb, hist, arrivals);
        k_scan_chunks<<<chunks, 1024, 0, st>>>(hist, h, sums, arrivals);
        if (payload && shift + 8 >= bit_hi)
            k_digit_scatter<K, true><<<nb, kSortThreads, 0, st>>>(ka, va, n, shift, range, nb, hist, sums, kb, vb,
                                                                 payload, payload_last, payload_out);
        else
            k_digit_scatter<K, false><<<nb, kSortThreads, 0, st>>>(ka, va, n, shift, range, nb, hist, sums, kb, vb,
                                                                  nullptr, 0, nullptr);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        range = KeyRange{};
        std::swap(ka, kb);
        std::swap(va, vb);
        *in_alt = !*in_alt;
    }
    return cudaSuccess;
}

cudaError_t radix_sort_pairs(uint64_t *keys, uint64_t *keys_alt, uint32_t *vals, uint32_t *vals_alt, int64_t n,
                             int bit_lo, int bit_hi, void *temp, cudaStream_t st, bool *in_alt) {
    return sort_impl<uint64_t>(keys, keys_alt, vals, vals_alt, n, bit_lo, bit_hi, temp, st, in_alt, KeyRange{});
}

cudaError_t radix_sort_pairs(uint32_t *keys, uint32_t *keys_alt, uint32_t *vals, uint32_t *vals_alt, int64_t n,
                             int bit_lo, int bit_hi, void *temp, cudaStream_t st, bool *in_alt, KeyRange range) {
    return sort_impl<uint32_t>(keys, keys_alt, vals, vals_alt, n, bit_lo, bit_hi, temp, st, in_alt, range);
}

cudaError_t radix_sort_gather(uint32_t *keys, uint32_t *keys_alt, uint32_t *vals, uint32_t *vals_alt, int64_t n,
                              int bit_lo, int bit_hi, void *temp, const float4 *payload, int64_t payload_n,
                              float4 *payload_out, cudaStream_t st) {
    bool alt = false;
    return sort_impl<uint32_t>(keys, keys_alt, vals, vals_alt, n, bit_lo, bit_hi, temp, st, &alt, KeyRange{},
                               payload, (uint32_t)(payload_n - 1), payload_out);
}

size_t scan_temp_bytes(int64_t n) {
    return sizeof(uint32_t) * (size_t)((std::max<int64_t>(1, n) + kScanChunk - 1) / kScanChunk) + 256;
}

uint32_t *scan_arrivals(int64_t n, void *temp) {
    return (uint32_t *)temp + (std::max<int64_t>(1, n) + kScanChunk - 1) / kScanChunk;
}

// Exclusive scan of a[0, n) in two parts (the total must stay below 2^32): entry i of the scan is
// a[i] + temp[i / kScanChunk].  *scan_arrivals must be 0.
cudaError_t exclusive_scan_u32(uint32_t *a, int64_t n, void *temp, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int chunks = (int)((n + kScanChunk - 1) / kScanChunk);
    k_scan_chunks<<<chunks, 1024, 0, st>>>(a, n, (uint32_t *)temp, scan_arrivals(n, temp));
    return cudaGetLastError();
}

}  // namespace spl
