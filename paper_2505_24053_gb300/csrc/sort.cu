// sort.cu -- SortByKeys (Algorithm 1): stable LSD radix sort of u32 keys with
// u32 values, 8-bit digits, two kernels per digit and no device-side waits:
//
//   k_radix_hist     per sort tile (ITEMS x 256 keys): the 256-bin digit
//                    histogram, stored per tile and summed into its group of
//                    32 tiles. The last block to finish (an atomic
//                    counter after a memory fence; nothing waits) scans the
//                    group sums down the tiles per digit and the digit totals
//                    (the digit bases);
//   k_radix_scatter  per sort tile: stable warp-level ranking (peer masks from a
//                    vote per bit of the digit), the tile's offset per
//                    digit = digit base + group prefix + sum over the earlier
//                    tiles of its group, reordering by digit in shared memory and
//                    contiguous writes of each digit run.
//
// Tiles hold 3072 keys. The key count stays on the device. The histogram's blocks go
// through the tiles, each with the next tile's keys in flight: bound by the latency of
// a tile's loads, votes and sums, and a block and a fence per tile took 48 us where
// these take 23 (12M keys; 16 -> 14 us at 3.4M). The scatter launches a block per tile
// of the workspace capacity and the blocks past the count exit at once.
#include <algorithm>

#include "geer_internal.cuh"

namespace geer {
namespace {

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ uint32_t key_count(const uint32_t *misc, int count_slot, int check_capacity) {
    if (check_capacity && (misc[kMiscStatus] & kStatusCapacity)) return 0u;
    return misc[count_slot];
}

// dev_buf: the pass's input buffer is chosen on the device (kin0 or kin1): the
// one the previous pass wrote, or read, if that pass was skipped (its digit the
// same for every key). Otherwise kin0 is the input.
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *__restrict__ kin0,
                                                             const uint32_t *__restrict__ kin1, int dev_buf,
                                                             uint32_t *__restrict__ misc, int count_slot,
                                                             int check_capacity, int shift,
                                                             uint32_t *__restrict__ tile_hist,
                                                             uint32_t *__restrict__ group_sum,
                                                             uint32_t *__restrict__ group_excl,
                                                             uint32_t *__restrict__ digit_base) {
    grid_dep_sync();
    constexpr int W = kSortThreads / 32, TILE = kSortThreads * ITEMS, GROUP = kGroupTiles;
    __shared__ uint32_t s_h[2][kRadix];  // this tile's counts and, being cleared, the next one's
    __shared__ uint32_t s_wsum[W];
    __shared__ bool s_is_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = key_count(misc, count_slot, check_capacity);
    const uint32_t ntiles = (uint32_t)(((uint64_t)n + TILE - 1) / TILE);
    if (blockIdx.x >= ntiles) return;
    // read before the last block of this pass updates them (it finishes after every block started)
    const int in = dev_buf ? depth_sorted_buf(misc) : 0;
    const uint32_t *__restrict__ kin = in ? kin1 : kin0;
    uint32_t key[ITEMS];
    const auto load = [&](uint32_t tile) {
        const uint64_t t0 = (uint64_t)tile * TILE;
        const uint32_t nt = tile < ntiles ? (uint32_t)min((uint64_t)TILE, (uint64_t)n - t0) : 0u;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) key[k] = (uint32_t)(k * kSortThreads + tid) < nt ? kin[t0 + k * kSortThreads + tid] : 0u;
        return nt;
    };
    uint32_t nt = load(blockIdx.x);
    s_h[0][tid] = 0u;
    __syncthreads();
    int b = 0;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, b ^= 1) {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k)
            if ((uint32_t)(k * kSortThreads + tid) < nt) atomicAdd(&s_h[b][(key[k] >> shift) & 0xffu], 1u);
        nt = load(tile + gridDim.x);  // the next tile's keys, in flight meanwhile
        s_h[b ^ 1][tid] = 0u;
        __syncthreads();
        const uint32_t c = s_h[b][tid];
        tile_hist[(uint64_t)tile * kRadix + tid] = c;
        if (c) atomicAdd(&group_sum[(uint64_t)(tile / GROUP) * kRadix + tid], c);
    }

    // the last block to finish scans the group sums (threadFenceReduction pattern)
    __threadfence();
    __syncthreads();
    if (tid == 0) s_is_last = atomicAdd(&misc[kMiscSortDone], 1u) == min(ntiles, gridDim.x) - 1u;
    __syncthreads();
    if (!s_is_last) return;
    __threadfence();
    const int d = tid;  // one digit per thread
    const uint32_t ngroups = (ntiles + GROUP - 1) / GROUP;
    uint32_t run = 0;
    for (uint32_t g = 0; g < ngroups; g += 16) {
        uint32_t v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = g + u < ngroups ? __ldcg(&group_sum[(uint64_t)(g + u) * kRadix + d]) : 0u;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            if (g + u < ngroups) {
                group_excl[(uint64_t)(g + u) * kRadix + d] = run;
                group_sum[(uint64_t)(g + u) * kRadix + d] = 0u;  // zero for the next pass
            }
            run += v[u];
        }
    }
    // digit bases: exclusive scan of the digit totals over the 256 digits
    uint32_t v = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) s_wsum[warp] = v;
    __syncthreads();
    uint32_t pre = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) pre += w < warp ? s_wsum[w] : 0u;
    digit_base[d] = pre + v - run;
    // one digit holds every key: the pass keeps the order (its scatter copies, or
    // with dev_buf is skipped, the data staying in its input buffer)
    const bool all = __syncthreads_or(run == n);
    if (tid == 0) {
        misc[kMiscSortSame] = all ? 1u : 0u;
        if (dev_buf) misc[kMiscSortCur] = (uint32_t)in;
        misc[kMiscSortDone] = 0u;
    }
}

// With W > 0 every key also carries W 32-bit words (min_ -> mout_, W per key: the
// super-tile sort's tile masks), reordered through the values' shared buffer after
// the values have left it.
// Bound by the latency of shared memory in the ranking, so by the blocks resident per
// SM: with the values loaded after the ranking and no shared lane masks (atomics and
// reads of a mask per digit before) 64 registers hold without values to carry or with
// one word, 48 with two. 12M keys with two words: 167 -> 137 us; 3.4M without: 40 -> 36.
template <int ITEMS, int W>
__global__ void __launch_bounds__(kSortThreads, W == 2 ? 5 : 4) k_radix_scatter(
    const uint32_t *__restrict__ kin_, const uint32_t *__restrict__ vin_, uint32_t *__restrict__ kout_,
    uint32_t *__restrict__ vout_, int dev_buf, const uint32_t *__restrict__ misc, int count_slot,
    int check_capacity, int shift, const uint32_t *__restrict__ tile_hist, const uint32_t *__restrict__ group_excl,
    const uint32_t *__restrict__ digit_base, const uint32_t *__restrict__ min_, uint32_t *__restrict__ mout_) {
    grid_dep_sync();
    // dev_buf: (kin_, vin_) is buffer 0 and (kout_, vout_) buffer 1; the input is
    // the one the histogram kernel recorded, and an identity pass is skipped
    if (dev_buf && misc[kMiscSortSame]) return;
    const bool swap = dev_buf && misc[kMiscSortCur];
    const uint32_t *__restrict__ kin = swap ? kout_ : kin_;
    const uint32_t *__restrict__ vin = swap ? vout_ : vin_;
    uint32_t *__restrict__ kout = swap ? const_cast<uint32_t *>(kin_) : kout_;
    uint32_t *__restrict__ vout = swap ? const_cast<uint32_t *>(vin_) : vout_;
    constexpr int NW = kSortThreads / 32, TILE = kSortThreads * ITEMS, GROUP = kGroupTiles;
    __shared__ uint32_t s_whist[NW][kRadix];
    __shared__ uint32_t s_lbase[kRadix];  // start of each digit inside the tile
    __shared__ uint32_t s_out[kRadix];    // global position of the tile's first key of each digit
    __shared__ uint32_t s_wsum[NW];
    __shared__ uint32_t s_key[TILE];
    __shared__ uint32_t s_val[TILE];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = key_count(misc, count_slot, check_capacity);
    const uint32_t tile = blockIdx.x;
    if ((uint64_t)tile * TILE >= n) return;
    const uint64_t t0 = (uint64_t)tile * TILE;
    const uint32_t nt = (uint32_t)min((uint64_t)TILE, (uint64_t)n - t0);  // keys of the tile
    if (misc[kMiscSortSame]) {  // identity pass: coalesced copy of the tile
        for (uint32_t i = tid; i < nt; i += kSortThreads) {
            kout[t0 + i] = kin[t0 + i];
            vout[t0 + i] = vin[t0 + i];
        }
        if (W > 0)
            for (uint32_t i = tid; i < nt * W; i += kSortThreads) mout_[t0 * W + i] = min_[t0 * W + i];
        return;
    }
    const uint32_t base_d = digit_base[tid];
    for (int i = tid; i < NW * kRadix; i += kSortThreads) (&s_whist[0][0])[i] = 0u;
    // this tile's global offset for digit tid
    const uint32_t g0 = (tile / GROUP) * GROUP;
    uint32_t off = base_d + group_excl[(uint64_t)(tile / GROUP) * kRadix + tid];
    static_assert(GROUP % 16 == 0, "the group's tiles in steps of 16");
#pragma unroll 1
    for (uint32_t r0 = g0; r0 < tile; r0 += 16) {
        uint32_t part[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) part[r] = r0 + r < tile ? tile_hist[(uint64_t)(r0 + r) * kRadix + tid] : 0u;
#pragma unroll
        for (int r = 0; r < 16; ++r) off += part[r];
    }
    s_out[tid] = off;
    __syncthreads();

    uint32_t key[ITEMS], val[ITEMS], rank[ITEMS];
    const uint32_t base = (uint32_t)(warp * 32 * ITEMS + lane);  // in the tile
    kin += t0;
    vin += t0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) key[k] = base + k * 32 < nt ? kin[base + k * 32] : 0u;
    // stable ranking: warp by warp, item k by item k, lane by lane. The lanes sharing a
    // digit find each other by a vote per bit of the digit, and all read its count so far.
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const bool v = base + k * 32 < nt;
        const uint32_t d = (key[k] >> shift) & 0xffu;
        uint32_t peers = __ballot_sync(0xffffffffu, v);
#pragma unroll
        for (int b = 0; b < kRadixBits; ++b) {
            const bool bit = (d >> b) & 1u;
            const uint32_t m = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? m : ~m;
        }
        const uint32_t b = s_whist[warp][d];
        const uint32_t before = (uint32_t)__popc(peers & lanemask_lt());
        __syncwarp();
        if (v && before == 0) s_whist[warp][d] = b + (uint32_t)__popc(peers);
        rank[k] = v ? b + before : 0xffffffffu;
        __syncwarp();
    }
    // the values, needed from here on only (held through the ranking they cost a block per SM)
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) val[k] = base + k * 32 < nt ? vin[base + k * 32] : 0u;
    __syncthreads();
    // warp offsets inside the tile per digit, tile count per digit
    uint32_t cnt = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const uint32_t c = s_whist[w][tid];
        s_whist[w][tid] = cnt;
        cnt += c;
    }
    // exclusive scan of the counts over the digits: start of each digit in the tile
    uint32_t v = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) s_wsum[warp] = v;
    __syncthreads();
    uint32_t pre = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) pre += w < warp ? s_wsum[w] : 0u;
    s_lbase[tid] = pre + v - cnt;
    __syncthreads();
    // reorder the tile by digit in shared memory
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        if (rank[k] != 0xffffffffu) {
            const uint32_t d = (key[k] >> shift) & 0xffu;
            const uint32_t lp = s_lbase[d] + s_whist[warp][d] + rank[k];
            s_key[lp] = key[k];
            s_val[lp] = val[k];
            if (W > 0) rank[k] = lp;
        }
    }
    __syncthreads();
    // contiguous writes of each digit run
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const uint32_t lp = (uint32_t)(k * kSortThreads + tid);
        if (lp < nt) {
            const uint32_t kk = s_key[lp];
            const uint32_t d = (kk >> shift) & 0xffu;
            const uint32_t pos = s_out[d] + (lp - s_lbase[d]);
            if (pos < n) {
                kout[pos] = kk;
                vout[pos] = s_val[lp];
            }
        }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint32_t m[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) m[k] = base + k * 32 < nt ? min_[(t0 + base + k * 32) * W + w] : 0u;
        __syncthreads();  // s_val has been read
#pragma unroll
        for (int k = 0; k < ITEMS; ++k)
            if (rank[k] != 0xffffffffu) s_val[rank[k]] = m[k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const uint32_t lp = (uint32_t)(k * kSortThreads + tid);
            if (lp < nt) {
                const uint32_t d = (s_key[lp] >> shift) & 0xffu;
                const uint32_t pos = s_out[d] + (lp - s_lbase[d]);
                if (pos < n) mout_[(uint64_t)pos * W + w] = s_val[lp];
            }
        }
    }
}

}  // namespace

// One stable pass over digit `pass` of the keys in buffer `cur` (count in
// misc[slot]); with dev_buf the buffers are chosen on the device and a pass
// whose digit is the same for every key is skipped. mbuf (words > 0): the 32-bit
// words that travel with the keys.
// (Tiles of 1024 keys for small sorts were measured slower: 0.106 against 0.079 ms
// for the four passes over 1M depth keys.)
static cudaError_t radix_pass(geer_workspace *ws, uint32_t *const kbuf[2], uint32_t *const vbuf[2], int cur, int slot,
                              int check, int pass, int64_t cap_keys, cudaStream_t s, uint32_t *const *mbuf, int words,
                              int dev_buf) {
    constexpr int TILE = kSortThreads * kSortItems;
    const int shift = kRadixBits * pass;
    const unsigned tiles = (unsigned)std::max<int64_t>(1, (cap_keys + TILE - 1) / TILE);
    const unsigned hist_blocks = std::min(tiles, (unsigned)(ws->num_sms * 8));
    launch_k(k_radix_hist<kSortItems>, dim3(hist_blocks), dim3(kSortThreads), 0, s, kbuf[cur], kbuf[cur ^ 1], dev_buf,
             ws->d_misc, slot, check, shift, ws->d_tile_hist, ws->d_group_sum, ws->d_group_excl, ws->d_digit_base);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launch_k(words == 0   ? k_radix_scatter<kSortItems, 0>
             : words == 1 ? k_radix_scatter<kSortItems, 1>
                          : k_radix_scatter<kSortItems, 2>,
             dim3(tiles), dim3(kSortThreads), 0, s, kbuf[cur], vbuf[cur], kbuf[cur ^ 1], vbuf[cur ^ 1], dev_buf,
             ws->d_misc, slot, check, shift, ws->d_tile_hist, ws->d_group_excl, ws->d_digit_base,
             words ? mbuf[cur] : nullptr, words ? mbuf[cur ^ 1] : nullptr);
    return cudaGetLastError();
}

// Stable sort of the live items by depth key (4 digits of the FP32 bits). The
// passes choose their buffers on the device (see depth_sorted_buf): a digit
// that is the same for every key (the exponent's high bits when the depths span
// less than a factor of two) costs its histogram only.
cudaError_t launch_depth_sort(geer_workspace *ws, cudaStream_t s) {
    const int64_t items = (int64_t)ws->n_cams * ws->n_gauss;
    if (items > 0 && !small_front(ws)) {
        for (int p = 0; p < 4; ++p) {
            cudaError_t e = radix_pass(ws, ws->d_ikey, ws->d_iid, 0, kMiscLive, 0, p, items, s, nullptr, 0, 1);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

// Stable sort of the (super-tile, item) pairs by super-tile id (one or two
// 8-bit digits); the pairs' tile masks travel with them.
cudaError_t launch_tile_sort(geer_workspace *ws, cudaStream_t s) {
    int cur = 0;
    for (int p = 0; p < ws->n_sort_passes; ++p) {
        cudaError_t e = radix_pass(ws, ws->d_keys, ws->d_vals, cur, kMiscPairs, 1, p, ws->cap_pairs, s, ws->d_smask,
                                   mask_words(ws->super_size), 0);
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    ws->sorted_buf = cur;
    return launch_masks_order(ws, s);
}

}  // namespace geer
