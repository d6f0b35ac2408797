// K4: tile binning.  Walks the visible records in depth order and emits one
// (bin id, record) pair per bin that the record's tile rect touches (Sec. 3
// "Preliminaries: 3DGS": each 2D Gaussian is assigned to every 16x16 tile it
// overlaps).  A bin is the tile itself or a square of 2^bin_log2 tiles; the
// compositing then drops, per tile, the records of its bin that miss the
// tile.  Key offsets by block scan plus decoupled look-back (or count, scan and
// write launches for large frames), the keys of a warp's records written by
// its lanes together; frames of large records write one record per warp.
//
// K6: per-bin [begin, end) ranges of the bin-sorted keys.
#include "common.cuh"

namespace lodge {

namespace {

// Pass 1: per depth-sorted visible record, its bin count; block scan plus
// decoupled look-back give the exclusive key offset koff[i] (koff[n_vis] =
// total).  The record id and rect are gathered into depth order (srec,
// srect, in bins) so that pass 2 reads them contiguously.
__global__ void __launch_bounds__(kEmitThreads)
emit_offsets_kernel(const uint32_t* __restrict__ sorted_rec, int64_t n_vis,
                    const uint2* __restrict__ rec_rect, uint32_t* __restrict__ koff,
                    uint32_t* __restrict__ srec, uint2* __restrict__ srect,
                    int bin_log2, uint32_t* __restrict__ status, uint32_t* __restrict__ counter,
                    uint32_t* __restrict__ err) {
    __shared__ uint32_t s_scan[33];
    __shared__ uint32_t s_tile, s_prefix;
    if (threadIdx.x == 0) s_tile = atomicAdd(counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint32_t ntiles = (uint32_t)((n_vis + kEmitThreads - 1) / kEmitThreads);
    const int64_t i = (int64_t)tile * kEmitThreads + threadIdx.x;
    uint32_t cnt = 0;
    if (i < n_vis) {
        uint32_t rec = sorted_rec[i];
        if ((int64_t)rec >= n_vis) { atomicOr(err, kErrBadIndex); rec = 0; }
        const uint2 p = rec_rect[rec];   // pixel range -> tile range -> bin range
        const uint2 r = make_uint2((((p.x & 0xffffu) / kTile) >> bin_log2) |
                                       ((((p.x >> 16) / kTile) >> bin_log2) << 16),
                                   (((p.y & 0xffffu) / kTile) >> bin_log2) |
                                       ((((p.y >> 16) / kTile) >> bin_log2) << 16));
        uint32_t w = (r.y & 0xffffu) - (r.x & 0xffffu) + 1u;
        uint32_t h = (r.y >> 16) - (r.x >> 16) + 1u;
        cnt = w * h;
        srec[i] = rec;
        srect[i] = r;
    }
    uint32_t total;
    uint32_t excl = block_exclusive_scan(cnt, s_scan, &total);
    if (threadIdx.x < 32) {
        uint32_t prefix = 0;
        if (tile == 0) {
            if (threadIdx.x == 0) st_volatile(status, kStInc | total);
        } else {
            if (threadIdx.x == 0) st_volatile(status + tile, kStAgg | total);
            prefix = warp_lookback(status, tile, err);
            if (threadIdx.x == 0) st_volatile(status + tile, kStInc | (prefix + total));
        }
        if (threadIdx.x == 0) {
            s_prefix = prefix;
            if (tile == ntiles - 1) koff[n_vis] = prefix + total;
        }
    }
    __syncthreads();
    if (i < n_vis) koff[i] = s_prefix + excl;
}

// What a CTA needs to write its records' keys.
struct KeyWriter {
    int32_t bins_x;
    uint32_t* tile_key;
    uint32_t* tile_val;
    int rbits, passes;
    uint32_t last_mask;
    uint32_t (*hist)[256];   // the bin sort's digit counts, shared memory

    __device__ __forceinline__ void put(int64_t at, uint32_t bin, uint32_t rec) const {
        if (rbits) {
            tile_key[at] = (bin << rbits) | rec;
        } else {
            tile_key[at] = bin;
            tile_val[at] = rec;
        }
        atomicAdd(&hist[0][bin & (passes == 1 ? last_mask : 0xffu)], 1u);
    }
    // the digits above the lowest, counted per row of a record's bins
    // [x0, x0 + w): one contiguous range of ids, split where a digit changes
    __device__ __forceinline__ void count_row(uint32_t x0, uint32_t y, uint32_t w) const {
        for (int p = 1; p < passes; ++p) {
            const uint32_t mask = p == passes - 1 ? last_mask : 0xffu;
            const int sh = 8 * p;
            uint32_t a = y * (uint32_t)bins_x + x0;
            const uint32_t b = a + w - 1u;
            while (a <= b) {
                const uint32_t end = min(b, ((a >> sh) + 1u << sh) - 1u);
                atomicAdd(&hist[p][(a >> sh) & mask], end - a + 1u);
                a = end + 1u;
            }
        }
    }
    // The keys of a warp's records, one record per lane: cnt keys (w bins a
    // row from (x0, y0)) at position `at`; lanes with nothing to write have
    // cnt = 0.  The lanes take consecutive keys: a key's record is found by
    // a binary search over the lanes' running counts, so that a warp takes
    // as many turns as it has keys / 32 and stores whole sectors, instead of
    // as many as its largest record has keys, each lane storing its own run.
    __device__ __forceinline__ void warp_records(uint32_t cnt, uint32_t at, uint32_t x0, uint32_t y0, uint32_t w,
                                                 uint32_t rec) const {
        const int lane = threadIdx.x & 31;
        uint32_t incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const uint32_t excl = incl - cnt, total = __shfl_sync(0xffffffffu, incl, 31);
        const uint32_t xy = x0 | (y0 << 16);   // bin coordinates < 2^16
        for (uint32_t k0 = 0; k0 < total; k0 += 32) {
            const uint32_t k = k0 + lane;
            int own = 0;   // the last lane with excl <= k
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, excl, own + step) <= k) own += step;
            const uint32_t j = k - __shfl_sync(0xffffffffu, excl, own);
            const uint32_t oxy = __shfl_sync(0xffffffffu, xy, own), ow = __shfl_sync(0xffffffffu, w, own);
            const uint32_t oat = __shfl_sync(0xffffffffu, at, own), orec = __shfl_sync(0xffffffffu, rec, own);
            if (k < total) {
                // j, w <= kWarpKeys: j + 1/2 is 1/(2 w) of a row or more from
                // a whole one, far above the quotient's error
                const uint32_t row = (uint32_t)__fdividef((float)j + 0.5f, (float)ow);
                put((int64_t)oat + j, ((oxy >> 16) + row) * (uint32_t)bins_x + (oxy & 0xffffu) + (j - row * ow), orec);
            }
        }
        if (cnt)
            for (uint32_t r = 0; r * w < cnt; ++r) count_row(x0, y0 + r, w);
    }
    // one record by a whole warp
    __device__ __forceinline__ void large_record(uint32_t cnt, int64_t at, uint32_t x0, uint32_t y0, uint32_t w,
                                                 uint32_t rec) const {
        const int lane = threadIdx.x & 31;
        // key k = lane + 32 j sits at row k / w, column k % w (stepped)
        uint32_t row = lane / w, col = lane - row * w;
        const uint32_t drow = 32u / w, dcol = 32u - drow * w;
        for (uint32_t k = lane; k < cnt; k += 32) {
            put(at + k, (y0 + row) * (uint32_t)bins_x + x0 + col, rec);
            row += drow;
            col += dcol;
            if (col >= w) { col -= w; ++row; }
        }
        for (uint32_t r = lane; r * w < cnt; r += 32) count_row(x0, y0 + r, w);
    }
};

// Large records: one warp per depth-sorted record writes the record's keys,
// koff[i] .. koff[i+1]-1 (warps of a CTA take consecutive records, CTAs
// stride over the list).
__global__ void __launch_bounds__(kEmitThreads)
emit_keys_rect_kernel(const uint32_t* __restrict__ koff, const uint32_t* __restrict__ srec,
                 const uint2* __restrict__ srect, int64_t n_vis, int32_t bins_x,
                 uint32_t* __restrict__ tile_key, uint32_t* __restrict__ tile_val, int rbits,
                 int passes, uint32_t last_mask, uint32_t* __restrict__ digit_hist) {
    __shared__ uint32_t s_hist[3][256];
    for (int i = threadIdx.x; i < 3 * 256; i += kEmitThreads) (&s_hist[0][0])[i] = 0;
    __syncthreads();
    const KeyWriter kw{bins_x, tile_key, tile_val, rbits, passes, last_mask, s_hist};
    const int64_t wstride = (int64_t)gridDim.x * (kEmitThreads / 32);
    for (int64_t i = (int64_t)blockIdx.x * (kEmitThreads / 32) + (threadIdx.x >> 5); i < n_vis;
         i += wstride) {
        const uint2 rr = srect[i];
        kw.large_record(koff[i + 1] - koff[i], koff[i], rr.x & 0xffffu, rr.x >> 16,
                        (rr.y & 0xffffu) - (rr.x & 0xffffu) + 1u, srec[i]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += kEmitThreads) {
        const uint32_t c = (&s_hist[0][0])[i];
        if (c) atomicAdd(digit_hist + i, c);
    }
}

// Tile t of depth-sorted records: the first one, and how many (before the
// end of the list is taken into account).  With equal tiles the CTAs of the
// nearest records wrote most of the keys while the others had finished: four
// full-detail 1080p frames 1908 -> 1771 us, an LOD frame 286 -> 271 us (with
// the first 1024 records instead of 4096 in near tiles 1825 and 265).
__device__ __forceinline__ int64_t emit_first(uint32_t t, int rest, int& size) {
    constexpr uint32_t kNearTiles = kEmitNear / kEmitNearTile;
    size = t < kNearTiles ? kEmitNearTile : rest;
    return t < kNearTiles ? (int64_t)t * kEmitNearTile : kEmitNear + (int64_t)(t - kNearTiles) * rest;
}

// Offsets and emission in one pass.  A CTA takes a tile of depth-sorted records,
// scans their bin counts and finds its key offset by decoupled look-back.
// Records of at most kWarpKeys keys are written by their warp together; larger
// ones (the nearest records, which all fall in the first CTAs) go to a shared
// list that the CTA's warps take one record at a time.  The bin sort's digit
// counts are kept in shared memory and flushed once.  Bound by the latency of
// its chain (ticket, records, look-back), not by its bytes: a chunk frame's
// 124k records and 450k keys take 16.5 us where a thread writing its own
// record's keys took 25.8.
constexpr uint32_t kWarpKeys = 32;   // at most 2^10 (warp_records)
__global__ void __launch_bounds__(kEmitThreads)
emit_fused_kernel(const uint32_t* sorted_rec, int64_t n_vis,
                  const uint2* rec_rect, int bin_log2, int32_t bins_x, int64_t n_keys,
                  uint32_t* tile_key, uint32_t* tile_val, int rbits,
                  int passes, uint32_t last_mask, uint32_t* digit_hist,
                  uint32_t* status, uint32_t* counter,
                  uint32_t* err, const unsigned long long* d_nvis,
                  const unsigned long long* d_nkeys) {
    chain_wait();
    // with device counts, n_vis and n_keys are capacities: the counts decide
    // which CTAs work and the keys must fit n_keys
    if (d_nvis) {
        const unsigned long long c = *d_nvis;
        if (c < (unsigned long long)n_vis) n_vis = (int64_t)c;
    }
    const int64_t key_cap = n_keys;
    if (d_nkeys) n_keys = (int64_t)*d_nkeys;
    __shared__ uint32_t s_scan[33];
    __shared__ uint32_t s_tile, s_prefix, s_nbig;
    __shared__ uint32_t s_big[kEmitThreads];
    __shared__ uint32_t s_off[kEmitThreads];
    __shared__ uint32_t s_cnt[kEmitThreads];
    __shared__ uint2 s_rect[kEmitThreads];
    __shared__ uint32_t s_rec[kEmitThreads];
    __shared__ uint32_t s_hist[3][256];
    for (int i = threadIdx.x; i < 3 * 256; i += kEmitThreads) (&s_hist[0][0])[i] = 0;
    if (threadIdx.x == 0) { s_tile = atomicAdd(counter, 1u); s_nbig = 0; }
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint32_t ntiles = (uint32_t)emit_tiles(n_vis, kEmitThreads);
    if (tile >= ntiles) return;   // past the device count (later tiles too)
    int size;
    const int64_t i = emit_first(tile, kEmitThreads, size) + threadIdx.x;
    uint32_t cnt = 0, rec = 0, x0 = 0, y0 = 0, w = 1;
    if ((int)threadIdx.x < size && i < n_vis) {
        rec = sorted_rec[i];
        if ((int64_t)rec >= n_vis) { atomicOr(err, kErrBadIndex); rec = 0; }
        const uint2 p = rec_rect[rec];   // pixel range -> tile range -> bin range
        x0 = ((p.x & 0xffffu) / kTile) >> bin_log2;
        y0 = ((p.x >> 16) / kTile) >> bin_log2;
        const uint32_t x1 = ((p.y & 0xffffu) / kTile) >> bin_log2, y1 = ((p.y >> 16) / kTile) >> bin_log2;
        w = x1 - x0 + 1u;
        cnt = w * (y1 - y0 + 1u);
    }
    uint32_t total;
    const uint32_t excl = block_exclusive_scan(cnt, s_scan, &total);
    if (cnt > kWarpKeys) {
        const uint32_t slot = atomicAdd(&s_nbig, 1u);
        s_big[slot] = threadIdx.x;
        s_off[threadIdx.x] = excl;
        s_cnt[threadIdx.x] = cnt;
        s_rect[threadIdx.x] = make_uint2(x0 | (y0 << 16), w);   // bin coordinates < 2^12
        s_rec[threadIdx.x] = rec;
    }
    if (threadIdx.x < 32) {
        uint32_t prefix = 0;
        if (tile == 0) {
            if (threadIdx.x == 0) st_volatile(status, kStInc | total);
        } else {
            if (threadIdx.x == 0) st_volatile(status + tile, kStAgg | total);
            prefix = warp_lookback(status, tile, err);
            if (threadIdx.x == 0) st_volatile(status + tile, kStInc | (prefix + total));
        }
        if (threadIdx.x == 0) {
            s_prefix = prefix;
            if (tile == ntiles - 1 && (int64_t)prefix + total != n_keys) atomicOr(err, kErrOverflow);
        }
    }
    __syncthreads();
    const int64_t base = s_prefix;
    if ((int64_t)base + total > n_keys || (int64_t)base + total > key_cap) {
        // more keys than counted (never for consistent counts) or than fit
        if (threadIdx.x == 0) atomicOr(err, kErrOverflow);
        return;
    }
    const KeyWriter kw{bins_x, tile_key, tile_val, rbits, passes, last_mask, s_hist};
    kw.warp_records(cnt <= kWarpKeys ? cnt : 0u, (uint32_t)base + excl, x0, y0, w, rec);
    const uint32_t nbig = s_nbig;
    for (uint32_t b = threadIdx.x >> 5; b < nbig; b += kEmitThreads / 32) {
        const uint32_t t = s_big[b];
        const uint2 rr = s_rect[t];
        kw.large_record(s_cnt[t], base + s_off[t], rr.x & 0xffffu, rr.x >> 16, rr.y, s_rec[t]);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < passes * 256; j += kEmitThreads) {
        const uint32_t c = (&s_hist[0][0])[j];
        if (c) atomicAdd(digit_hist + j, c);
    }
}

// Emission for large frames in three launches without look-back: count the
// bin keys of each tile of 1024 depth-sorted records, scan the tile counts
// in one CTA, then write each tile's keys at its offset.  With thousands of
// tiles in flight the fused kernel's CTAs spend most of their time at the
// barrier behind their look-back; here every CTA works independently and
// the records' rects are read twice instead.
constexpr int64_t kEmitSplitMin = 1ll << 21;                 // record capacity above which it is used

__device__ __forceinline__ uint32_t rec_bin_rect(const uint2* rec_rect, uint32_t rec,
                                                 int bin_log2, uint32_t& x0, uint32_t& y0, uint32_t& w) {
    const uint2 p = rec_rect[rec];   // pixel range -> tile range -> bin range
    x0 = ((p.x & 0xffffu) / kTile) >> bin_log2;
    y0 = ((p.x >> 16) / kTile) >> bin_log2;
    const uint32_t x1 = ((p.y & 0xffffu) / kTile) >> bin_log2, y1 = ((p.y >> 16) / kTile) >> bin_log2;
    w = x1 - x0 + 1u;
    return w * (y1 - y0 + 1u);
}

__device__ __forceinline__ int64_t device_count(int64_t cap, const unsigned long long* d) {
    if (!d) return cap;
    const unsigned long long c = *d;
    return c < (unsigned long long)cap ? (int64_t)c : cap;
}

template <int kEmitRecs>
__global__ void __launch_bounds__(kEmitThreads)
emit_count_kernel(const uint32_t* sorted_rec, int64_t n_vis_cap,
                  const unsigned long long* d_nvis, const uint2* rec_rect,
                  int bin_log2, uint32_t* tile_sum, uint32_t* err) {
    constexpr int kEmitTileRecs = kEmitThreads * kEmitRecs;
    __shared__ uint32_t s_part[kEmitThreads / 32];
    chain_wait();
    const int64_t n_vis = device_count(n_vis_cap, d_nvis);
    int size;
    const int64_t t0 = emit_first(blockIdx.x, kEmitTileRecs, size);
    if (t0 >= n_vis) return;   // past the device count (later tiles too)
    const int64_t t1 = min(n_vis, t0 + size);
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < kEmitRecs; ++j) {
        const int64_t i = t0 + (int64_t)j * kEmitThreads + threadIdx.x;
        if (i < t1) {
            uint32_t rec = sorted_rec[i];
            if ((int64_t)rec >= n_vis) { atomicOr(err, kErrBadIndex); rec = 0; }
            uint32_t x0, y0, w;
            sum += rec_bin_rect(rec_rect, rec, bin_log2, x0, y0, w);
        }
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
        for (int w = 0; w < kEmitThreads / 32; ++w) tot += s_part[w];
        tile_sum[blockIdx.x] = tot;
    }
}

// One CTA of 1024 threads: the tile counts become exclusive offsets in place;
// their total must equal the keys the projection counted and fit key_cap.
__global__ void __launch_bounds__(1024)
emit_scan_kernel(int tile_recs, uint32_t* tile_sum, int64_t n_vis_cap, const unsigned long long* d_nvis,
                 int64_t key_cap, const unsigned long long* d_nkeys, uint32_t* err) {
    __shared__ uint32_t s_scan[33];
    chain_wait();
    const int64_t n_vis = device_count(n_vis_cap, d_nvis);
    const int64_t ntiles = emit_tiles(n_vis, tile_recs);
    uint64_t carry = 0;
    for (int64_t base = 0; base < ntiles; base += 1024) {
        const int64_t t = base + threadIdx.x;
        const uint32_t v = t < ntiles ? tile_sum[t] : 0u;
        uint32_t total;
        const uint32_t e = block_exclusive_scan(v, s_scan, &total);
        if (t < ntiles) tile_sum[t] = (uint32_t)(carry + e);
        carry += total;
    }
    if (threadIdx.x == 0) {
        const int64_t n_keys = d_nkeys ? (int64_t)*d_nkeys : key_cap;
        if ((int64_t)carry != n_keys || (int64_t)carry > key_cap) atomicOr(err, kErrOverflow);
    }
}

template <int kEmitRecs>
__global__ void __launch_bounds__(kEmitThreads)
emit_write_kernel(const uint32_t* sorted_rec, int64_t n_vis_cap,
                  const unsigned long long* d_nvis, const uint2* rec_rect,
                  int bin_log2, int32_t bins_x, int64_t key_cap, const uint32_t* tile_off,
                  uint32_t* tile_key, uint32_t* tile_val, int rbits, int passes,
                  uint32_t last_mask, uint32_t* digit_hist, uint32_t* err) {
    constexpr int kEmitTileRecs = kEmitThreads * kEmitRecs;
    __shared__ uint32_t s_scan[33];
    __shared__ uint32_t s_nbig;
    __shared__ uint32_t s_big[kEmitTileRecs];     // (thread << 2 | j) of records with many keys
    __shared__ uint32_t s_off[kEmitTileRecs];
    __shared__ uint32_t s_hist[3][256];
    chain_wait();
    const int64_t n_vis = device_count(n_vis_cap, d_nvis);
    int size;
    const int64_t t0 = emit_first(blockIdx.x, kEmitTileRecs, size);
    if (t0 >= n_vis) return;
    const int64_t t1 = min(n_vis, t0 + size);
    for (int i = threadIdx.x; i < 3 * 256; i += kEmitThreads) (&s_hist[0][0])[i] = 0;
    if (threadIdx.x == 0) s_nbig = 0;
    // a thread's records are j * kEmitThreads + thread, so that the loads
    // are coalesced; the keys follow record order, which the scan below
    // gives as (j, thread) order
    uint32_t rec[kEmitRecs], cnt[kEmitRecs], bx[kEmitRecs], by[kEmitRecs], bw[kEmitRecs];
#pragma unroll
    for (int j = 0; j < kEmitRecs; ++j) {
        const int64_t i = t0 + (int64_t)j * kEmitThreads + threadIdx.x;
        rec[j] = 0; cnt[j] = 0; bx[j] = 0; by[j] = 0; bw[j] = 1;
        if (i < t1) {
            rec[j] = sorted_rec[i];
            if ((int64_t)rec[j] >= n_vis) rec[j] = 0;   // flagged by the count kernel
            cnt[j] = rec_bin_rect(rec_rect, rec[j], bin_log2, bx[j], by[j], bw[j]);
        }
    }
    const int64_t tbase = tile_off[blockIdx.x];
    const KeyWriter kw{bins_x, tile_key, tile_val, rbits, passes, last_mask, s_hist};
    uint32_t run = 0;   // keys of the record groups before group j in this tile
    __syncthreads();   // s_hist and s_nbig are set
#pragma unroll
    for (int j = 0; j < kEmitRecs; ++j) {
        uint32_t total;
        const uint32_t excl = block_exclusive_scan(cnt[j], s_scan, &total);
        const int64_t at0 = tbase + run + excl;
        uint32_t mine = cnt[j];
        if (at0 + cnt[j] > key_cap) {
            if (cnt[j]) atomicOr(err, kErrOverflow);
            mine = 0;
        } else if (cnt[j] > kWarpKeys) {
            const uint32_t slot = atomicAdd(&s_nbig, 1u);
            s_big[slot] = (threadIdx.x << 2) | (uint32_t)j;
            s_off[slot] = run + excl;
            mine = 0;
        }
        kw.warp_records(mine, (uint32_t)at0, bx[j], by[j], bw[j], rec[j]);
        // the next record group's keys follow this group's
        run += total;
    }
    __syncthreads();
    // records with many keys: one warp each; their rects are read again
    const uint32_t nbig = s_nbig;
    for (uint32_t b = threadIdx.x >> 5; b < nbig; b += kEmitThreads / 32) {
        const uint32_t tj = s_big[b];
        const int64_t i = t0 + (int64_t)(tj & 3u) * kEmitThreads + (tj >> 2);
        uint32_t r = sorted_rec[i];
        if ((int64_t)r >= n_vis) r = 0;
        uint32_t x0, y0, w;
        const uint32_t c = rec_bin_rect(rec_rect, r, bin_log2, x0, y0, w);
        kw.large_record(c, tbase + s_off[b], x0, y0, w, r);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < passes * 256; j += kEmitThreads) {
        const uint32_t c = (&s_hist[0][0])[j];
        if (c) atomicAdd(digit_hist + j, c);
    }
}

// K6: per tile [begin, end) of the tile-sorted keys (tile = key >> shift);
// 4 keys per thread.
__global__ void ranges_kernel(const uint32_t* __restrict__ key, int64_t n, uint2* __restrict__ ranges,
                              uint32_t ntiles, int shift) {
    const int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (i0 >= n) return;
    uint32_t prev = i0 > 0 ? key[i0 - 1] >> shift : 0xffffffffu;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int64_t i = i0 + j;
        if (i >= n) break;
        const uint32_t t = key[i] >> shift;
        const uint32_t next = i + 1 < n ? key[i + 1] >> shift : 0xffffffffu;
        if (t < ntiles) {
            if (t != prev) ranges[t].x = (uint32_t)i;
            if (t != next) ranges[t].y = (uint32_t)(i + 1);
        }
        prev = t;
    }
}

}  // namespace

// digits of the bin ids: passes and the mask of the last one
static void bin_digits(int key_bits, int* passes, uint32_t* last_mask) {
    const int P = (key_bits + 7) / 8;
    const int last_bits = key_bits - 8 * (P - 1);
    *passes = P;
    *last_mask = last_bits >= 8 ? 0xffu : ((1u << last_bits) - 1u);
}

int launch_emit(const uint32_t* sorted_rec, int64_t n_vis, const uint2* rec_rect,
                int32_t bins_x, int bin_log2, uint32_t* koff, uint32_t* srec, uint2* srect,
                int64_t n_keys, uint32_t* tile_key, uint32_t* tile_val, int rbits, int key_bits,
                uint32_t* digit_hist, uint32_t* status, uint32_t* tile_counter, uint32_t* err,
                cudaStream_t s) {
    if (n_vis == 0 || n_keys == 0) return 0;
    if (!emit_by_record(n_vis, n_keys))
        return launch_emit_counted(sorted_rec, n_vis, nullptr, rec_rect, bins_x, bin_log2, n_keys, nullptr,
                                   tile_key, tile_val, rbits, key_bits, digit_hist, status, tile_counter, err, s);
    // records average a warp's worth of keys or more: one warp per record
    int P;
    uint32_t last_mask;
    bin_digits(key_bits, &P, &last_mask);
    emit_offsets_kernel<<<(unsigned)((n_vis + kEmitThreads - 1) / kEmitThreads), kEmitThreads, 0, s>>>(
        sorted_rec, n_vis, rec_rect, koff, srec, srect, bin_log2, status, tile_counter, err);
    const unsigned grid = (unsigned)std::min<int64_t>((n_vis + kEmitThreads / 32 - 1) / (kEmitThreads / 32),
                                                      (int64_t)device_sms() * 8);
    emit_keys_rect_kernel<<<grid, kEmitThreads, 0, s>>>(koff, srec, srect, n_vis, bins_x, tile_key,
                                                        tile_val, rbits, P, last_mask, digit_hist);
    return 2;
}

int launch_emit_counted(const uint32_t* sorted_rec, int64_t n_vis_cap, const unsigned long long* d_nvis,
                        const uint2* rec_rect, int32_t bins_x, int bin_log2, int64_t key_cap,
                        const unsigned long long* d_nkeys, uint32_t* tile_key, uint32_t* tile_val,
                        int rbits, int key_bits, uint32_t* digit_hist, uint32_t* status,
                        uint32_t* tile_counter, uint32_t* err, cudaStream_t s, bool chained) {
    const int64_t nb = emit_tiles(n_vis_cap, kEmitThreads);
    if (nb == 0) return 0;
    int P;
    uint32_t last_mask;
    bin_digits(key_bits, &P, &last_mask);
    if (n_vis_cap > kEmitSplitMin) {
        // count, scan, write (the tile counts and offsets live in `status`,
        // which holds a word per tile of the fused kernel)
        const unsigned nt = (unsigned)emit_tiles(n_vis_cap, 4 * kEmitThreads);
        launch_chained(chained, emit_count_kernel<4>, nt, kEmitThreads, s, sorted_rec, n_vis_cap, d_nvis, rec_rect, bin_log2,
                                                         status, err);
        launch_chained(chained, emit_scan_kernel, 1, 1024, s, 4 * kEmitThreads, status, n_vis_cap, d_nvis, key_cap, d_nkeys, err);
        launch_chained(chained, emit_write_kernel<4>, nt, kEmitThreads, s, sorted_rec, n_vis_cap, d_nvis, rec_rect, bin_log2, bins_x,
                                                         key_cap, status, tile_key, tile_val, rbits, P, last_mask,
                                                         digit_hist, err);
        return 3;
    }
    launch_chained(chained, emit_fused_kernel, (unsigned)nb, kEmitThreads, s, sorted_rec, n_vis_cap, rec_rect, bin_log2, bins_x,
                                                            key_cap, tile_key, tile_val, rbits, P, last_mask,
                                                            digit_hist, status, tile_counter, err, d_nvis,
                                                            d_nkeys);
    return 1;
}

void launch_ranges(const uint32_t* tile_key, int64_t n_keys, uint2* ranges, int64_t ntiles,
                   int shift, cudaStream_t s) {
    if (n_keys == 0) return;
    const int64_t nt = (n_keys + 3) / 4;
    ranges_kernel<<<(unsigned)((nt + 255) / 256), 256, 0, s>>>(tile_key, n_keys, ranges,
                                                             (uint32_t)ntiles, shift);
}

}  // namespace lodge
