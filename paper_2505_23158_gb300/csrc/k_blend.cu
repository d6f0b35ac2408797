// K7: per-tile front-to-back alpha compositing (Eq. 1; Sec. 3
// "Preliminaries: 3DGS").  One CTA of 128 threads per 16x16 tile, two pixels
// per thread (one column, 4 rows apart), so each record read from shared
// memory serves two pixels; each warp covers an 8x8 block so that its
// pixels terminate together.  The tile's Gaussians arrive in batches of 128
// records, gathered from the projection records into shared memory with
// cp.async and double-buffered (batch b+1 is in flight while batch b is
// composited; the keys of batch b+2 are already being read, so that no
// thread waits for a key before it can start a gather).
//
// Filtered walk: each thread tests the record it staged against the tile's
// four 8x8 blocks (walk.cuh, blocks_met), the warps ballot the results, and
// every warp makes a list of the records that can reach its own block and
// visits only those, in list order.  A record failing the test would be
// skipped by every pixel of the block (alpha < 1/255 there), so the image is
// that of walking the whole list, bit for bit.  With coarse bins (squares of
// 2^bin_log2 tiles) the tile walks its bin's key list the same way (a record
// meeting a block has a tile rect holding the tile, so it is on the tile's
// own list).
//
// Per pixel and Gaussian (record = mean', upper-triangular U with
// U^T U = (1/2) log2(e) Sigma'^-1, -log2 o', colour):
//   q = (u00 dx + u01 dy)^2 + (u11 dy)^2,  alpha = min(0.99, 2^-(q - log2 o'))
//   skip if alpha < 1/255; T' = T (1 - alpha); stop if T' < 1e-4;
//   C += T alpha rgb; T = T'.
// The step has no branches: alpha becomes 0 where the pixel skips (T' = T,
// weight 0); a pixel that stops keeps its T' < 1e-4, which makes the weight
// of every later step 0 (T only falls).  A thread's two pixels run in packed
// FP32 pairs.
//
// What bounds it: instruction issue and the FP32 pipes.  A visit of a record
// by a warp (64 pixels) takes about 38 instructions, 30 FP32 pipe cycles of
// them, against 58 with scalar steps, the hits taken bit by bit from the
// masks and every block testing every record for itself.  A 1080p chunk
// frame of 120k visible records (83M evaluated pairs): 97.1M -> 70.6M warp
// instructions, 135 -> 102 us (whole GPU to itself); a full-detail frame of
// 858k records 455 -> 254 us, its longest lists being walked four records at
// a time instead of one after the other.  Storing the scalars that enter
// packed steps twice in shared memory measured no fewer FP32 instructions (a
// packed operand may be one register used twice).  A list's last one to three
// records are visited as a pair and a single (filling the turn up with a
// record that nothing composites, and zeroing a stopped pixel's T: lone
// chunk frame 276 against 270 us, four 4K frames 1298 against 1276).  64 registers (8 CTAs per
// SM): 10 CTAs with 48 measured 2-4% slower, no limit (66-72 registers) 1-3%.
#include <type_traits>

#include "walk.cuh"

namespace lodge {

namespace {

constexpr int kBlendThreads = 128; // blend: two pixels per thread
constexpr int kBlendBatch = 128;   // blend: records per batch (one per thread)
constexpr int kUnroll = 4;         // records visited per turn of the walk

constexpr float kStop = 1e-4f;      // a pixel stops before its transmittance falls below

// two pixels of one thread
struct PixelPair {
    f32x2 T, C0, C1, C2;
};

// per half: a where the flag is set, else b
__device__ __forceinline__ f32x2 keep2(bool lo, bool hi, f32x2 a, f32x2 b) {
    float a0, a1, b0, b1;
    unpack2(a, a0, a1);
    unpack2(b, b0, b1);
    return pack2(lo ? a0 : b0, hi ? a1 : b1);
}

// One record against the thread's two pixels (Eq. 1).  Returns the weights
// T alpha (0 where the pixel skips or has stopped); T becomes the
// transmittance after the record (below kStop where it has stopped).
__device__ __forceinline__ void blend_pair(const char* rec, float pxf, float py0, PixelPair& p,
                                           f32x2& wgt) {
    constexpr int kNext = sizeof(float4) * kBlendBatch;
    const float4 a = *reinterpret_cast<const float4*>(rec);
    const float4 b = *reinterpret_cast<const float4*>(rec + kNext);
    const float cz = *reinterpret_cast<const float*>(rec + 2 * kNext);
    float t0, w0, t1, w1;
    row_pair_tw(a, b, pxf - a.x, py0, t0, w0, t1, w1);
    const f32x2 t = pack2(t0, t1), w = pack2(w0, w1);
    float z0, z1;
    unpack2(fma2(t, t, fma2(w, w, pack2(b.y, b.y))), z0, z1);
    const float a0 = fminf(0.99f, ex2_approx(-z0)), a1 = fminf(0.99f, ex2_approx(-z1));
    // alpha, or 0 below 1/255
    const f32x2 al = mul2(pack2(a0, a1), pack2(ge01(a0, 1.0f / 255.0f), ge01(a1, 1.0f / 255.0f)));
    const f32x2 Tn = mul2(p.T, fma2(al, pack2(-1.f, -1.f), pack2(1.f, 1.f)));
    float n0, n1;
    unpack2(Tn, n0, n1);
    wgt = mul2(mul2(p.T, al), pack2(ge01(n0, kStop), ge01(n1, kStop)));
    p.T = Tn;
    p.C0 = fma2(wgt, pack2(b.z, b.z), p.C0);
    p.C1 = fma2(wgt, pack2(b.w, b.w), p.C1);
    p.C2 = fma2(wgt, pack2(cz, cz), p.C2);
}

// kSave: frames kept for the adjoint also store the final transmittance and
// the list position (1-based) of the last composited record.  kCount: count
// the evaluated and composited (pixel, Gaussian) pairs.  kScore: raise
// f.rec_score[record] to the largest weight T alpha it receives.
template <bool kSave, bool kCount = false, bool kScore = false>
__device__ __forceinline__ void blend_tile(const BlendFrame& f, int tile) {
    __shared__ uint32_t s_id[kScore ? 2 : 1][kScore ? kBlendBatch : 1];   // staged records
    __shared__ uint32_t s_top[kScore ? kBlendBatch : 1];                  // their largest weights here
    __shared__ float4 s_rec[2][3][kBlendBatch];
    __shared__ uint32_t s_met[4][kBlendBatch / 32];        // per block: which records reach it
    __shared__ __align__(8) uint16_t s_hit[4][kBlendBatch];   // per warp: their offsets
    const int32_t width = f.width, height = f.height, tiles_x = f.tiles_x;
    const uint32_t* tile_val = f.tile_val;
    const uint32_t vmask = f.vmask, n_keys = f.n_keys, n_rec = f.n_rec;
    const float4* rec_a = f.rec_a;
    const float4* rec_b = f.rec_b;
    const float* rec_c = f.rec_c;
    const uint2* rec_rect = f.rec_rect;
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // warp w covers the 8x8 block (w & 1, w >> 1) of the tile; a lane owns
    // two pixels of one column, 4 rows apart
    const int x = tx * kTile + (warp & 1) * 8 + (lane & 7);
    const int y0 = ty * kTile + (warp >> 1) * 8 + (lane >> 3), y1 = y0 + 4;
    const bool in0 = x < width && y0 < height, in1 = x < width && y1 < height;
    const float pxf = (float)x + 0.5f, py0 = (float)y0 + 0.5f;
    const int bin = f.bin_log2 > 0 ? (ty >> f.bin_log2) * f.bins_x + (tx >> f.bin_log2) : tile;
    uint2 rg = f.ranges[bin];
    if (rg.y > n_keys || rg.x > rg.y) rg = make_uint2(0, 0);  // never for a consistent sort
    const int n = (int)(rg.y - rg.x);
    const int nb = (n + kBlendBatch - 1) / kBlendBatch;
    tile_val += rg.x;

    // a pixel outside the image counts as stopped (T = 0)
    PixelPair p{pack2(in0 ? 1.f : 0.f, in1 ? 1.f : 0.f), 0ull, 0ull, 0ull};
    float Tk0 = 1.f, Tk1 = 1.f;        // kSave: the transmittance behind the last composited record
    uint32_t last0 = 0, last1 = 0;
    uint32_t n_eval = 0, n_used = 0;   // counting mode only

    auto stopped = [&]() {
        float T0, T1;
        unpack2(p.T, T0, T1);
        return T0 < kStop && T1 < kStop;
    };
    auto stage = [&](int buf, uint32_t key) {
        const uint32_t j = min(key & vmask, n_rec - 1u);
        if (kScore) s_id[buf][tid] = j;
        cp_async16(&s_rec[buf][0][tid], rec_a + j);
        cp_async16(&s_rec[buf][1][tid], rec_b + j);
        cp_async4(&s_rec[buf][2][tid].x, rec_c + j);
        cp_async8(&s_rec[buf][2][tid].z, rec_rect + j);
    };
    if (kScore) s_top[tid] = 0u;
    if (tid < n) stage(0, tile_val[tid]);
    cp_async_commit();
    uint32_t key = kBlendBatch + tid < n ? tile_val[kBlendBatch + tid] : 0u;
    for (int b = 0; b < nb; ++b) {
        const int buf = b & 1;
        const int k1 = (b + 1) * kBlendBatch + tid;
        if (k1 < n) stage(buf ^ 1, key);
        cp_async_commit();
        key = k1 + kBlendBatch < n ? tile_val[k1 + kBlendBatch] : 0u;
        cp_async_wait1();
        {   // the record this thread staged against the tile's four blocks
            uint32_t met = 0;
            if (b * kBlendBatch + tid < n) {
                const float4 c = s_rec[buf][2][tid];
                met = blocks_met<kSave || kScore>(s_rec[buf][0][tid], s_rec[buf][1][tid],
                                                  make_uint2(__float_as_uint(c.z), __float_as_uint(c.w)),
                                                  tx * kTile, ty * kTile);
            }
            uint32_t m = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t v = __ballot_sync(0xffffffffu, met >> q & 1u);
                if (lane == q) m = v;
            }
            if (lane < 4) s_met[lane][warp] = m;
        }
        __syncthreads();
        if (!__all_sync(0xffffffffu, stopped())) {
            // the records that can reach this warp's block, in list order
            int nh = 0;
#pragma unroll
            for (int w = 0; w < kBlendBatch / 32; ++w) {
                const uint32_t m = s_met[warp][w];
                if (m >> lane & 1u)
                    s_hit[warp][nh + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(16 * (w * 32 + lane));
                nh += __popc(m);
            }
            __syncwarp();
            const char* base = reinterpret_cast<const char*>(&s_rec[buf][0][0]);
            // the next kN records of the list, together
            auto visit = [&](auto count, int i) {
                constexpr int kN = decltype(count)::value;
                uint32_t off[kN];
                if (kN == kUnroll) {
                    const uint2 h = *reinterpret_cast<const uint2*>(&s_hit[warp][i]);
                    off[0] = h.x & 0xffffu; off[1 % kN] = h.x >> 16; off[2 % kN] = h.y & 0xffffu; off[3 % kN] = h.y >> 16;
                } else if (kN == 2) {
                    const uint32_t h = *reinterpret_cast<const uint32_t*>(&s_hit[warp][i]);
                    off[0] = h & 0xffffu; off[1 % kN] = h >> 16;
                } else {
                    off[0] = s_hit[warp][i];
                }
                uint32_t top = 0u, top_at = 0u;   // lane u: largest weight of record u
#pragma unroll
                for (int u = 0; u < kN; ++u) {
                    f32x2 wgt;
                    if (kCount) {
                        float T0, T1;
                        unpack2(p.T, T0, T1);
                        n_eval += (T0 < kStop ? 0u : 1u) + (T1 < kStop ? 0u : 1u);
                    }
                    const PixelPair before = p;
                    blend_pair(base + off[u], pxf, py0, p, wgt);
                    if (kScore) {
                        float w0, w1;
                        unpack2(wgt, w0, w1);
                        const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(w0, w1)));
                        if (lane == u) { top = m; top_at = off[u] / 16u; }
                    }
                    if (kSave || kCount || kScore) {
                        float w0, w1, T0, T1;
                        unpack2(wgt, w0, w1);
                        unpack2(p.T, T0, T1);
                        if (kSave || kScore) {   // an infinite colour reaches only the pixels that composite it
                            p.C0 = keep2(w0 > 0.f, w1 > 0.f, p.C0, before.C0);
                            p.C1 = keep2(w0 > 0.f, w1 > 0.f, p.C1, before.C1);
                            p.C2 = keep2(w0 > 0.f, w1 > 0.f, p.C2, before.C2);
                        }
                        const uint32_t pos = (uint32_t)(b * kBlendBatch + 1) + off[u] / 16u;
                        if (w0 > 0.f) { Tk0 = T0; last0 = pos; ++n_used; }
                        if (w1 > 0.f) { Tk1 = T1; last1 = pos; ++n_used; }
                    }
                }
                if (kScore && top > s_top[top_at]) atomicMax(&s_top[top_at], top);
            };
            int i = 0;
            for (; i + kUnroll <= nh; i += kUnroll) {
                visit(std::integral_constant<int, kUnroll>{}, i);
                if (__all_sync(0xffffffffu, stopped())) break;
            }
            // the list's end, without visits that composite nothing
            if (i + kUnroll > nh) {
                if (nh & 2) { visit(std::integral_constant<int, 2>{}, i); i += 2; }
                if (nh & 1) visit(std::integral_constant<int, 1>{}, i);
            }
        }
        const bool end = __syncthreads_count(stopped()) == kBlendThreads;
        if (kScore) {
            // one atomic per tile and record that gains by it (the scores
            // only grow, so a stale read costs an atomic, never a score)
            const uint32_t top = s_top[tid];
            if (top) {
                s_top[tid] = 0u;   // (the next batch's walk is behind a barrier)
                uint32_t* to = f.rec_score + s_id[buf][tid];
                if (top > ld_volatile(to)) atomicMax(to, top);
            }
        }
        if (end) break;
    }
    cp_async_wait0();
    if (kCount) {
        for (int off = 16; off > 0; off >>= 1) {
            n_eval += __shfl_xor_sync(0xffffffffu, n_eval, off);
            n_used += __shfl_xor_sync(0xffffffffu, n_used, off);
        }
        if (lane == 0 && f.pairs) {
            atomicAdd(f.pairs, (unsigned long long)n_eval);
            atomicAdd(f.pairs + 1, (unsigned long long)n_used);
        }
    }
    float r0, r1, g0, g1, b0, b1;
    unpack2(p.C0, r0, r1);
    unpack2(p.C1, g0, g1);
    unpack2(p.C2, b0, b1);
    if (in0) {
        const int64_t pix = (int64_t)y0 * width + x;
        f.rgb[3 * pix + 0] = r0;
        f.rgb[3 * pix + 1] = g0;
        f.rgb[3 * pix + 2] = b0;
        if (kSave) { f.T_final[pix] = Tk0; f.last[pix] = last0; }
    }
    if (in1) {
        const int64_t pix = (int64_t)y1 * width + x;
        f.rgb[3 * pix + 0] = r1;
        f.rgb[3 * pix + 1] = g1;
        f.rgb[3 * pix + 2] = b1;
        if (kSave) { f.T_final[pix] = Tk1; f.last[pix] = last1; }
    }
}

template <bool kSave, bool kCount>
__global__ void __launch_bounds__(kBlendThreads, 8) blend_kernel(BlendFrame f) {
    chain_wait();
    blend_tile<kSave, kCount>(f, blockIdx.x);
}

// fewer CTAs than tiles: each takes the next tile from the counter
template <bool kCount>
__global__ void __launch_bounds__(kBlendThreads, 8) blend_loop_kernel(BlendFrame f, uint32_t* __restrict__ tile_ctr) {
    __shared__ int s_t;
    for (;;) {
        if (threadIdx.x == 0) s_t = (int)atomicAdd(tile_ctr, 1u);
        __syncthreads();
        const int t = s_t;
        __syncthreads();   // s_t is rewritten for the next tile
        if (t >= f.ntiles) break;
        blend_tile<false, kCount>(f, t);
    }
}

// One persistent launch for the tiles of several frames (a serving step): each
// CTA takes the next (frame, tile) item b of the step from the counter until
// all `total` are done; it is tile b - tile_base of the last frame whose
// tile_base <= b.
__global__ void __launch_bounds__(kBlendThreads, 8) blend_batch_loop_kernel(BlendBatch bb, uint32_t total,
                                                                         uint32_t* __restrict__ tile_ctr) {
    __shared__ uint32_t s_t;
    for (;;) {
        if (threadIdx.x == 0) s_t = atomicAdd(tile_ctr, 1u);
        __syncthreads();
        const uint32_t b = s_t;
        __syncthreads();   // s_t is rewritten for the next item
        if (b >= total) break;
        int lo = 0, hi = bb.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (bb.f[mid].tile_base <= b) lo = mid; else hi = mid - 1;
        }
        blend_tile<false>(bb.f[lo], (int)(b - bb.f[lo].tile_base));
    }
}


// K12: importance score (Sec. 3 "Importance pruning" / "Visibility
// filtering", after RadSplat): the compositing's walk, image included, and
// for every composited (pixel, record) pair the blending weight T * alpha.
// A visit takes the maximum over the warp's 64 pixels (one warp reduction of
// the FP32 bits: the weights are non-negative, so the unsigned maximum is
// the float maximum); a turn's four maxima raise the tile's shared maximum
// of each record with one instruction, and after each batch the staging
// thread raises rec_score[record] with one global atomic.
// Bound by instruction issue as the compositing.  Walking every record with
// one pixel per thread, a reduction and a global atomic per record and warp,
// a call over six 720p views of a chunk set took 3090 us; this walk 1870 us,
// 1940 with a shared atomic of its own per visit.
__global__ void __launch_bounds__(kBlendThreads, 8) importance_kernel(BlendFrame f) {
    blend_tile<false, false, true>(f, blockIdx.x);
}
__global__ void __launch_bounds__(kBlendThreads, 8)
importance_loop_kernel(BlendFrame f, uint32_t* __restrict__ tile_ctr) {
    __shared__ int s_t;
    for (;;) {
        if (threadIdx.x == 0) s_t = (int)atomicAdd(tile_ctr, 1u);
        __syncthreads();
        const int t = s_t;
        __syncthreads();   // s_t is rewritten for the next tile
        if (t >= f.ntiles) break;
        blend_tile<false, false, true>(f, t);
    }
}

// raise score[gid] to each record's score
__global__ void record_score_to_gid_kernel(const uint32_t* __restrict__ rec_score,
                                           const uint32_t* __restrict__ rec_gid, int64_t n_rec,
                                           int64_t n_total, uint32_t* __restrict__ score,
                                           const unsigned long long* __restrict__ d_nvis,
                                           const uint32_t* __restrict__ err) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rec || (d_nvis && (unsigned long long)r >= *d_nvis) || (*err & kErrOverflow)) return;
    const uint32_t v = rec_score[r];
    const uint32_t g = rec_gid[r];
    if (v && (int64_t)g < n_total) atomicMax(score + g, v);
}
}  // namespace

BlendFrame blend_frame(const DevCamera& cam, const uint2* ranges, const uint32_t* tile_val, uint32_t vmask,
                       int64_t n_keys, const float4* rec_a, const float4* rec_b, const float* rec_c,
                       int64_t n_rec, const BlendOut& o, int bin_log2, const uint2* rec_rect) {
    BlendFrame f;
    f.width = cam.width;
    f.height = cam.height;
    f.tiles_x = cam.tiles_x;
    f.ntiles = cam.tiles_x * cam.tiles_y;
    f.tile_base = 0;
    f.vmask = vmask;
    f.n_keys = (uint32_t)n_keys;
    f.n_rec = (uint32_t)std::max<int64_t>(n_rec, 1);
    f.bin_log2 = bin_log2;
    f.bins_x = (cam.tiles_x + (1 << f.bin_log2) - 1) >> f.bin_log2;
    f.ranges = ranges;
    f.tile_val = tile_val;
    f.rec_rect = rec_rect;
    f.pairs = nullptr;
    f.rec_a = rec_a;
    f.rec_b = rec_b;
    f.rec_c = rec_c;
    f.rgb = o.rgb;
    f.T_final = o.T_final;
    f.last = o.last;
    f.rec_score = nullptr;
    return f;
}

void launch_blend(const DevCamera& cam, const uint2* ranges, const uint32_t* tile_val, uint32_t vmask,
                  int64_t n_keys, const float4* rec_a, const float4* rec_b, const float* rec_c,
                  int64_t n_rec, const BlendOut& o, cudaStream_t s, int bin_log2, const uint2* rec_rect,
                  unsigned long long* pairs, uint32_t* tile_ctr, bool chained) {
    BlendFrame f = blend_frame(cam, ranges, tile_val, vmask, n_keys, rec_a, rec_b, rec_c, n_rec, o,
                               bin_log2, rec_rect);
    if (f.ntiles == 0) return;
    f.pairs = pairs;
    unsigned grid = (unsigned)f.ntiles;
    if (tile_ctr) {
        grid = (unsigned)std::min<int64_t>(f.ntiles, (int64_t)device_sms() * kBlendCtasPerSM);
    }
    const bool save = o.T_final != nullptr;   // (always a lone frame)
    if (save) {
        if (pairs)
            blend_kernel<true, true><<<(unsigned)f.ntiles, kBlendThreads, 0, s>>>(f);
        else
            blend_kernel<true, false><<<(unsigned)f.ntiles, kBlendThreads, 0, s>>>(f);
    } else if (tile_ctr) {
        if (pairs)   // counting variant (profiling), same walk
            blend_loop_kernel<true><<<grid, kBlendThreads, 0, s>>>(f, tile_ctr);
        else
            blend_loop_kernel<false><<<grid, kBlendThreads, 0, s>>>(f, tile_ctr);
    } else if (pairs) {
        blend_kernel<false, true><<<grid, kBlendThreads, 0, s>>>(f);
    } else {
        launch_chained(chained, blend_kernel<false, false>, grid, kBlendThreads, s, f);
    }
}

void launch_blend_batch(const BlendFrame* frames, int n, cudaStream_t s, uint32_t* tile_ctr) {
    BlendBatch bb;
    uint32_t base = 0;
    bb.n = 0;
    for (int i = 0; i < n && i < kMaxBlendBatch; ++i) {
        if (frames[i].ntiles == 0) continue;
        bb.f[bb.n] = frames[i];
        bb.f[bb.n].tile_base = base;
        base += (uint32_t)frames[i].ntiles;
        ++bb.n;
    }
    if (bb.n == 0) return;
    // as many CTAs as fit on the device at once (the step's compositing runs
    // after every frame's earlier stages)
    int per_sm = 1;
    const int nsm = device_sms();
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, blend_batch_loop_kernel, kBlendThreads, 0);
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)base, (int64_t)nsm * std::max(per_sm, 1));
    blend_batch_loop_kernel<<<grid, kBlendThreads, 0, s>>>(bb, base, tile_ctr);
}

void launch_importance(const DevCamera& cam, const uint2* ranges, const uint32_t* tile_val,
                       uint32_t vmask, int64_t n_keys, const float4* rec_a, const float4* rec_b,
                       const float* rec_c, int64_t n_rec, const uint32_t* rec_gid, float* rgb,
                       uint32_t* rec_score, int64_t n_total, float* score, cudaStream_t s, int bin_log2,
                       const uint2* rec_rect, uint32_t* tile_ctr, const unsigned long long* d_nvis,
                       const uint32_t* err) {
    BlendFrame f = blend_frame(cam, ranges, tile_val, vmask, n_keys, rec_a, rec_b, rec_c, n_rec,
                               BlendOut{rgb, nullptr, nullptr}, bin_log2, rec_rect);
    if (f.ntiles == 0) return;
    f.rec_score = rec_score;
    if (tile_ctr)
        importance_loop_kernel<<<(unsigned)std::min<int64_t>(f.ntiles, (int64_t)device_sms() * kBlendCtasPerSM),
                                 kBlendThreads, 0, s>>>(f, tile_ctr);
    else
        importance_kernel<<<(unsigned)f.ntiles, kBlendThreads, 0, s>>>(f);
    if (n_rec > 0)
        record_score_to_gid_kernel<<<(unsigned)((n_rec + 255) / 256), 256, 0, s>>>(
            rec_score, rec_gid, n_rec, n_total, reinterpret_cast<uint32_t*>(score), d_nvis, err);
}

}  // namespace lodge
