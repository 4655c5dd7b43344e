// Many views in one persistent launch: Algorithm 1's selection and blend fused
// per screen tile, over the tiles of every view of a batch (the paper renders
// 4 random training views per scene per step, Appendix D; inference renders
// many views of several scenes).
//
// GB300 design: a grid of (SMs x resident CTAs) persistent CTAs pulls
// (view, tile) work items from one atomic counter, so views of very different
// sizes balance without a host round trip.  Each CTA is warp-specialised and
// double-buffered, so the latency-bound selection of one tile overlaps the
// bandwidth-bound blend of the previous one:
//   1. selection (warps 0-3, select_tile.cuh, the same code as qr_select):
//      each warp walks an 8 x 8 block of the tile on its own; the kept ids and
//      normalised weights go to one of two shared-memory buffers and are also
//      written out (coalesced runs) for a backward pass;
//   2. blend (8 warps, warp per 2x2 pixel group whatever K is, as in qr_blend, one
//      channel chunk of the rows after the other): equal ids of the group are
//      merged with __match_any_sync, the group's weights of each distinct row
//      are gathered into a per-warp table, each distinct feature row (or its
//      chunk) is read once with 16-byte loads and accumulated into every pixel
//      of the group, and the rows of the map are written with streaming
//      stores.  The same groups and the same order of rows make the map of 16 x
//      16 tiles qr_blend's bit for bit.
// Hand-over between the roles uses named barriers (below).  Per-view
// descriptors live in device memory (qr_batch_prepare), the counter is
// cleared by a memset on the stream, so the launch can sit in a CUDA graph.
// Bound by the blend warps' latency chains and the write of the maps: 8 views
// of two rooms (5.0M pixels, 512 BF16 channels, 10.3 GB of maps) 2,025 us with
// the group's table built for every channel chunk, 1,895 us with one table
// for all of a group's chunks (0.80 of a plain copy's rate).
// K > 8, two pixels (K <= 16) or one per group -> four, us, six views of a 200k
// room, scores not asked for: 512 FP32 channels K = 9 2298 -> 2086, K = 16 2997 ->
// 2812, K = 17 4643 -> 2958, K = 24 6395 -> 4760, K = 32 8837 -> 5761; 512 BF16 K =
// 16 2596 -> 2447, K = 32 8279 -> 5377; 128 FP32 K = 16 1418 -> 1322, K = 24 2654 ->
// 2605 (the larger tables leave one CTA per SM from K = 24 on), K = 32 3801 -> 3014.
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "quad.cuh"
#include "select_tile.cuh"

namespace qr {

struct BatchView {
    const float4 *rec_m;
    const float4 *rec_w;
    const float *rec_a;
    const float *rec_h;
    const uint32_t *igid;
    const uint2 *ranges;
    const unsigned char *feat;
    const float *fscale;
    int32_t *ids;
    float *w;
    uint8_t *cnt;
    float *out;
    int64_t n_gauss;
    int W, H, tile_w, tiles_x, tiles_y, K;
    float alpha_min, alpha_max;
    uint32_t tile_base;     // first work item of this view
    uint32_t vec;           // ids and weights take 16-byte stores
};

namespace {

__device__ __forceinline__ void fma2b(float *acc, float w, float x0, float x1) {
    asm("{\n .reg .b64 a, ww, xx;\n mov.b64 a, {%0, %1};\n mov.b64 ww, {%2, %2};\n"
        " mov.b64 xx, {%3, %4};\n fma.rn.f32x2 a, ww, xx, a;\n mov.b64 {%0, %1}, a;\n}\n"
        : "+f"(acc[0]), "+f"(acc[1]) : "f"(w), "f"(x0), "f"(x1));
}

__device__ __forceinline__ void st_cs(float4 *p, float4 v) {
    asm volatile("st.global.cs.v4.f32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// ------------------------------------------------------------------ the kernel
// Warp roles of a CTA: warps 0..3 select (select_block, an 8 x 8 block of the
// tile each), warps 4..4+nbw-1 blend (nbw = 4 or 8, from the launch's block size).  Two shared-memory buffers hold a tile's
// kept ids, normalised weights and counts; the selection fills one while the
// blend warps read the other.  Hand-over uses hardware named barriers:
//   FULL[b]  (ids 2, 3): selection arrives once buffer b holds tile n (or the
//                        end marker), blend warps wait;
//   EMPTY[b] (ids 4, 5): blend warps arrive once done with buffer b, the
//                        selection waits before refilling it (from its third
//                        tile on) and once more after the end marker for the
//                        last tile's arrival, so every arrival is matched;
//   id 1:                the selection threads among themselves, once per
//                        tile (the item that thread 0 took).
// Every thread of both roles runs the same number of barrier phases on each
// id, so no phase is left open and no wait can be missed.
constexpr int kSelThreads = 128;                      // selection: 4 warps, an 8 x 8 block each
constexpr int kNBW = 8;                               // blend warps at most
constexpr int kBT = kSelThreads + 32 * kNBW;          // threads per CTA at most
constexpr int kItemEnd = -1;

// Barrier ids are immediates (2 + b or 4 + b picked by a branch on b), so
// the kernel uses barriers 0..5 only; nt = the CTA's thread count.
template <int ID>
__device__ __forceinline__ void bar_sync_id(int nt) {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(nt) : "memory");
}
template <int ID>
__device__ __forceinline__ void bar_arrive_id(int nt) {
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "r"(nt) : "memory");
}
__device__ __forceinline__ void full_sync(int b, int nt) { if (b) bar_sync_id<3>(nt); else bar_sync_id<2>(nt); }
__device__ __forceinline__ void full_arrive(int b, int nt) { if (b) bar_arrive_id<3>(nt); else bar_arrive_id<2>(nt); }
__device__ __forceinline__ void empty_sync(int b, int nt) { if (b) bar_sync_id<5>(nt); else bar_sync_id<4>(nt); }
__device__ __forceinline__ void empty_arrive(int b, int nt) { if (b) bar_arrive_id<5>(nt); else bar_arrive_id<4>(nt); }

__device__ __forceinline__ int find_view(const BatchView *views, int n_views, uint32_t item) {
    int lo = 0, hi = n_views;   // last view with tile_base <= item
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (views[mid].tile_base <= item) lo = mid; else hi = mid;
    }
    return lo;
}

// Dynamic shared memory: ids [2][256][KSB] int32, weights [2][256][KSB] float.
// QPL quads (4 channels) per lane per channel chunk, NCH chunks per row, EPL of
// a pixel group's G K entries per lane (lane l holds entries l, l + 32, ...), as
// in qr_blend's kernel.
template <int DT, int QPL, int G, int NCH, int EPL>
__global__ void __launch_bounds__(kBT, DT == QR_FP8E4M3 ? 1 : 2)
batch_kernel(const BatchView *__restrict__ views, int n_views, uint32_t total_items,
             uint32_t *__restrict__ counter, int KSB) {
    __shared__ SelStage st[kSelThreads / 32];
    __shared__ float s_thr[kKMax + 1];
    __shared__ int s_item[2];
    // per blend warp: row-weight table.  92 rows, not 96, for three entries per
    // lane: with K = 22 or 23 two CTAs share an SM's memory then
    constexpr int ROWS = EPL == 3 ? 92 : 32 * EPL;
    __shared__ __align__(16) float s_tw[kNBW][ROWS][G];
    __shared__ int s_tid[kNBW][ROWS];
    extern __shared__ __align__(16) unsigned char s_dyn[];
    int32_t *s_ids0 = reinterpret_cast<int32_t *>(s_dyn);
    float *s_w0 = reinterpret_cast<float *>(s_dyn) + 2 * kSelPix * KSB;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nt = int(blockDim.x), nbw = nt / 32 - kSelThreads / 32;
    select_boundaries(s_thr, views[0].K);   // the batch's views share K
    __syncthreads();

    if (warp < kSelThreads / 32) {
        // ------------------------------------------------ selection role
        for (int n = 0;; ++n) {
            const int b = n & 1;
            if (n >= 2) empty_sync(b, nt);   // the blend warps are done with buffer b
            if (threadIdx.x == 0) {
                const uint32_t it = atomicAdd(counter, 1u);
                s_item[b] = it < total_items ? int(it) : kItemEnd;
            }
            bar_sync_id<1>(kSelThreads);
            const int item = s_item[b];
            if (item == kItemEnd) {
                full_arrive(b, nt);
                if (n >= 1) empty_sync(b ^ 1, nt);   // the last tile's arrival
                break;
            }
            const BatchView &V = views[find_view(views, n_views, uint32_t(item))];
            const int K = V.K;
            int32_t *s_ids = s_ids0 + b * kSelPix * KSB;
            float *s_w = s_w0 + b * kSelPix * KSB;
            const int tile = item - int(V.tile_base);
            const int tile_w = V.tile_w, across = tile_w >> 3;
            // this warp's 8 x 8 block of the tile; slots are the tile's pixels
            const int bx = (warp % across) * 8, by = (warp / across) * 8;
            const int x0 = (tile % V.tiles_x) * tile_w + bx;
            const int y0 = (tile / V.tiles_x) * (kSelPix / tile_w) + by;
            const int blk = by * tile_w + bx;
            const int sa = blk + 2 * (lane >> 3) * tile_w + (lane & 7), sb = sa + tile_w;
            Walk w0, w1;
            select_block(V.rec_m, V.rec_w, V.rec_a, V.rec_h, V.igid, V.ranges[tile], V.W, V.H, x0,
                         y0, K, V.alpha_min, V.alpha_max, s_thr, st[warp], s_ids + sa * KSB,
                         s_w + sa * KSB, s_ids + sb * KSB, s_w + sb * KSB, w0, w1);
            finish_pixel(w0, K, s_ids + sa * KSB, s_w + sa * KSB);
            finish_pixel(w1, K, s_ids + sb * KSB, s_w + sb * KSB);
            __syncwarp();
            // ids, weights and counts are also written out for a backward pass
            store_block(V.W, V.H, x0, y0, K, V.vec != 0, s_ids, s_w,
                        [&](int x, int y) { return blk + y * tile_w + x; }, V.ids, V.w);
            const int px = x0 + (lane & 7), py = y0 + 2 * (lane >> 3);
            if (px < V.W && py < V.H) V.cnt[int64_t(py) * V.W + px] = uint8_t(w0.m);
            if (px < V.W && py + 1 < V.H) V.cnt[int64_t(py + 1) * V.W + px] = uint8_t(w1.m);
            full_arrive(b, nt);
        }
        return;
    }
    // ---------------------------------------------------- blend role
    constexpr int QB = Quad<DT>::B;
    constexpr int CQ = 32 * QPL;                 // quads of a channel chunk
    constexpr int ROWQ = CQ * NCH;               // quads of a row (C / 4)
    constexpr int U = QPL * QB >= 32 ? 2 : 4;    // rows in flight
    constexpr unsigned FULL = 0xffffffffu;
    const int bw = warp - kSelThreads / 32;
    for (int n = 0;; ++n) {
        const int b = n & 1;
        full_sync(b, nt);   // buffer b holds a selected tile (or the end marker)
        const int item = s_item[b];
        if (item == kItemEnd) break;
        const BatchView &V = views[find_view(views, n_views, uint32_t(item))];
        const int K = V.K;
        const int32_t *s_ids = s_ids0 + b * kSelPix * KSB;
        const float *s_w = s_w0 + b * kSelPix * KSB;
        const int tile = item - int(V.tile_base);
        const int tx = tile % V.tiles_x, ty = tile / V.tiles_x;
        const int tile_w = V.tile_w, tile_h = kSelPix / tile_w;
        const int half_w = tile_w / 2;
        const unsigned char *feat = V.feat;
        int mm[EPL], j[EPL];   // pixel of the group and entry that the lane holds
#pragma unroll
        for (int h = 0; h < EPL; ++h) {
            mm[h] = (lane + 32 * h) / K;
            j[h] = lane + 32 * h - mm[h] * K;
        }
        for (int gi = bw; gi < kSelPix / G; gi += nbw) {
            // pixel m of the group: place in the tile, number in the image (-1: none)
            auto pixel = [&](int m, int &loc) -> int64_t {
                int lx, ly;
                if (G == 4) { lx = 2 * (gi % half_w) + (m & 1); ly = 2 * (gi / half_w) + (m >> 1); }
                else if (G == 2) { lx = 2 * (gi % half_w) + m; ly = gi / half_w; }
                else { lx = gi % tile_w; ly = gi / tile_w; }
                loc = ly * tile_w + lx;
                const int px = tx * tile_w + lx, py = ty * tile_h + ly;
                int64_t p = -1;
                if (m < G && px < V.W && py < V.H) p = int64_t(py) * V.W + px;
                return p;
            };
            int64_t p = -1;   // pixel g in lane g K (one entry per lane) or g
            int id[EPL];
            float w[EPL];
#pragma unroll
            for (int h = 0; h < EPL; ++h) {
                int loc;
                const int64_t ph = pixel(mm[h], loc);
                if (EPL == 1) p = ph;
                id[h] = -1;
                w[h] = 0.f;
                if (ph >= 0) {
                    id[h] = s_ids[loc * KSB + j[h]];
                    w[h] = s_w[loc * KSB + j[h]];
                }
            }
            if (EPL > 1) {
                int loc;
                p = pixel(lane, loc);
            }
            // the G weights of each distinct row, gathered once (a pixel that
            // lists an id twice gets the sum)
            unsigned peers = __match_any_sync(FULL, id[0]);
            int leader = __ffs(peers) - 1;
            unsigned fresh = __ballot_sync(FULL, id[0] >= 0 && lane == leader);
            int nrows = __popc(fresh);
#pragma unroll
            for (int h = 0; h < EPL; ++h)
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (32 * h + 32 <= ROWS || lane + 32 * h < ROWS) s_tw[bw][lane + 32 * h][g] = 0.f;
            __syncwarp();
            if (id[0] >= 0) {
                const int slot = __popc(fresh & ((1u << leader) - 1u));
                atomicAdd(&s_tw[bw][slot][mm[0]], w[0]);
                if (lane == leader) s_tid[bw][slot] = id[0];
            }
            __syncwarp();
#pragma unroll
            for (int h = 1; h < EPL; ++h) {   // further entries: among the rows so far, or new ones
                int slot = -1;
                for (int k = 0; k < nrows; ++k)
                    if (s_tid[bw][k] == id[h]) slot = k;
                peers = __match_any_sync(FULL, id[h]);
                leader = __ffs(peers) - 1;
                fresh = __ballot_sync(FULL, id[h] >= 0 && slot < 0 && lane == leader);
                if (slot < 0) slot = nrows + __popc(fresh & ((1u << leader) - 1u));
                if (id[h] >= 0) {
                    atomicAdd(&s_tw[bw][slot][mm[h]], w[h]);
                    if ((fresh >> lane) & 1u) s_tid[bw][slot] = id[h];
                }
                nrows += __popc(fresh);
                __syncwarp();
            }
#pragma unroll 1
            for (int ch = 0; ch < NCH; ++ch) {   // the group's table serves every chunk
                float acc[G][QPL][4];
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int v = 0; v < QPL; ++v)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[g][v][q] = 0.f;
                const unsigned char *fch = feat + size_t(ch * CQ + lane) * QB;
                for (int r0 = 0; r0 < nrows; r0 += U) {
                    typename Quad<DT>::T r[U][QPL];
                    float sc[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const bool ok = r0 + u < nrows;
                        const int rid = ok ? s_tid[bw][r0 + u] : 0;
                        const unsigned char *row = fch + size_t(rid) * (size_t(ROWQ) * QB);
#pragma unroll
                        for (int v = 0; v < QPL; ++v)
                            r[u][v] = ok ? ld_quad<DT>(row + size_t(32 * v) * QB) : zero_quad<DT>();
                        if (DT == QR_FP8E4M3) sc[u] = ok ? V.fscale[rid] : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (r0 + u >= nrows) break;
                        float wg[G];
#pragma unroll
                        for (int g = 0; g < G; ++g)
                            wg[g] = DT == QR_FP8E4M3 ? s_tw[bw][r0 + u][g] * sc[u] : s_tw[bw][r0 + u][g];
                        float fv[QPL][4];
#pragma unroll
                        for (int v = 0; v < QPL; ++v) dec_quad<DT>(r[u][v], fv[v]);
#pragma unroll
                        for (int g = 0; g < G; ++g)
                            if (wg[g] != 0.f) {
#pragma unroll
                                for (int v = 0; v < QPL; ++v) {
                                    fma2b(acc[g][v] + 0, wg[g], fv[v][0], fv[v][1]);
                                    fma2b(acc[g][v] + 2, wg[g], fv[v][2], fv[v][3]);
                                }
                            }
                    }
                }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int64_t pg = __shfl_sync(FULL, p, EPL == 1 ? (g * K < 32 ? g * K : 0) : g);
                    if (pg >= 0) {
                        float4 *o = reinterpret_cast<float4 *>(V.out) + pg * int64_t(ROWQ) + ch * CQ + lane;
#pragma unroll
                        for (int v = 0; v < QPL; ++v)
                            st_cs(o + 32 * v, make_float4(acc[g][v][0], acc[g][v][1], acc[g][v][2],
                                                          acc[g][v][3]));
                    }
                }
            }
            __syncwarp();   // the table is rewritten by the next group
        }
        empty_arrive(b, nt);   // buffer b may be refilled
    }
}

template <int DT, int QT, int G, int NCH, int EPL = 1>
cudaError_t run_batch(const BatchView *dviews, int n_views, uint32_t total, uint32_t *counter,
                      int K, int nbw, int ctas_per_sm, cudaStream_t s) {
    auto kern = batch_kernel<DT, QT / NCH, G, NCH, EPL>;
    const int KSB = K | 1;
    const int nt = kSelThreads + 32 * nbw;
    const size_t dyn = size_t(KSB) * kSelPix * 2 * 8;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(dyn));
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int occ = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, nt, dyn);
    if (ctas_per_sm > 0 && ctas_per_sm < occ) occ = ctas_per_sm;
    if (occ < 1) occ = 1;
    const uint32_t grid = uint32_t(sms) * uint32_t(occ);
    kern<<<grid < total ? grid : total, nt, dyn, s>>>(dviews, n_views, total, counter, KSB);
    count_launch();
    return cudaGetLastError();
}

// Channel chunks per row by default: at most 2 quads (8 accumulators) per
// pixel and lane, so the blend warps fit the register budget of two CTAs
// per SM.
template <int QT>
constexpr int batch_default_chunks() {
    return QT <= 2 ? 1 : QT / 2;
}

// QT = C / 128 quads per lane over the whole row (1 .. 16).  group picks the
// pixel-group size (0 = 4), chunks the channel chunks per row for groups of 4
// and K <= 8 (0 = default; 1, 2, 4 where they divide QT and leave at most 4
// quads per lane).
template <int DT, int QT>
cudaError_t pick(const BatchView *d, int n, uint32_t total, uint32_t *counter, int K, int group,
                 int chunks, int nbw, int ctas, cudaStream_t s) {
    constexpr int DEF = batch_default_chunks<QT>();
    const int g = group > 0 ? group : 4;
    if (g == 4 && K > 8) {
        if (K <= 16) return run_batch<DT, QT, 4, DEF, 2>(d, n, total, counter, K, nbw, ctas, s);
        if (K <= 23) return run_batch<DT, QT, 4, DEF, 3>(d, n, total, counter, K, nbw, ctas, s);
        return run_batch<DT, QT, 4, DEF, 4>(d, n, total, counter, K, nbw, ctas, s);
    }
    if (g == 4) {
        const int c = chunks > 0 ? chunks : DEF;
        if constexpr (QT <= 4)
            if (c == 1) return run_batch<DT, QT, 4, 1>(d, n, total, counter, K, nbw, ctas, s);
        if constexpr (QT % 2 == 0 && QT <= 8)
            if (c == 2) return run_batch<DT, QT, 4, 2>(d, n, total, counter, K, nbw, ctas, s);
        if constexpr (QT % 4 == 0 && QT <= 16)
            if (c == 4) return run_batch<DT, QT, 4, 4>(d, n, total, counter, K, nbw, ctas, s);
        if (chunks > 0) return cudaErrorInvalidValue;
        return run_batch<DT, QT, 4, DEF>(d, n, total, counter, K, nbw, ctas, s);
    }
    if (g >= 2 && K <= 16) return run_batch<DT, QT, 2, DEF>(d, n, total, counter, K, nbw, ctas, s);
    return run_batch<DT, QT, 1, DEF>(d, n, total, counter, K, nbw, ctas, s);
}

}  // namespace

bool batch_supported(qr_dtype dt, int C) {
    const int cpv = dt == QR_F32 ? 4 : dt == QR_BF16 ? 8 : 16;
    if (C <= 0 || C % cpv) return false;
    const int rowv = C / cpv;
    return rowv == 32 || rowv == 64 || rowv == 128;
}

bool batch_chunks_ok(int C, int chunks) {
    const int qt = C / 128;
    return chunks == 0 || (qt % chunks == 0 && qt / chunks <= 4);
}

size_t batch_desc_bytes(int n_views) { return (size_t(n_views) * sizeof(BatchView) + 255) / 256 * 256 + 256; }

cudaError_t launch_batch(const void *ws, int n_views, uint32_t total_items, qr_dtype dt, int C,
                         int K, int group, int chunks, int blend_warps, int ctas_per_sm,
                         cudaStream_t s) {
    const int nbw = blend_warps > 0 ? blend_warps : kNBW;
    const BatchView *d = static_cast<const BatchView *>(ws);
    uint32_t *counter = reinterpret_cast<uint32_t *>(static_cast<char *>(const_cast<void *>(ws)) +
                                                     batch_desc_bytes(n_views) - 256);
    cudaError_t e = cudaMemsetAsync(counter, 0, 4, s);
    if (e != cudaSuccess) return e;
    const int qt = C / 128;   // quads per lane over the whole row
    auto by_qt = [&](auto dtc) -> cudaError_t {
        constexpr int DT = decltype(dtc)::value;
        switch (qt) {
            case 1: return pick<DT, 1>(d, n_views, total_items, counter, K, group, chunks, nbw, ctas_per_sm, s);
            case 2: return pick<DT, 2>(d, n_views, total_items, counter, K, group, chunks, nbw, ctas_per_sm, s);
            case 4: return pick<DT, 4>(d, n_views, total_items, counter, K, group, chunks, nbw, ctas_per_sm, s);
            case 8: return pick<DT, 8>(d, n_views, total_items, counter, K, group, chunks, nbw, ctas_per_sm, s);
            case 16: return pick<DT, 16>(d, n_views, total_items, counter, K, group, chunks, nbw, ctas_per_sm, s);
        }
        return cudaErrorInvalidValue;
    };
    switch (dt) {
        case QR_F32: return by_qt(std::integral_constant<int, QR_F32>());
        case QR_BF16: return by_qt(std::integral_constant<int, QR_BF16>());
        case QR_FP8E4M3: return by_qt(std::integral_constant<int, QR_FP8E4M3>());
    }
    return cudaErrorInvalidValue;
}

// Host side of qr_batch_prepare: build the descriptors and copy them to ws.
cudaError_t prepare_batch(const qr_view *views, int n_views, void *ws, uint32_t *total_items,
                          cudaStream_t s, BatchView *host_scratch) {
    uint32_t base = 0;
    for (int i = 0; i < n_views; ++i) {
        const qr_frame &f = *views[i].frame;
        BatchView &b = host_scratch[i];
        b.rec_m = slot<float4>(f, S_REC_M);
        b.rec_w = slot<float4>(f, S_REC_C);
        b.rec_a = slot<float>(f, S_REC_A);
        b.rec_h = slot<float>(f, S_REC_H);
        b.igid = slot<uint32_t>(f, S_IGID);
        b.ranges = slot<uint2>(f, S_RANGES);
        b.feat = static_cast<const unsigned char *>(views[i].feat);
        b.fscale = views[i].feat_scale;
        b.ids = views[i].ids;
        b.w = views[i].weights;
        b.cnt = views[i].counts;
        b.out = views[i].out;
        b.n_gauss = f.n;
        b.W = f.camera.width;
        b.H = f.camera.height;
        b.tile_w = f.params.tile_w;
        b.tiles_x = f.tiles_x;
        b.tiles_y = f.tiles_y;
        b.K = f.params.K;
        b.alpha_min = f.params.alpha_min;
        b.alpha_max = f.params.alpha_max;
        b.tile_base = base;
        b.vec = f.params.K % 4 == 0 &&
                ((reinterpret_cast<uintptr_t>(b.ids) | reinterpret_cast<uintptr_t>(b.w)) & 15) == 0;
        base += uint32_t(f.tiles_x * f.tiles_y);
    }
    *total_items = base;
    return cudaMemcpyAsync(ws, host_scratch, sizeof(BatchView) * size_t(n_views),
                           cudaMemcpyHostToDevice, s);
}

size_t batch_view_size() { return sizeof(BatchView); }

}  // namespace qr
