// K5a: the selection half of Algorithm 1 (Sec. 4.2, "sampling quantile
// Gaussians") for every pixel.
//
// Per pixel, front to back over its tile's depth-ordered list:
//   alpha' = min(alpha_max, alpha exp(-q/2)); entries with alpha' < alpha_min
//   are not members of I and leave T unchanged;
//   T_test = T (1 - alpha');
//   if T_test < tau_k (tau_k = (K-k)/(K+1), the boundary 1-(k+1)/(K+1)):
//       keep the Gaussian with weight w = T^Q alpha', T^Q *= 1 - alpha',
//       advance k past every boundary T_test is below;
//   stop once T_test < 1/(K+1); otherwise T = T_test.
// Outputs are the kept ids in depth order and the weights divided by
// 1 - T^Q (the normalisation step folded into the weights).  The same kernel
// serves App. C's Riemann-weight form (QR_RULE_RIEMANN): the same selection,
// each kept Gaussian weighted by the number of boundaries T_test crosses at
// it, divided by the number crossed in all.
//
// GB300 design: one warp per 8 x 8 pixel block or half of one (select_tile.cuh) and per CTA,
// so an SM takes a new block as soon as one is done.  Measured with K = 8
// (512-D VGA frames but for the last; CTAs of four warps walking a 16 x 16
// tile in step, 128 staged entries at a time -> now):
//   room, 500k Gaussians, 457 entries per tile       39.9 -> 22.9 us (issue)
//   object, 500k Gaussians, up to 5,166 entries       273 -> 110 us (longest lists)
//   room, 1M Gaussians at 1296 x 968                  126 -> 79 us
//   2,000 Gaussians at 128 x 128 (256 warps in all)  41.8 -> 18.8 us (latency)
// Two or four warps per CTA measured 0-5 % slower; a bound of 32 warps per SM
// (64 registers) instead of 24 cost up to 13 %.
// Where latency bounds it, a warp takes half a block (8 x 4 pixels, one per
// lane): each step of its chain is shorter, the list is culled twice as often.
// That is so for images of few blocks, and where walks are long: an object's
// silhouette, not a room, whose walks end at its surfaces.  The host knows
// neither; it takes a capacity of 2,048 entries per tile for long lists, but for
// K <= 8 on images so large that whole blocks fill the chip many times over.
// Whole blocks / halves, us, K = 8 and 16: 2,000 Gaussians at 128 x 128 25 / 17;
// VGA, object of 50k Gaussians (227 entries per tile) 52 / 49, 68 / 60, 200k (912)
// 87 / 75, 113 / 91, 500k (2,279) 135 / 122, 176 / 142; VGA, room of 500k (456) 39 / 41,
// 54 / 50, 2M (1,782) 42 / 46, 54 / 55; 1000 x 700, object of 500k 134 / 130, 176 / 156;
// 1296 x 968, room of 1M 92 / 116, 141 / 150, 3M 101 / 129, 154 / 168, object of 1M 201 /
// 216, 301 / 277.  So a guess that is wrong, as for a room with capacity to
// spare (render_frame's default of 8 entries per Gaussian), costs up to a
// tenth up to VGA.
// Halving only the blocks of long lists (the second halves' CTAs leave early
// elsewhere) cost 2-9 us wherever lists are short.
#include "select_tile.cuh"

namespace qr {
namespace {

// 8 x 8 blocks up to which blocks are halved; capacity per tile from which they
// are too, for K <= 8 up to kManyBlocks of them
constexpr int kSmallBlocks = 152 * 8;
constexpr int kManyBlocks = 152 * 100;
constexpr int64_t kLongLists = 2048;

// One CTA of one warp per 8 x (4 PX) pixels.
// kCount: App. C's Riemann weights in place of Algorithm 1's (select_block).
template <bool kCount, int PX>
__global__ void __launch_bounds__(32, 24)
select_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
              const float *__restrict__ rec_a, const float *__restrict__ rec_h,
              const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
              int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
              int32_t *__restrict__ ids, float *__restrict__ wout, uint8_t *__restrict__ cnt,
              int vec) {
    constexpr int N = 8 / PX;                                     // blocks per tile
    __shared__ SelStage st;
    __shared__ float s_thr[kKMax + 1];
    extern __shared__ unsigned char s_dyn[];
    const int KS = K | 1;
    const int lane = threadIdx.x & 31;
    int32_t *s_ids = reinterpret_cast<int32_t *>(s_dyn);          // [32 PX][KS]
    float *s_w = reinterpret_cast<float *>(s_dyn) + 32 * PX * KS;
    select_boundaries(s_thr, K);
    __syncthreads();
    pdl_wait();   // the predecessor's outputs are complete and visible
    const int tile = int(blockIdx.x) / N, part = int(blockIdx.x) % N, across = tile_w >> 3;
    const int x0 = (tile % tiles_x) * tile_w + (part % across) * 8;
    const int y0 = (tile / tiles_x) * (kSelPix / tile_w) + (part / across) * 4 * PX;
    const int px = x0 + (lane & 7), py = y0 + PX * (lane >> 3);
    const int sa = PX * (lane >> 3) * 8 + (lane & 7), sb = sa + 8;
    Walk w0, w1;
    if constexpr (PX == 2) {
        select_block<kCount>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[tile], W, H, x0, y0, K,
                             alpha_min, alpha_max, s_thr, st, s_ids + sa * KS, s_w + sa * KS,
                             s_ids + sb * KS, s_w + sb * KS, w0, w1);
        finish_pixel<kCount>(w1, K, s_ids + sb * KS, s_w + sb * KS);
    } else {
        select_block1<kCount>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[tile], W, H, x0, y0, K,
                              alpha_min, alpha_max, s_thr, st, s_ids + sa * KS, s_w + sa * KS, w0);
    }
    finish_pixel<kCount>(w0, K, s_ids + sa * KS, s_w + sa * KS);
    __syncwarp();
    store_block<32 * PX>(W, H, x0, y0, K, vec != 0, s_ids, s_w, [](int x, int y) { return y * 8 + x; }, ids, wout);
    if (px < W && py < H) cnt[int64_t(py) * W + px] = uint8_t(w0.m);
    if constexpr (PX == 2)
        if (px < W && py + 1 < H) cnt[int64_t(py + 1) * W + px] = uint8_t(w1.m);
}

}  // namespace

cudaError_t launch_select(const qr_frame &f, int32_t *ids, float *w, uint8_t *cnt, bool riemann,
                          cudaStream_t s) {
    const int tiles = num_tiles(f);
    if (tiles == 0) return cudaSuccess;
    const int K = f.params.K;
    const int vec = K % 4 == 0 && ((reinterpret_cast<uintptr_t>(ids) | reinterpret_cast<uintptr_t>(w)) & 15) == 0;
    auto go = [&](auto kern, int px) -> cudaError_t {
        return pdl_launch(kern, dim3(unsigned(tiles) * (8 / px)), dim3(32), size_t(K | 1) * 32 * px * 8, s,
                          (const float4 *)slot<float4>(f, S_REC_M),
                          (const float4 *)slot<float4>(f, S_REC_C),
                          (const float *)slot<float>(f, S_REC_A),
                          (const float *)slot<float>(f, S_REC_H),
                          (const uint32_t *)slot<uint32_t>(f, S_IGID),
                          (const uint2 *)slot<uint2>(f, S_RANGES), f.camera.width,
                          f.camera.height, f.params.tile_w, f.tiles_x, K, f.params.alpha_min,
                          f.params.alpha_max, ids, w, cnt, vec);
    };
    cudaError_t e;
    const bool many = K <= 8 && tiles * 4 > kManyBlocks;
    if (tiles * 4 <= kSmallBlocks || (!many && f.max_isect >= kLongLists * tiles))
        e = riemann ? go(select_kernel<true, 1>, 1) : go(select_kernel<false, 1>, 1);
    else
        e = riemann ? go(select_kernel<true, 2>, 2) : go(select_kernel<false, 2>, 2);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace qr
