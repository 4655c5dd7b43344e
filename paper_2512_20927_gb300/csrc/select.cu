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
// GB300 design: one warp per 8 x 8 pixel block (select_tile.cuh) and per CTA,
// so an SM takes a new block as soon as one is done.  Measured with K = 8
// (512-D VGA frames but for the last; CTAs of four warps walking a 16 x 16
// tile in step, 128 staged entries at a time -> now):
//   room, 500k Gaussians, 457 entries per tile       39.9 -> 22.9 us (issue)
//   object, 500k Gaussians, up to 5,166 entries       273 -> 110 us (longest lists)
//   room, 1M Gaussians at 1296 x 968                  126 -> 79 us
//   2,000 Gaussians at 128 x 128 (256 warps in all)  41.8 -> 18.8 us (latency)
// Two or four warps per CTA measured 0-5 % slower; a bound of 32 warps per SM
// (64 registers) instead of 24 cost up to 13 %.
#include "select_tile.cuh"

namespace qr {
namespace {

constexpr int kSelWarps = 1;      // divides 4

// kCount: App. C's Riemann weights in place of Algorithm 1's (select_block).
template <bool kCount>
__global__ void __launch_bounds__(32 * kSelWarps, 24 / kSelWarps)
select_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
              const float *__restrict__ rec_a, const float *__restrict__ rec_h,
              const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
              int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
              int32_t *__restrict__ ids, float *__restrict__ wout, uint8_t *__restrict__ cnt,
              int vec) {
    __shared__ SelStage st[kSelWarps];
    __shared__ float s_thr[kKMax + 1];
    extern __shared__ unsigned char s_dyn[];
    const int KS = K | 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *s_ids = reinterpret_cast<int32_t *>(s_dyn) + warp * kSelBlock * KS;   // [64][KS] per warp
    float *s_w = reinterpret_cast<float *>(s_dyn) + (kSelWarps + warp) * kSelBlock * KS;
    select_boundaries(s_thr, K);
    __syncthreads();
    pdl_wait();   // the predecessor's outputs are complete and visible
    const int block = int(blockIdx.x) * kSelWarps + warp;
    const int tile = block >> 2, part = block & 3, across = tile_w >> 3;
    const int x0 = (tile % tiles_x) * tile_w + (part % across) * 8;
    const int y0 = (tile / tiles_x) * (kSelPix / tile_w) + (part / across) * 8;
    const int sa = (2 * (lane >> 3)) * 8 + (lane & 7), sb = sa + 8;
    Walk w0, w1;
    select_block<kCount>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[tile], W, H, x0, y0, K,
                         alpha_min, alpha_max, s_thr, st[warp], s_ids + sa * KS, s_w + sa * KS,
                         s_ids + sb * KS, s_w + sb * KS, w0, w1);
    finish_pixel<kCount>(w0, K, s_ids + sa * KS, s_w + sa * KS);
    finish_pixel<kCount>(w1, K, s_ids + sb * KS, s_w + sb * KS);
    __syncwarp();
    store_block(W, H, x0, y0, K, vec != 0, s_ids, s_w, [](int x, int y) { return y * 8 + x; }, ids, wout);
    const int px = x0 + (lane & 7), py = y0 + 2 * (lane >> 3);
    if (px < W && py < H) cnt[int64_t(py) * W + px] = uint8_t(w0.m);
    if (px < W && py + 1 < H) cnt[int64_t(py + 1) * W + px] = uint8_t(w1.m);
}

}  // namespace

cudaError_t launch_select(const qr_frame &f, int32_t *ids, float *w, uint8_t *cnt, bool riemann,
                          cudaStream_t s) {
    const int tiles = num_tiles(f);
    if (tiles == 0) return cudaSuccess;
    const int K = f.params.K;
    const size_t dyn = size_t(K | 1) * kSelBlock * kSelWarps * 8;
    const int vec = K % 4 == 0 && ((reinterpret_cast<uintptr_t>(ids) | reinterpret_cast<uintptr_t>(w)) & 15) == 0;
    auto go = [&](auto kern) -> cudaError_t {
        return pdl_launch(kern, dim3(unsigned(tiles) * 4 / kSelWarps), dim3(32 * kSelWarps), dyn, s,
                          (const float4 *)slot<float4>(f, S_REC_M),
                          (const float4 *)slot<float4>(f, S_REC_C),
                          (const float *)slot<float>(f, S_REC_A),
                          (const float *)slot<float>(f, S_REC_H),
                          (const uint32_t *)slot<uint32_t>(f, S_IGID),
                          (const uint2 *)slot<uint2>(f, S_RANGES), f.camera.width,
                          f.camera.height, f.params.tile_w, f.tiles_x, K, f.params.alpha_min,
                          f.params.alpha_max, ids, w, cnt, vec);
    };
    const cudaError_t e = riemann ? go(select_kernel<true>) : go(select_kernel<false>);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace qr
