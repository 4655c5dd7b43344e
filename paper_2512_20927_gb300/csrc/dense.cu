// K6: dense alpha compositing, Eq. 1 of the paper (V-Render, the plain method
// Q-Render is compared against):
//     out[p] = sum_i T_i alpha'_i f_i,   T_i = prod_{j<i} (1 - alpha'_j)
// over the pixel's whole depth-ordered list, with the same alpha' rules as the
// selection and a stop before the Gaussian whose test transmittance would
// fall below T_min.
//
// GB300 design: every pixel of a tile walks the same list, so the blend is a
// dense product W (pixels x entries) * F (entries x channels).  Rows of 64,
// 128, 256 or 512 channels go to dense_block_kernel (below: warp-specialised walk,
// row copies and accumulation over 8 x 8 pixel blocks).  Other widths use
// dense_kernel, 32 list entries at a time, where one CTA owns a screen tile
// and a 16/32/64-channel slice:
//   1. the batch's Gaussian records and feature-row slices are staged in
//      shared memory (coalesced 16-byte loads; BF16/FP8 widened here),
//   2. each thread walks its own pixel over the batch (scalar FP32, the exact
//      T recurrence) and writes the weights w = T alpha' to shared memory,
//   3. the accumulation runs as a register-tiled FP32 outer product (8 pixels
//      x 8 channels per thread for 64-channel slices), so every shared-memory
//      load feeds 8 FMAs.
// FP32 is kept on purpose: Eq. 1 is compared element by element with an FP64
// oracle, which a TF32/BF16 tensor-core product would not meet.
#include "quad.cuh"
#include "select_tile.cuh"
#include "tma.cuh"

namespace qr {
namespace {

constexpr int kThreads = 256;
constexpr int kBatch = 32;

template <int DT>
__device__ __forceinline__ void widen16(const uint4 v, float scale, float *o);

template <>
__device__ __forceinline__ void widen16<QR_F32>(const uint4 v, float, float *o) {
    o[0] = __uint_as_float(v.x); o[1] = __uint_as_float(v.y);
    o[2] = __uint_as_float(v.z); o[3] = __uint_as_float(v.w);
}
template <>
__device__ __forceinline__ void widen16<QR_BF16>(const uint4 v, float, float *o) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[2 * i] = __uint_as_float(u[i] << 16);
        o[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
    }
}
template <>
__device__ __forceinline__ void widen16<QR_FP8E4M3>(const uint4 v, float scale, float *o) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2_raw lo = __nv_cvt_fp8x2_to_halfraw2(__nv_fp8x2_storage_t(u[i] & 0xFFFFu), __NV_E4M3);
        const __half2_raw hi = __nv_cvt_fp8x2_to_halfraw2(__nv_fp8x2_storage_t(u[i] >> 16), __NV_E4M3);
        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&lo));
        const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&hi));
        o[4 * i] = a.x * scale; o[4 * i + 1] = a.y * scale;
        o[4 * i + 2] = b.x * scale; o[4 * i + 3] = b.y * scale;
    }
}
template <int DT> struct Cpv;
template <> struct Cpv<QR_F32> { static constexpr int v = 4; };
template <> struct Cpv<QR_BF16> { static constexpr int v = 8; };
template <> struct Cpv<QR_FP8E4M3> { static constexpr int v = 16; };

// CC channels per CTA; thread tile PX x CH with (256/PX) * (CC/CH) == 256.
template <int DT, int CC, int PX, int CH>
__global__ void __launch_bounds__(kThreads)
dense_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
              const float *__restrict__ rec_a, const float *__restrict__ rec_h,
             const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges,
             const unsigned char *__restrict__ feat, const float *__restrict__ fscale, int C,
             int W, int H, int tile_w, int tiles_x, float alpha_min, float alpha_max,
             float T_min, float *__restrict__ out, float *__restrict__ T_final) {
    static_assert((kThreads / PX) * (CC / CH) == kThreads, "thread tile");
    constexpr int CPV = Cpv<DT>::v;
    constexpr int ESZ = DT == QR_F32 ? 4 : DT == QR_BF16 ? 2 : 1;
    __shared__ float4 s_m[kBatch];
    __shared__ float4 s_c[kBatch];
    __shared__ float s_a[kBatch];
    __shared__ float s_h[kBatch];
    __shared__ __align__(16) float s_F[kBatch][CC];
    __shared__ __align__(16) float s_W[kBatch][kThreads];

    const int tile = blockIdx.x;
    const int c0 = blockIdx.y * CC;
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    const int tile_h = kThreads / tile_w;
    const int lx = threadIdx.x % tile_w, ly = threadIdx.x / tile_w;
    const int px = tx * tile_w + lx, py = ty * tile_h + ly;
    const bool inside = px < W && py < H;
    const float ux = float(px) + 0.5f, uy = float(py) + 0.5f;
    const uint2 range = ranges[tile];

    // GEMM roles
    constexpr int PG = kThreads / PX;  // pixel groups
    const int pg = threadIdx.x % PG, cg = threadIdx.x / PG;
    float acc[PX][CH];
#pragma unroll
    for (int i = 0; i < PX; ++i)
#pragma unroll
        for (int j = 0; j < CH; ++j) acc[i][j] = 0.f;

    float T = 1.0f;
    bool done = !inside;
    const size_t row_bytes = size_t(C) * ESZ;

    for (uint32_t b = range.x; b < range.y; b += kBatch) {
        if (__syncthreads_count(done) == kThreads) break;
        const int nb = int(min(uint32_t(kBatch), range.y - b));
        // stage records and feature slices
        if (threadIdx.x < nb) {
            const uint32_t g = isect_gid[b + threadIdx.x];
            s_m[threadIdx.x] = rec_m[g];
            s_c[threadIdx.x] = rec_w[g];
            s_a[threadIdx.x] = rec_a[g];
            s_h[threadIdx.x] = rec_h[g];
        }
        constexpr int VPR = CC / CPV;  // 16-byte vectors per row slice
        for (int i = threadIdx.x; i < kBatch * VPR; i += kThreads) {
            const int r = i / VPR, v = i % VPR;
            float tmp[CPV];
            if (r < nb) {
                const uint32_t g = isect_gid[b + r];
                const uint4 x = *reinterpret_cast<const uint4 *>(feat + size_t(g) * row_bytes +
                                                                 size_t(c0 + v * CPV) * ESZ);
                widen16<DT>(x, DT == QR_FP8E4M3 ? fscale[g] : 1.f, tmp);
            } else {
#pragma unroll
                for (int q = 0; q < CPV; ++q) tmp[q] = 0.f;
            }
#pragma unroll
            for (int q = 0; q < CPV; ++q) s_F[r][v * CPV + q] = tmp[q];
        }
        __syncthreads();
        // weights: thread = pixel, exact T recurrence
        for (int j = 0; j < kBatch; ++j) {
            float w = 0.f;
            if (!done && j < nb) {
                const float4 mm = s_m[j];
                const float4 cc = s_c[j];
                const PixelTerm pt = eval_half_q(ux, uy, mm, cc);
                const float a = pt.half_q > s_h[j] ? 0.f : eval_alpha(s_a[j], pt.half_q, alpha_max);
                if (a >= alpha_min) {
                    const float Tt = T * (1.0f - a);
                    if (T_min > 0.f && Tt < T_min) {
                        done = true;
                    } else {
                        w = T * a;
                        T = Tt;
                    }
                }
            }
            s_W[j][threadIdx.x] = w;
        }
        __syncthreads();
        // accumulate: acc[px][ch] += W[j][px] * F[j][ch]
        for (int j = 0; j < nb; ++j) {
            float wv[PX], fv[CH];
            if constexpr (PX % 4 == 0) {
#pragma unroll
                for (int i = 0; i < PX; i += 4) {
                    const float4 t = *reinterpret_cast<const float4 *>(&s_W[j][pg * PX + i]);
                    wv[i] = t.x; wv[i + 1] = t.y; wv[i + 2] = t.z; wv[i + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < PX; ++i) wv[i] = s_W[j][pg * PX + i];
            }
#pragma unroll
            for (int i = 0; i < CH; i += 4) {
                const float4 t = *reinterpret_cast<const float4 *>(&s_F[j][cg * CH + i]);
                fv[i] = t.x; fv[i + 1] = t.y; fv[i + 2] = t.z; fv[i + 3] = t.w;
            }
#pragma unroll
            for (int a = 0; a < PX; ++a)
#pragma unroll
                for (int c = 0; c < CH; ++c) acc[a][c] = fmaf(wv[a], fv[c], acc[a][c]);
        }
    }
    // write the slice
#pragma unroll
    for (int a = 0; a < PX; ++a) {
        const int t = pg * PX + a;
        const int qx = tx * tile_w + t % tile_w, qy = ty * tile_h + t / tile_w;
        if (qx < W && qy < H) {
            float *o = out + (int64_t(qy) * W + qx) * C + c0 + cg * CH;
#pragma unroll
            for (int c = 0; c < CH; c += 4)
                *reinterpret_cast<float4 *>(o + c) =
                    make_float4(acc[a][c], acc[a][c + 1], acc[a][c + 2], acc[a][c + 3]);
        }
    }
    if (T_final && blockIdx.y == 0 && inside) T_final[int64_t(py) * W + px] = T;
}

// ------------------------------------------------------------------ block kernel
// Rows of 64, 128, 256 or 512 channels.  One persistent CTA per SM; a work item is
// an 8 x 8 pixel block over all C channels, so each pixel's alpha' / T walk
// runs once.  The blend itself (8 pixels x C channels per group and kept
// entry) is bound by the FP32 pipe, so everything else runs beside it in
// warps of its own, far enough ahead that the consumers never wait for a walk
// or a row:
//   consumers (8 pixel groups of 4 x 2 pixels, WPG warps each): per kept entry
//     of their group 8 weights and 4 QPT channels per lane from shared memory,
//     8 x 4 QPT multiply-adds in packed FP32x2 instructions; a bit mask per
//     group and slot holds the entries with a nonzero weight in it;
//   producers (kProd warps, a block each in turn): walk_block's cull and
//     alpha', T, and w = T alpha'; the entries with a nonzero weight anywhere
//     in the block go, in list order, to the producer's ring of kSlots slots
//     of kEnt entries (weights, ids, group masks), a whole block ahead;
//   loader (1 warp): in consumption order, copies the rows of a slot's entries
//     as stored (cp.async.bulk, one copy per row) into a ring of kRows row
//     slots; BF16 / FP8 are widened in the consumers' registers.
// A producer that takes a block asks for the next one, which goes to the next
// producer: the launch of a CTA that has not begun is cancelled and its work
// taken over (clusterlaunchcontrol), so lists of very different lengths
// balance without a counter in memory.
// Every hand-over is an mbarrier with a bounded wait; a wait that runs out
// sets a flag that ends every role, the copies in flight are waited for, and
// the frame's status reports QR_ERR_DEVICE_TIMEOUT.
// Zero weights add nothing (fmaf(0, f, acc) == acc) and the entries are summed
// in list order, so the result equals dense_kernel's bit for bit.
// stats (nullable): [0] += blended (pixel, Gaussian) pairs, [1] += executed
// multiply-adds.
// Room VGA, 500k Gaussians, 512 FP32 channels (21.5 GFLOP useful, 1.1 times
// that executed): 1379 us with one CTA per 16 x 4 pixels that walked, staged
// rows and accumulated 32 list entries (9 survivors) at a time behind named
// barriers; 556 us now.  The roles alone: consumers 320 us at the FP32 peak,
// walk and copies without the multiply-adds 326 us.  Five warps per scheduler
// (20 in all) leave a consumer 96 registers; a 21st warp cost 80 and spills
// (1096 us), two producers 585 us.  Other rows (slices of 64 channels that walk
// again, or the 16 x 4 kernel -> now): room VGA C = 64 FP32 401 -> 332 us, C = 128
// FP8 757 -> 343 us; object VGA C = 256 BF16 1470 -> 813 us, C = 512 FP32 1752 ->
// 868 us; object 320 x 240 C = 64 BF16 585 -> 327 us; room 160 x 100 C = 64 47 ->
// 30 us.
constexpr int kProd = 3;                     // producer warps
constexpr int kSlots = 6;                    // weight slots per producer
constexpr int kEnt = 16;                     // entries per slot
constexpr int kRows = 4;                     // row slots
constexpr int kItemEnd = -1;
constexpr unsigned kDenseSpin = 1u << 26;    // polls of the waits for copies in flight

struct DenseSlot {
    float w[kEnt][kSelBlock];                // pixel slot 8 g + i of group g
    uint32_t gid[kEnt];
    uint32_t mask[8];                        // per group: entries with a nonzero weight
    int n, last, block;                      // entries; last slot of its block; block or kItemEnd
    int pad;
};
struct DenseRow {                            // what a row slot holds
    int slot, n, last, block;                // slot: producer * kSlots + weight slot
    float scale[kEnt];
};
struct DenseShared {
    DenseSlot slot[kProd][kSlots];
    DenseRow row[kRows];
    SelStage st[kProd];
    uint64_t w_full[kProd][kSlots], w_empty[kProd][kSlots];
    uint64_t r_full[kRows], r_empty[kRows];
    uint64_t mail_full[kProd], mail_empty[kProd], clc;
    alignas(16) uint4 response;
    int mail[kProd];
    int abort;
};
constexpr size_t kDenseShared = (sizeof(DenseShared) + 127) / 128 * 128;

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tma_smem_addr(bar)) : "memory");
}
// Wait bounded to `rounds` rounds of polls; false when it ran out or another role
// has given up.  (A round of a length known only at run time cost the kernel
// 5-15 us: the room below 557 -> 571.)
constexpr unsigned kPolls = 1024;
__device__ __forceinline__ bool dense_wait(uint64_t *bar, uint32_t parity, volatile int *abort,
                                           unsigned rounds) {
    for (unsigned i = 0; i < rounds; ++i) {
        if (tma_mbar_wait(bar, parity, kPolls)) return true;
        if (*abort) return false;
    }
    *abort = 1;
    return false;
}
__device__ __forceinline__ void bulk_row(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(tma_smem_addr(dst)), "l"(src), "r"(bytes), "r"(tma_smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void try_cancel(uint4 *response, uint64_t *bar) {
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 :: "r"(tma_smem_addr(response)), "r"(tma_smem_addr(bar)) : "memory");
}
// The CTA whose launch was cancelled, or -1 when none was left.
__device__ __forceinline__ int cancelled_cta(const uint4 *response) {
    int got, x;
    asm volatile("{\n .reg .b128 r;\n .reg .pred p;\n ld.shared.b128 r, [%2];\n"
                 " clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n"
                 " selp.s32 %0, 1, 0, p;\n mov.s32 %1, 0;\n"
                 " @p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, r;\n}\n"
                 : "=r"(got), "=r"(x) : "r"(tma_smem_addr(response)) : "memory");
    return got ? x : -1;
}

__device__ __forceinline__ void fma2d(float *acc, float w, float x0, float x1) {
    asm("{\n .reg .b64 a, ww, xx;\n mov.b64 a, {%0, %1};\n mov.b64 ww, {%2, %2};\n"
        " mov.b64 xx, {%3, %4};\n fma.rn.f32x2 a, ww, xx, a;\n mov.b64 {%0, %1}, a;\n}\n"
        : "+f"(acc[0]), "+f"(acc[1]) : "f"(w), "f"(x0), "f"(x1));
}

struct BlockPos {
    int tile, x0, y0;
};
__device__ __forceinline__ BlockPos dense_block(int block, int tile_w, int tiles_x) {
    const int tile = block >> 2, part = block & 3, across = tile_w >> 3;
    return {tile, (tile % tiles_x) * tile_w + (part % across) * 8,
            (tile / tiles_x) * (kSelPix / tile_w) + (part / across) * 8};
}

// Warps per pixel group and quads per lane of a row of C channels (64 channels
// leave half of a warp's lanes without one).
constexpr int dense_wpg(int C) { return C >= 256 ? 2 : 1; }
constexpr int dense_qpt(int C) { return C > 128 ? C / 256 : 1; }
constexpr int dense_threads(int C) { return 32 * (8 * dense_wpg(C) + kProd + 1); }

template <int DT, int C>
__global__ void __launch_bounds__(dense_threads(C), 1)
dense_block_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
                   const float *__restrict__ rec_a, const float *__restrict__ rec_h,
                   const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges,
                   const unsigned char *__restrict__ feat, const float *__restrict__ fscale, int W,
                   int H, int tile_w, int tiles_x, float alpha_min, float alpha_max, float T_min,
                   float *__restrict__ out, float *__restrict__ T_final,
                   unsigned long long *__restrict__ stats, uint32_t *__restrict__ counters,
                   unsigned rounds) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int QB = Quad<DT>::B;
    constexpr int WPG = dense_wpg(C), QPT = dense_qpt(C);
    constexpr uint32_t ROW = uint32_t(C / 4) * QB;           // bytes of a row
    constexpr int NCW = 8 * WPG;                             // consumer warps
    extern __shared__ __align__(128) unsigned char s_dyn[];
    DenseShared &sh = *reinterpret_cast<DenseShared *>(s_dyn);
    unsigned char *s_rows = s_dyn + kDenseShared;            // [kRows][kEnt][ROW]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int p = 0; p < kProd; ++p) {
            for (int s = 0; s < kSlots; ++s) {
                tma_mbar_init(&sh.w_full[p][s], 1);
                tma_mbar_init(&sh.w_empty[p][s], NCW);
            }
            tma_mbar_init(&sh.mail_full[p], 1);
            tma_mbar_init(&sh.mail_empty[p], 1);
        }
        for (int r = 0; r < kRows; ++r) {
            tma_mbar_init(&sh.r_full[r], 1);
            tma_mbar_init(&sh.r_empty[r], NCW);
        }
        tma_mbar_init(&sh.clc, 1);
        sh.abort = 0;
        sh.mail[0] = int(blockIdx.x);      // the first block, already delivered
        mbar_arrive(&sh.mail_full[0]);
        tma_fence_init();
    }
    __syncthreads();
    volatile int *abort = &sh.abort;

    if (warp < NCW) {
        // ------------------------------------------------------ consumers
        const int g = warp / WPG;
        const int q0 = ((warp % WPG) * 32 + lane) % (C / 4);   // first quad; then + 32 WPG
        const bool spare = C < 128 && lane >= C / 4;         // a lane without a quad of its own
        float acc[8][QPT][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int k = 0; k < QPT; ++k)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[i][k][c] = 0.f;
        unsigned long long n_exec = 0;
        for (uint32_t it = 0;; ++it) {
            const uint32_t r = it % kRows, ph = (it / kRows) & 1u;
            bool ok = dense_wait(&sh.r_full[r], ph, abort, rounds);
            const DenseRow &R = sh.row[r];
            const int block = ok ? R.block : kItemEnd, last = R.last, at = ok ? R.slot : 0;
            ok = block != kItemEnd;
            const DenseSlot &S = sh.slot[0][at];
            const unsigned char *rows = s_rows + size_t(r) * kEnt * ROW + size_t(q0) * QB;
            uint32_t mask = ok ? S.mask[g] : 0u;
            n_exec += __popc(mask);
            while (mask) {
                const int e = __ffs(mask) - 1;
                mask &= mask - 1u;
                const float4 *wr = reinterpret_cast<const float4 *>(&S.w[e][8 * g]);
                const float4 wa = wr[0], wb = wr[1];
                const float wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
                const float sc = DT == QR_FP8E4M3 ? R.scale[e] : 1.f;
#pragma unroll
                for (int k = 0; k < QPT; ++k) {
                    float f[4];
                    dec_quad<DT>(*reinterpret_cast<const typename Quad<DT>::T *>(rows + uint32_t(e) * ROW +
                                                                                 uint32_t(32 * WPG * k) * QB), f);
                    if constexpr (DT == QR_FP8E4M3) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) f[c] *= sc;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        fma2d(acc[i][k], wv[i], f[0], f[1]);
                        fma2d(acc[i][k] + 2, wv[i], f[2], f[3]);
                    }
                }
            }
            // one verdict per warp: its lanes go on, or leave, together
            if (!__all_sync(FULL, ok)) break;
            if (lane == 0) {
                mbar_arrive(&sh.r_empty[r]);
                mbar_arrive(&sh.w_empty[0][at]);
            }
            if (last) {
                const BlockPos b = dense_block(block, tile_w, tiles_x);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int x = b.x0 + (g & 1) * 4 + (i >> 1), y = b.y0 + (g >> 1) * 2 + (i & 1);
                    float4 *o = reinterpret_cast<float4 *>(out) + (int64_t(y) * W + x) * (C / 4) + q0;
#pragma unroll
                    for (int k = 0; k < QPT; ++k) {
                        if (x < W && y < H && !spare)
                            __stcs(o + 32 * WPG * k, make_float4(acc[i][k][0], acc[i][k][1], acc[i][k][2], acc[i][k][3]));
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[i][k][c] = 0.f;
                    }
                }
            }
        }
        if (stats && lane == 0) atomicAdd(&stats[1], n_exec * 8ull * (C / WPG));
    } else if (warp < NCW + kProd) {
        // ------------------------------------------------------ producers
        const int p = warp - NCW;
        SelStage &st = sh.st[p];
        uint32_t sc = 0;                   // slots begun
        int e = -1;                        // entries of the open slot, -1: none open
        uint32_t gmask = 0;                // lane g < 8: the open slot's mask of group g
        bool ok = true;
        auto open = [&]() {
            if (e >= 0) return;
            ok = ok && dense_wait(&sh.w_empty[p][sc % kSlots], ((sc / kSlots) & 1u) ^ 1u, abort, rounds);
            ok = __all_sync(FULL, ok);
            e = 0;
            gmask = 0;
        };
        auto commit = [&](int last, int block) {
            DenseSlot &S = sh.slot[p][sc % kSlots];
            if (lane < 8) S.mask[lane] = gmask;
            if (lane == 0) {
                S.n = e;
                S.last = last;
                S.block = block;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.w_full[p][sc % kSlots]);
            ++sc;
            e = -1;
        };
        for (uint32_t j = 0; ok; ++j) {
            ok = __all_sync(FULL, dense_wait(&sh.mail_full[p], j & 1u, abort, rounds));
            if (!ok) break;
            const int block = sh.mail[p];
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sh.mail_empty[p]);
                // the next producer's block (none is asked for after a refusal)
                const uint32_t i = j * kProd + uint32_t(p), p1 = (i + 1) % kProd;
                int next = kItemEnd;
                if (block != kItemEnd) {
                    // the previous response was read through the generic proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    tma_expect_tx(&sh.clc, 16);
                    try_cancel(&sh.response, &sh.clc);
                    ok = dense_wait(&sh.clc, i & 1u, abort, rounds);
                    if (ok) next = cancelled_cta(&sh.response);
                    else tma_mbar_wait(&sh.clc, i & 1u, kDenseSpin);   // it lands before the CTA exits
                }
                ok = ok && dense_wait(&sh.mail_empty[p1], (((i + 1) / kProd) & 1u) ^ 1u, abort, rounds);
                if (ok) {
                    sh.mail[p1] = next;
                    mbar_arrive(&sh.mail_full[p1]);
                }
            }
            ok = __all_sync(FULL, ok);
            if (!ok) break;
            if (block == kItemEnd) {
                open();
                if (ok) commit(1, kItemEnd);
                break;
            }
            const BlockPos b = dense_block(block, tile_w, tiles_x);
            const int px = b.x0 + (lane & 7), py = b.y0 + 2 * (lane >> 3);
            const bool in0 = px < W && py < H, in1 = px < W && py + 1 < H;
            // T over all members (below T_min for good once a pixel has stopped),
            // and over the blended ones
            float T0 = 1.0f, T1 = 1.0f, B0 = 1.0f, B1 = 1.0f;
            uint32_t n_blend = 0;
            auto visit = [&](int js, const float (&a)[4][2]) -> bool {
                float2 w[4];
                unsigned any[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float t0 = __fmul_rn(T0, __fsub_rn(1.0f, a[u][0])), t1 = __fmul_rn(T1, __fsub_rn(1.0f, a[u][1]));
                    const bool b0 = in0 && a[u][0] > 0.0f && !(t0 < T_min), b1 = in1 && a[u][1] > 0.0f && !(t1 < T_min);
                    w[u] = make_float2(b0 ? __fmul_rn(T0, a[u][0]) : 0.0f, b1 ? __fmul_rn(T1, a[u][1]) : 0.0f);
                    n_blend += uint32_t(b0) + uint32_t(b1);
                    T0 = t0;
                    T1 = t1;
                    B0 = b0 ? t0 : B0;
                    B1 = b1 ? t1 : B1;
                    any[u] = __ballot_sync(FULL, w[u].x != 0.0f || w[u].y != 0.0f);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (any[u] == 0u) continue;
                    open();
                    if (!ok) return false;
                    DenseSlot &S = sh.slot[p][sc % kSlots];
                    // lanes 4 g .. 4 g + 3 hold the 8 pixels of group g
                    reinterpret_cast<float2 *>(S.w[e])[lane] = w[u];
                    if (lane == 0) S.gid[e] = st.g[js + u];
                    if (lane < 8 && ((any[u] >> (4 * lane)) & 15u)) gmask |= 1u << e;
                    if (++e == kEnt) commit(0, block);
                }
                return !__all_sync(FULL, (T0 < T_min || !in0) && (T1 < T_min || !in1));
            };
            walk_block<false, 2>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[b.tile], W, H, b.x0, b.y0,
                              alpha_min, alpha_max, st, visit);
            __syncwarp();
            if (ok) open();
            if (!ok) break;
            commit(1, block);
            if (T_final) {
                if (in0) T_final[int64_t(py) * W + px] = B0;
                if (in1) T_final[int64_t(py + 1) * W + px] = B1;
            }
            if (stats && n_blend) atomicAdd(&stats[0], (unsigned long long)n_blend);
        }
    } else {
        // ------------------------------------------------------ loader
        uint32_t rc = 0;                   // row slots filled
        uint32_t sc[kProd] = {};           // slots taken per producer
        bool ok = true, end = false;
        while (ok && !end) {
#pragma unroll
            for (int p = 0; p < kProd; ++p) {
                for (bool last = false; ok && !end && !last;) {
                    const uint32_t s = sc[p] % kSlots, r = rc % kRows;
                    ok = __all_sync(FULL, dense_wait(&sh.w_full[p][s], (sc[p] / kSlots) & 1u, abort, rounds));
                    if (ok) ok = __all_sync(FULL, dense_wait(&sh.r_empty[r], ((rc / kRows) & 1u) ^ 1u, abort, rounds));
                    if (!ok) break;
                    ++sc[p];
                    ++rc;
                    const DenseSlot &S = sh.slot[p][s];
                    DenseRow &R = sh.row[r];
                    const int n = S.n;
                    last = S.last != 0;
                    end = S.block == kItemEnd;
                    if (lane == 0) {
                        R.slot = p * kSlots + int(s);
                        R.n = n;
                        R.last = S.last;
                        R.block = S.block;
                    }
                    const uint32_t gid = lane < n ? S.gid[lane] : 0u;
                    if (DT == QR_FP8E4M3 && lane < n) R.scale[lane] = fscale[gid];
                    __syncwarp();
                    if (lane == 0) tma_expect_tx(&sh.r_full[r], uint32_t(n) * ROW);
                    __syncwarp();
                    if (lane < n)
                        bulk_row(s_rows + (size_t(r) * kEnt + lane) * ROW, feat + size_t(gid) * ROW, ROW, &sh.r_full[r]);
                }
            }
        }
        // the copies issued last land before the CTA exits, whichever role gave
        // up and whenever it did
        for (uint32_t i = rc > kRows ? rc - kRows : 0; i < rc; ++i)
            tma_mbar_wait(&sh.r_full[i % kRows], (i / kRows) & 1u, kDenseSpin);
    }
    __syncthreads();
    if (threadIdx.x == 0 && *abort) atomicExch(&counters[CNT_STATUS], uint32_t(QR_ERR_DEVICE_TIMEOUT));
}

template <int DT, int C>
cudaError_t run_block(const qr_frame &f, const void *feat, const float *scale, float *out,
                      float *T_final, unsigned long long *stats, cudaStream_t s) {
    constexpr size_t dyn = kDenseShared + size_t(kRows) * kEnt * (C / 4) * Quad<DT>::B;
    static_assert(dyn <= 227 * 1024, "shared memory");
    cudaError_t e = cudaFuncSetAttribute(dense_block_kernel<DT, C>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, int(dyn));
    if (e != cudaSuccess) return e;
    dense_block_kernel<DT, C><<<unsigned(num_tiles(f)) * 4, dense_threads(C), dyn, s>>>(
        slot<float4>(f, S_REC_M), slot<float4>(f, S_REC_C), slot<float>(f, S_REC_A),
        slot<float>(f, S_REC_H), slot<uint32_t>(f, S_IGID), slot<uint2>(f, S_RANGES),
        static_cast<const unsigned char *>(feat), scale, f.camera.width, f.camera.height,
        f.params.tile_w, f.tiles_x, f.params.alpha_min, f.params.alpha_max, f.params.T_min, out,
        T_final, stats, slot<uint32_t>(f, S_COUNTERS), wait_limit() / kPolls);
    count_launch();
    return cudaGetLastError();
}

template <int DT, int CC, int PX, int CH>
cudaError_t run(const qr_frame &f, const void *feat, const float *scale, int C, float *out,
                float *T_final, cudaStream_t s) {
    dim3 grid(unsigned(num_tiles(f)), unsigned(C / CC));
    dense_kernel<DT, CC, PX, CH><<<grid, kThreads, 0, s>>>(
        slot<float4>(f, S_REC_M), slot<float4>(f, S_REC_C), slot<float>(f, S_REC_A), slot<float>(f, S_REC_H),
        slot<uint32_t>(f, S_IGID),
        slot<uint2>(f, S_RANGES), static_cast<const unsigned char *>(feat), scale, C, f.camera.width,
        f.camera.height, f.params.tile_w, f.tiles_x, f.params.alpha_min, f.params.alpha_max,
        f.params.T_min, out, T_final);
    count_launch();
    return cudaGetLastError();
}

template <int DT>
cudaError_t dispatch(const qr_frame &f, const void *feat, const float *scale, int C, float *out,
                     float *T_final, unsigned long long *stats, cudaStream_t s) {
    constexpr int cpv = Cpv<DT>::v;
    // the block kernel: one walk per pixel, culled and skipped entries.  It wants
    // C / 4 quads that fill the 32 or 64 lanes of a pixel group's warps (64
    // channels: half of them) and 64 rows in shared memory, so 64 to 512
    // channels; widths in between are not instantiated and walk every pixel once
    // per slice below (room 500k at 100 x 70: 192 channels 468 us, 256 120 us)
    if (C == 512) return run_block<DT, 512>(f, feat, scale, out, T_final, stats, s);
    if (C == 256) return run_block<DT, 256>(f, feat, scale, out, T_final, stats, s);
    if (C == 128) return run_block<DT, 128>(f, feat, scale, out, T_final, stats, s);
    if (C == 64) return run_block<DT, 64>(f, feat, scale, out, T_final, stats, s);
    if (C % 64 == 0) return run<DT, 64, 8, 8>(f, feat, scale, C, out, T_final, s);
    if (C % 32 == 0) return run<DT, 32, 8, 4>(f, feat, scale, C, out, T_final, s);
    if (C % 16 == 0) return run<DT, 16, 4, 4>(f, feat, scale, C, out, T_final, s);
    if constexpr (cpv <= 8)
        if (C % 8 == 0) return run<DT, 8, 2, 4>(f, feat, scale, C, out, T_final, s);
    if constexpr (cpv <= 4)
        if (C % 4 == 0) return run<DT, 4, 1, 4>(f, feat, scale, C, out, T_final, s);
    return cudaErrorInvalidValue;
}

}  // namespace

bool dense_supported(qr_dtype dt, int C) {
    const int cpv = dt == QR_F32 ? 4 : dt == QR_BF16 ? 8 : 16;
    return C > 0 && C % cpv == 0;
}

cudaError_t launch_dense(const qr_frame &f, const void *feat, const float *scale, qr_dtype dt,
                         int C, float *out, float *T_final, cudaStream_t s,
                         unsigned long long *stats) {
    if (num_tiles(f) == 0) return cudaSuccess;
    switch (dt) {
        case QR_F32: return dispatch<QR_F32>(f, feat, scale, C, out, T_final, stats, s);
        case QR_BF16: return dispatch<QR_BF16>(f, feat, scale, C, out, T_final, stats, s);
        case QR_FP8E4M3: return dispatch<QR_FP8E4M3>(f, feat, scale, C, out, T_final, stats, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace qr
