// The selection half of Algorithm 1 for a block of 8 x 8 pixels by one warp,
// shared by the single-view selection kernel (select.cu) and the many-view
// persistent kernel (batch.cu), so both keep exactly the same Gaussians with
// the same FP32 weights.
//
// Per pixel, front to back over the tile's depth-ordered list:
//   alpha' = min(alpha_max, alpha exp(-q/2)); entries with alpha' < alpha_min
//   are not members of I and leave T unchanged;
//   T_test = T (1 - alpha');
//   if T_test < tau_k (tau_k = (K-k)/(K+1), the boundary 1-(k+1)/(K+1)):
//       keep the Gaussian with weight w = T^Q alpha', T^Q *= 1 - alpha',
//       advance k past every boundary T_test is below;
//   stop once T_test < 1/(K+1) = tau_{K-1}, i.e. when k reaches K; otherwise
//   T = T_test.
//
// What bounds it: instruction issue where every SM has its 24 warps (a VGA frame
// is little more than one wave), and the latency of the longest lists' chain
// of steps where it has not (a thumbnail, a silhouette tile).  Hence:
//   * A warp works alone: it owns an 8 x 8 block (two vertically adjacent
//     pixels per lane), stages the tile's list for itself and stops when its
//     own 64 pixels have stopped; no CTA barrier ties it to the other warps
//     of the tile, whose lists end elsewhere.  8 x 8 is the block with the
//     fewest entries within reach.
//   * Each lane holds one of 32 list entries in registers (the records of the
//     next 32 are loaded while these are used, the ids of the 32 after that
//     too), culls it against the block's box of pixel centres (the minimum of
//     q/2 over the box against the entry's reject bound), and only the
//     survivors (a fifth) go to shared memory, compacted in list order; up to
//     three left over are carried to the next 32, so the walk below always
//     takes four.
//   * Four survivors per step: eight independent alpha' (packed FP32x2 for
//     q/2; each half rounds like the scalar instruction), zero for entries
//     that are no members, then the four prefix products T (1 - alpha').  A
//     product with 1 - 0 is exact, so they are Algorithm 1's T_test, and T
//     never rises, so no boundary is crossed within the step unless the last
//     product is below the pixel's next boundary: one comparison per pixel
//     and one vote per step stand for the eight entry tests.  Only crossings
//     branch off, all pixels' first ones together, then their next ones; the
//     boundaries (K-k)/(K+1) come from a table.
// Kept (id, unnormalised weight) pairs go to per-pixel shared-memory slots of
// KS = K|1 entries; finish_block normalises and pads them, store_block writes
// them out.
#pragma once

#include "qr_internal.cuh"

namespace qr {

constexpr int kSelPix = 256;       // pixels per tile
constexpr int kSelBlock = 64;      // pixels per warp: 8 x 8
constexpr int kSelSurv = 36;       // survivors held: 3 carried + 32, rounded up to 4

// One warp's survivors.
struct SelStage {
    float4 m[kSelSurv];
    float4 c[kSelSurv];
    float2 ah[kSelSurv];
    uint32_t g[kSelSurv];
};

// Algorithm 1 state of one pixel: T, T^Q, the next boundary (-1 once k == K),
// boundaries passed, Gaussians kept.  k == K: the walk has stopped.
struct Walk {
    float T, TQ, thr;
    int k, m;
};

__device__ __forceinline__ float2 sel_add2(float2 a, float2 b) {
    float2 d;
    asm("{\n .reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
        " add.rn.f32x2 x, x, y;\n mov.b64 {%0, %1}, x;\n}\n"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 sel_mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n .reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
        " mul.rn.f32x2 x, x, y;\n mov.b64 {%0, %1}, x;\n}\n"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 sel_fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
        " mov.b64 z, {%6, %7};\n fma.rn.f32x2 x, x, y, z;\n mov.b64 {%0, %1}, x;\n}\n"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

// The boundaries tau_k = (K-k)/(K+1), k < K, and -1 behind them (K + 1
// entries in shared memory, written by the CTA's threads; the caller joins
// them before the walk).
__device__ __forceinline__ void select_boundaries(float *s_thr, int K) {
    for (int k = int(threadIdx.x); k <= K; k += int(blockDim.x))
        s_thr[k] = k < K ? __fdiv_rn(float(K - k), float(K + 1)) : -1.0f;
}

// A member entry whose T_test = Tt crosses the pixel's next boundary: keep
// it with weight T^Q alpha' (Algorithm 1), or with kCount the number of
// boundaries Tt crosses (App. C's right-Riemann weights), and advance k.
template <bool kCount>
__device__ __forceinline__ void walk_event(Walk &w, float Tt, float a, uint32_t gid,
                                           const float *s_thr, int32_t *ids, float *wts) {
    const int k0 = w.k;
    ids[w.m] = int32_t(gid);
    if constexpr (!kCount) wts[w.m] = w.TQ * a;
    w.TQ = w.TQ * (1.0f - a);
    do {
        w.thr = s_thr[++w.k];
    } while (Tt < w.thr);
    if constexpr (kCount) wts[w.m] = float(w.k - k0);
    ++w.m;
}

// Walks the block at (x0, y0) -- 8 x 8 pixels, or 8 x 4 with PX = 1 -- over
// isect_gid[range.x, range.y), the depth-ordered list of the tile that holds
// it.  All lanes of the warp call it.  Lane l owns the PX pixels from
// (x0 + l % 8, y0 + PX (l / 8)) down.  The survivors of the cull come four at
// a time, in list order: visit(j, a) with the alpha' of entries st.g[j .. j +
// 3] at the lane's pixels, a[u][i], 0 where an entry is no member (alpha' <
// alpha_min; alpha_min > 0), returns false once every pixel of the warp has
// stopped.  st.g holds Gaussian ids, or with kPos positions in isect_gid.
// The last step is filled up with entries out of reach, so the step's code
// stands in the kernel once (twice, its misses in the instruction cache
// bounded the larger callers).
template <bool kPos, int PX, typename Visit>
__device__ __forceinline__ void walk_block(
    const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
    const float *__restrict__ rec_a, const float *__restrict__ rec_h,
    const uint32_t *__restrict__ isect_gid, uint2 range, int W, int H, int x0, int y0,
    float alpha_min, float alpha_max, SelStage &st, Visit visit) {
    constexpr unsigned FULL = 0xffffffffu;
    if (x0 >= W || y0 >= H) return;
    const int lane = threadIdx.x & 31;
    const int px = x0 + (lane & 7), py = y0 + PX * (lane >> 3);
    const float ux = float(px) + 0.5f;
    const float2 uy = make_float2(float(py) + 0.5f, float(py + 1) + 0.5f);
    // the block's box of pixel centres inside the image
    const float bx0 = float(x0) + 0.5f, bx1 = float(min(x0 + 7, W - 1)) + 0.5f;
    const float by0 = float(y0) + 0.5f, by1 = float(min(y0 + 4 * PX - 1, H - 1)) + 0.5f;

    // four survivors from st[j]
    auto step4 = [&](int j) -> bool {
        float a[4][PX];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 mm = st.m[j + u];
            const float4 cc = st.c[j + u];
            const float2 ah = st.ah[j + u];
            if constexpr (PX == 1) {
                const float hq = eval_half_q(ux, uy.x, mm, cc).half_q;
                const float e = eval_alpha(ah.x, hq, alpha_max);
                a[u][0] = (hq > ah.y || e < alpha_min) ? 0.0f : e;
            } else {
                // eval_half_q for both pixels: dx shared, the rest packed
                const float dx = (ux - mm.x) - mm.z;
                const float2 dy = sel_add2(sel_add2(uy, make_float2(-mm.y, -mm.y)), make_float2(-mm.w, -mm.w));
                const float2 dx2 = make_float2(dx, dx);
                const float2 p1 = sel_fma2(dx2, make_float2(cc.x, cc.x), sel_mul2(dy, make_float2(cc.y, cc.y)));
                const float2 p2 = sel_fma2(dx2, make_float2(cc.z, cc.z), sel_mul2(dy, make_float2(cc.w, cc.w)));
                const float2 hq = sel_fma2(p1, p1, sel_mul2(p2, p2));
                const float e0 = eval_alpha(ah.x, hq.x, alpha_max), e1 = eval_alpha(ah.x, hq.y, alpha_max);
                a[u][0] = (hq.x > ah.y || e0 < alpha_min) ? 0.0f : e0;
                a[u][1] = (hq.y > ah.y || e1 < alpha_min) ? 0.0f : e1;
            }
        }
        return visit(j, a);
    };

    // entry base + lane of the list in registers; g1 / g2: its successors' ids
    uint32_t b = range.x + lane, g1 = 0, g2 = 0;
    float4 nm = make_float4(0.f, 0.f, 0.f, 0.f), nc = nm;
    float na = 0.f, nh = 0.f;
    if (b < range.y) {
        g1 = isect_gid[b];
        nm = rec_m[g1];
        nc = rec_w[g1];
        na = rec_a[g1];
        nh = rec_h[g1];
    }
    if (b + 32 < range.y) g2 = isect_gid[b + 32];
    int left = 0;
    for (uint32_t base = range.x; base < range.y; base += 32, b += 32) {
        const float4 cm = nm, cc = nc;
        const float ca = na, ch = nh;
        const uint32_t cg = g1;
        g1 = g2;
        if (b + 32 < range.y) {
            nm = rec_m[g1];
            nc = rec_w[g1];
            na = rec_a[g1];
            nh = rec_h[g1];
        }
        if (b + 64 < range.y) g2 = isect_gid[b + 64];
        // an entry whose q/2 stays above its reject bound over the whole box is
        // skipped by every pixel of the warp anyway
        const bool pass = b < range.y &&
                          !(box_min_half_q(cm, cc, bx0, bx1, by0, by1) * 0.999f > ch + 1e-3f);
        const unsigned bal = __ballot_sync(FULL, pass);
        if (pass) {
            const int i = left + __popc(bal & ((1u << lane) - 1u));
            st.m[i] = cm;
            st.c[i] = cc;
            st.ah[i] = make_float2(ca, ch);
            st.g[i] = kPos ? b : cg;
        }
        int n = left + __popc(bal);
        if (range.y - base <= 32) {   // the end of the list: fill up to a whole step
            if (lane < ((4 - n) & 3)) {
                st.m[n + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                st.c[n + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                st.ah[n + lane] = make_float2(0.f, -1.f);
                st.g[n + lane] = 0u;
            }
            n = (n + 3) & ~3;
        }
        const int full = n & ~3;
        __syncwarp();
        for (int j = 0; j < full; j += 4)
            if (!step4(j)) return;
        left = n - full;
        if (full) {   // the rest to the front (at most 3; sources lie behind them)
            __syncwarp();
            if (lane < left) {
                st.m[lane] = st.m[full + lane];
                st.c[lane] = st.c[full + lane];
                st.ah[lane] = st.ah[full + lane];
                st.g[lane] = st.g[full + lane];
            }
            __syncwarp();
        }
    }
}

// Algorithm 1 over the block (walk_block): the kept entries of a lane's two
// pixels go to ids0 / wts0 and ids1 / wts1 (K entries each) and their final
// states to w0, w1.
template <bool kCount = false>
__device__ __forceinline__ void select_block(
    const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
    const float *__restrict__ rec_a, const float *__restrict__ rec_h,
    const uint32_t *__restrict__ isect_gid, uint2 range, int W, int H, int x0, int y0, int K,
    float alpha_min, float alpha_max, const float *s_thr, SelStage &st, int32_t *ids0, float *wts0,
    int32_t *ids1, float *wts1, Walk &w0, Walk &w1) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int px = x0 + (lane & 7), py = y0 + 2 * (lane >> 3);
    const bool in0 = px < W && py < H, in1 = px < W && py + 1 < H;
    const float thr0 = s_thr[0];
    w0 = Walk{1.0f, 1.0f, in0 ? thr0 : -1.0f, in0 ? 0 : K, 0};
    w1 = Walk{1.0f, 1.0f, in1 ? thr0 : -1.0f, in1 ? 0 : K, 0};
    auto visit = [&](int j, const float (&a)[4][2]) -> bool {
        float2 t[4];
        float2 T = make_float2(w0.T, w1.T);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            T = sel_mul2(T, sel_add2(make_float2(1.0f, 1.0f), make_float2(-a[u][0], -a[u][1])));
            t[u] = T;
        }
        w0.T = T.x;
        w1.T = T.y;
        if (!__any_sync(FULL, T.x < w0.thr || T.y < w1.thr)) return true;
        // the first crossing of each pixel, then the next (rarely a third)
        do {
            if (T.x < w0.thr) {
                const int u = t[0].x < w0.thr ? 0 : t[1].x < w0.thr ? 1 : t[2].x < w0.thr ? 2 : 3;
                const float e = u == 0 ? a[0][0] : u == 1 ? a[1][0] : u == 2 ? a[2][0] : a[3][0];
                const float Tt = u == 0 ? t[0].x : u == 1 ? t[1].x : u == 2 ? t[2].x : t[3].x;
                walk_event<kCount>(w0, Tt, e, st.g[j + u], s_thr, ids0, wts0);
            }
            if (T.y < w1.thr) {
                const int u = t[0].y < w1.thr ? 0 : t[1].y < w1.thr ? 1 : t[2].y < w1.thr ? 2 : 3;
                const float e = u == 0 ? a[0][1] : u == 1 ? a[1][1] : u == 2 ? a[2][1] : a[3][1];
                const float Tt = u == 0 ? t[0].y : u == 1 ? t[1].y : u == 2 ? t[2].y : t[3].y;
                walk_event<kCount>(w1, Tt, e, st.g[j + u], s_thr, ids1, wts1);
            }
        } while (__any_sync(FULL, T.x < w0.thr || T.y < w1.thr));
        return !__all_sync(FULL, w0.k == K && w1.k == K);
    };
    walk_block<false, 2>(rec_m, rec_w, rec_a, rec_h, isect_gid, range, W, H, x0, y0, alpha_min, alpha_max,
                      st, visit);
}

// The same over an 8 x 4 block, one pixel per lane.
template <bool kCount = false>
__device__ __forceinline__ void select_block1(
    const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
    const float *__restrict__ rec_a, const float *__restrict__ rec_h,
    const uint32_t *__restrict__ isect_gid, uint2 range, int W, int H, int x0, int y0, int K,
    float alpha_min, float alpha_max, const float *s_thr, SelStage &st, int32_t *ids, float *wts, Walk &w) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool inside = x0 + (lane & 7) < W && y0 + (lane >> 3) < H;
    w = Walk{1.0f, 1.0f, inside ? s_thr[0] : -1.0f, inside ? 0 : K, 0};
    auto visit = [&](int j, const float (&a)[4][1]) -> bool {
        float t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) t[u] = w.T = __fmul_rn(w.T, __fsub_rn(1.0f, a[u][0]));
        if (!__any_sync(FULL, w.T < w.thr)) return true;
        do {
            if (w.T < w.thr) {
                const int u = t[0] < w.thr ? 0 : t[1] < w.thr ? 1 : t[2] < w.thr ? 2 : 3;
                const float e = u == 0 ? a[0][0] : u == 1 ? a[1][0] : u == 2 ? a[2][0] : a[3][0];
                const float Tt = u == 0 ? t[0] : u == 1 ? t[1] : u == 2 ? t[2] : t[3];
                walk_event<kCount>(w, Tt, e, st.g[j + u], s_thr, ids, wts);
            }
        } while (__any_sync(FULL, w.T < w.thr));
        return !__all_sync(FULL, w.k == K);
    };
    walk_block<false, 1>(rec_m, rec_w, rec_a, rec_h, isect_gid, range, W, H, x0, y0, alpha_min, alpha_max,
                         st, visit);
}

// A pixel's kept weights divided by 1 - T^Q (kCount: by the boundaries crossed
// in all), the rest of its K slots padded with id -1 and weight 0.
template <bool kCount = false>
__device__ __forceinline__ void finish_pixel(const Walk &w, int K, int32_t *ids, float *wts) {
    const float D = kCount ? float(w.k) : 1.0f - w.TQ;
    for (int j = 0; j < w.m; ++j) wts[j] = __fdiv_rn(wts[j], D);
    for (int j = w.m; j < K; ++j) {
        ids[j] = -1;
        wts[j] = 0.0f;
    }
}

// Writes a finished array of the block at (x0, y0) (K entries per pixel, of
// pixel (x, y) at slot_of(x, y) KS in shared memory) to the image's array; the
// warp's lanes must have finished their pixels (__syncwarp between).  Rows of
// a block are 8 K consecutive entries of the image; vec (K % 4 == 0 and
// 16-byte aligned outputs) writes them four at a time.
template <int NPIX, typename SlotOf, typename Put>
__device__ __forceinline__ void for_block(int W, int H, int x0, int y0, int K, bool vec,
                                          SlotOf slot_of, Put put) {
    const int lane = threadIdx.x & 31;
    const int KS = K | 1;
    const int per = vec ? 4 : 1;
    const int KP = K / per;                        // units per pixel
    const uint32_t inv = (65536u + uint32_t(KP) - 1u) / uint32_t(KP);   // e / KP, e < 64 KP <= 2048
    for (int e = lane; e < NPIX * KP; e += 32) {
        const int pix = int((uint32_t(e) * inv) >> 16), j = (e - pix * KP) * per;
        const int x = x0 + (pix & 7), y = y0 + (pix >> 3);
        if (x >= W || y >= H) continue;
        put(slot_of(pix & 7, pix >> 3) * KS + j, (int64_t(y) * W + x) * K + j);
    }
}
template <int NPIX = kSelBlock, typename SlotOf>
__device__ __forceinline__ void store_block(int W, int H, int x0, int y0, int K, bool vec,
                                            const int32_t *s_ids, const float *s_w, SlotOf slot_of,
                                            int32_t *__restrict__ ids, float *__restrict__ wout) {
    for_block<NPIX>(W, H, x0, y0, K, vec, slot_of, [&](int at, int64_t o) {
        if (vec) {
            *reinterpret_cast<int4 *>(ids + o) = make_int4(s_ids[at], s_ids[at + 1], s_ids[at + 2], s_ids[at + 3]);
            *reinterpret_cast<float4 *>(wout + o) = make_float4(s_w[at], s_w[at + 1], s_w[at + 2], s_w[at + 3]);
        } else {
            ids[o] = s_ids[at];
            wout[o] = s_w[at];
        }
    });
}

}  // namespace qr
