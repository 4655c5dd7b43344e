// The two other select rules of the paper, behind the same outputs as the
// Algorithm 1 selection (ids [P][K] in depth order, normalised weights
// [P][K], counts [P]), so the blend serves all three:
//
//   top-K (Sec. 4.2 and the complexity table, the renderer Q-Render is
//   compared against): the K largest Eq. 1 weights w = T alpha' of the dense
//   walk (same alpha' rules, stop before T would fall below T_min), equal
//   weights keeping the earlier entry, blended with their weights divided by
//   the kept sum;
//
//   Stratified-K (App. E): pass 1 walks the list as Eq. 1 does and takes the
//   mean mu and standard deviation sigma of the transmittances after each
//   blended Gaussian; the K boundaries are spaced uniformly in the
//   probability of N(mu, sigma^2) over the transmittance interval [0, 1]
//   and mapped back (tau_k = mu + sigma Phi^-1(u_lo + (u_hi - u_lo)(1 -
//   k/(K+1))), u_lo = Phi(-mu/sigma), u_hi = Phi((1-mu)/sigma)); pass 2 is
//   Algorithm 1 with tau_k in place of 1 - k/(K+1).
//
// (App. C's Riemann-weight form of Algorithm 1 keeps Algorithm 1's
// selection, so it runs in the selection kernel itself, select.cu.)
//
// GB300 design: one warp per 8 x 8 pixel block, two pixels per lane, on the
// selection's walk (walk_block in select_tile.cuh: the warp culls the list
// for its own block and takes the survivors four at a time), so a warp stops
// when its own 64 pixels have and no CTA barrier ties it to others.  alpha'
// and the transmittance are evaluated as the dense blend does, so the walks
// agree with it bit for bit.
//   * top-K keeps its candidates in per-pixel shared-memory slots (weight and
//     list position); a strictly larger weight replaces the smallest (latest
//     among equal) one.  A step of four entries is passed over with one vote
//     unless some weight exceeds its pixel's smallest kept one; the warp's
//     first candidates then enter together, then their next ones.  The
//     smallest is found again over the minima of groups of four slots, of
//     which only the changed group is rescanned (K / 4 + 4 reads instead of
//     K).  Once fl(T alpha_max) is no larger than the smallest kept weight,
//     no later entry can enter (T only falls and alpha' <= alpha_max), so the
//     pixel stops early without changing the result.
//   * Stratified-K sums T and T^2 in compensated double-FP32 arithmetic, both
//     pixels of a lane in one packed FP32x2 instruction stream (adding an
//     exact 0 where an entry is no member), forms mu and sigma from them, and
//     the boundaries with the FP32 normal CDF and its inverse (normcdff,
//     normcdfinvf); the boundaries sit in shared memory for pass 2, which
//     re-walks the list as the selection does.
// Bound by instruction issue (room) and by the longest lists' chains (object).
// Measured (CTAs of eight warps walking a tile in step, one pixel per lane ->
// now): Stratified-K, room VGA, K = 8: 183 -> 139 us; top-K, object 517 x 389,
// 200k Gaussians, K = 16: 315 -> 238 us.
#include "select_tile.cuh"

namespace qr {
namespace {

enum { kTopK = 1, kStratified = 2 };

// ------------------------------------------------------------------ top-K
constexpr int kGroups = kKMax / 4;

// One pixel's walk: slots key[j 64] / w[j 64], j < K, and the group minima
// gw[g 64], gs[g 64] (weight and slot).  wmin: smallest kept weight, below 0
// until K are kept (every member enters), +inf once the pixel has stopped;
// wstop: the bound fl(T alpha_max) is compared with, -1 where it never is.
struct Top {
    float T, wmin, wstop;
    int m, smin;
};

__device__ __forceinline__ bool slot_less(float wa, int a, float wb, int b, const uint32_t *key) {
    return wa < wb || (wa == wb && key[a * kSelBlock] > key[b * kSelBlock]);
}
__device__ __forceinline__ void rescan_group(int g, int K, const uint32_t *key, const float *w,
                                             float *gw, int32_t *gs) {
    const int j0 = 4 * g;
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = j0 + i < K ? w[(j0 + i) * kSelBlock] : INFINITY;
    int s = j0;
    float b = v[0];
#pragma unroll
    for (int i = 1; i < 4; ++i)
        if (j0 + i < K && slot_less(v[i], j0 + i, b, s, key)) {
            s = j0 + i;
            b = v[i];
        }
    gw[g * kSelBlock] = b;
    gs[g * kSelBlock] = s;
}

// Keeps the member entry at list position pos with weight x > t.wmin.
__device__ __forceinline__ void top_insert(Top &t, int K, uint32_t pos, float x, uint32_t *key, float *w,
                                           float *gw, int32_t *gs) {
    const int G = (K + 3) >> 2;
    const int s = t.m < K ? t.m : t.smin;
    key[s * kSelBlock] = pos;
    w[s * kSelBlock] = x;
    if (t.m < K) {
        if (++t.m < K) return;
        for (int g = 0; g < G; ++g) rescan_group(g, K, key, w, gw, gs);
    } else {
        rescan_group(s >> 2, K, key, w, gw, gs);
    }
    float b = gw[0];
    int bs = gs[0];
    for (int g = 1; g < G; ++g) {
        const float v = gw[g * kSelBlock];
        const int vs = gs[g * kSelBlock];
        if (slot_less(v, vs, b, bs, key)) {
            b = v;
            bs = vs;
        }
    }
    t.wmin = t.wstop = b;
    t.smin = bs;
}

// Depth order (list position), the kept sum in that order, weights divided by
// it, Gaussian ids in place of positions, the rest padded.
__device__ __forceinline__ void top_finish(const Top &t, int K, const uint32_t *__restrict__ isect_gid,
                                           uint32_t *key, float *w) {
    for (int i = 1; i < t.m; ++i) {
        const uint32_t kk = key[i * kSelBlock];
        const float ww = w[i * kSelBlock];
        int j = i;
        while (j > 0 && key[(j - 1) * kSelBlock] > kk) {
            key[j * kSelBlock] = key[(j - 1) * kSelBlock];
            w[j * kSelBlock] = w[(j - 1) * kSelBlock];
            --j;
        }
        key[j * kSelBlock] = kk;
        w[j * kSelBlock] = ww;
    }
    float D = 0.0f;
    for (int j = 0; j < t.m; ++j) D = __fadd_rn(D, w[j * kSelBlock]);
    for (int j = 0; j < K; ++j) {
        key[j * kSelBlock] = j < t.m ? isect_gid[key[j * kSelBlock]] : 0xFFFFFFFFu;
        w[j * kSelBlock] = j < t.m ? __fdiv_rn(w[j * kSelBlock], D) : 0.0f;
    }
}

// The K entries of the block's pixels (slot of pixel (x, y): the lane's first
// or second 32) written to the image.
template <typename T>
__device__ __forceinline__ void store_slots(int W, int H, int x0, int y0, int K, bool vec, const T *s,
                                            T *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int per = vec ? 4 : 1;
    const int KP = K / per;
    const uint32_t inv = (65536u + uint32_t(KP) - 1u) / uint32_t(KP);   // e / KP, e < 64 KP <= 2048
    for (int e = lane; e < kSelBlock * KP; e += 32) {
        const int pix = int((uint32_t(e) * inv) >> 16), j = (e - pix * KP) * per;
        const int x = pix & 7, y = pix >> 3;
        if (x0 + x >= W || y0 + y >= H) continue;
        const T *v = s + j * kSelBlock + (y & 1) * 32 + (y >> 1) * 8 + x;
        T *o = out + (int64_t(y0 + y) * W + x0 + x) * K + j;
        if (vec) {
            struct alignas(16) V4 { T a, b, c, d; };
            *reinterpret_cast<V4 *>(o) = V4{v[0], v[kSelBlock], v[2 * kSelBlock], v[3 * kSelBlock]};
        } else {
            *o = *v;
        }
    }
}

struct BlockAt {
    int tile, x0, y0;
};
__device__ __forceinline__ BlockAt block_at(int block, int tile_w, int tiles_x) {
    const int tile = block >> 2, part = block & 3, across = tile_w >> 3;
    return {tile, (tile % tiles_x) * tile_w + (part % across) * 8,
            (tile / tiles_x) * (kSelPix / tile_w) + (part / across) * 8};
}

// Shared memory per warp: slots of 64 pixels, entry-major ([j][64], so a
// lane's accesses fall in its own bank whatever K is).
__global__ void __launch_bounds__(32, 24)
topk_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
            const float *__restrict__ rec_a, const float *__restrict__ rec_h,
            const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
            int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
            float T_min, int32_t *__restrict__ ids, float *__restrict__ wout,
            uint8_t *__restrict__ cnt, int vec) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ SelStage st;
    extern __shared__ unsigned char s_dyn[];
    const int lane = threadIdx.x & 31;
    const int G = (K + 3) >> 2;
    uint32_t *s_key = reinterpret_cast<uint32_t *>(s_dyn);       // [K][64]
    float *s_w = reinterpret_cast<float *>(s_key + K * kSelBlock);   // [K][64]
    float *s_gw = s_w + K * kSelBlock;                           // [G][64]
    int32_t *s_gs = reinterpret_cast<int32_t *>(s_gw + G * kSelBlock);   // [G][64]
    pdl_wait();   // the predecessor's outputs are complete and visible
    const BlockAt at = block_at(int(blockIdx.x), tile_w, tiles_x);
    const int px = at.x0 + (lane & 7), py = at.y0 + 2 * (lane >> 3);
    const bool in0 = px < W && py < H, in1 = px < W && py + 1 < H;
    Top p0{1.0f, in0 ? -0.5f : INFINITY, -1.0f, 0, 0}, p1{1.0f, in1 ? -0.5f : INFINITY, -1.0f, 0, 0};
    // T below this stops the pixel and is no member (never when T_min is 0)
    const float T_end = T_min;
    auto visit = [&](int j, const float (&a0)[4], const float (&a1)[4]) -> bool {
        float w0[4], w1[4];
        float t0 = p0.T, t1 = p1.T;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            // weight T alpha' of an entry that may enter, -1 of any other
            const float n0 = __fmul_rn(t0, __fsub_rn(1.0f, a0[u])), n1 = __fmul_rn(t1, __fsub_rn(1.0f, a1[u]));
            w0[u] = a0[u] > 0.0f && !(n0 < T_end) ? __fmul_rn(t0, a0[u]) : -1.0f;
            w1[u] = a1[u] > 0.0f && !(n1 < T_end) ? __fmul_rn(t1, a1[u]) : -1.0f;
            t0 = n0;
            t1 = n1;
        }
        p0.T = t0;
        p1.T = t1;
        float b0 = fmaxf(fmaxf(w0[0], w0[1]), fmaxf(w0[2], w0[3]));
        float b1 = fmaxf(fmaxf(w1[0], w1[1]), fmaxf(w1[2], w1[3]));
        while (__any_sync(FULL, b0 > p0.wmin || b1 > p1.wmin)) {
            if (b0 > p0.wmin) {
                const int u = w0[0] > p0.wmin ? 0 : w0[1] > p0.wmin ? 1 : w0[2] > p0.wmin ? 2 : 3;
                const float x = u == 0 ? w0[0] : u == 1 ? w0[1] : u == 2 ? w0[2] : w0[3];
                top_insert(p0, K, st.g[j + u], x, s_key + lane, s_w + lane, s_gw + lane, s_gs + lane);
                // this entry and those before it are settled
                w0[0] = -1.0f;
                w0[1] = u >= 1 ? -1.0f : w0[1];
                w0[2] = u >= 2 ? -1.0f : w0[2];
                w0[3] = u >= 3 ? -1.0f : w0[3];
                b0 = fmaxf(fmaxf(w0[1], w0[2]), w0[3]);
            }
            if (b1 > p1.wmin) {
                const int u = w1[0] > p1.wmin ? 0 : w1[1] > p1.wmin ? 1 : w1[2] > p1.wmin ? 2 : 3;
                const float x = u == 0 ? w1[0] : u == 1 ? w1[1] : u == 2 ? w1[2] : w1[3];
                top_insert(p1, K, st.g[j + u], x, s_key + 32 + lane, s_w + 32 + lane, s_gw + 32 + lane,
                           s_gs + 32 + lane);
                w1[0] = -1.0f;
                w1[1] = u >= 1 ? -1.0f : w1[1];
                w1[2] = u >= 2 ? -1.0f : w1[2];
                w1[3] = u >= 3 ? -1.0f : w1[3];
                b1 = fmaxf(fmaxf(w1[1], w1[2]), w1[3]);
            }
        }
        if (t0 < T_end || __fmul_rn(t0, alpha_max) <= p0.wstop) p0.wmin = INFINITY;
        if (t1 < T_end || __fmul_rn(t1, alpha_max) <= p1.wstop) p1.wmin = INFINITY;
        return !__all_sync(FULL, p0.wmin == INFINITY && p1.wmin == INFINITY);
    };
    walk_block<true>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[at.tile], W, H, at.x0, at.y0, alpha_min,
                     alpha_max, st, visit);
    top_finish(p0, K, isect_gid, s_key + lane, s_w + lane);
    top_finish(p1, K, isect_gid, s_key + 32 + lane, s_w + 32 + lane);
    __syncwarp();
    store_slots(W, H, at.x0, at.y0, K, vec != 0, reinterpret_cast<const int32_t *>(s_key), ids);
    store_slots(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_w, wout);
    if (in0) cnt[int64_t(py) * W + px] = uint8_t(p0.m);
    if (in1) cnt[int64_t(py + 1) * W + px] = uint8_t(p1.m);
}

// ------------------------------------------------------------------ Stratified-K
// Compensated sums of two pixels at a time (qr_internal.cuh's df operations,
// packed: each half rounds like the scalar instruction).
struct df2 {
    float2 hi, lo;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return sel_fma2(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ df2 two_sum2(float2 a, float2 b) {
    const float2 s = sel_add2(a, b);
    const float2 bb = sub2(s, a);
    return {s, sel_add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ df2 fast_two_sum2(float2 a, float2 b) {
    const float2 s = sel_add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ df2 df2_add(df2 a, df2 b) {
    df2 s = two_sum2(a.hi, b.hi);
    const df2 t = two_sum2(a.lo, b.lo);
    s.lo = sel_add2(s.lo, t.hi);
    s = fast_two_sum2(s.hi, s.lo);
    s.lo = sel_add2(s.lo, t.lo);
    return fast_two_sum2(s.hi, s.lo);
}
__device__ __forceinline__ df2 df2_add_f(df2 a, float2 b) {
    df2 s = two_sum2(a.hi, b);
    s.lo = sel_add2(s.lo, a.lo);
    return fast_two_sum2(s.hi, s.lo);
}
__device__ __forceinline__ df2 two_prod2(float2 a, float2 b) {
    const float2 p = sel_mul2(a, b);
    return {p, sel_fma2(a, b, make_float2(-p.x, -p.y))};
}

// The K boundaries of one pixel from its transmittance statistics.
__device__ __forceinline__ void boundaries(df s1, df s2, int nb, int K, float *tau) {
    if (nb >= 2) {
        const df n = df_from(float(nb));
        const df mu2 = df_div(s1, n);
        const df var = df_sub(df_div(s2, n), df_mul(mu2, mu2));
        const float mu = mu2.hi;
        const float sigma = df_sqrt(var).hi;
        const float zlo = __fdiv_rn(-mu, sigma);
        const float zhi = __fdiv_rn(__fsub_rn(1.0f, mu), sigma);
        const float ulo = normcdff(zlo), uhi = normcdff(zhi);
        const float d = __fsub_rn(uhi, ulo);
        for (int k = 1; k <= K; ++k) {
            const float c = __fdiv_rn(float(K + 1 - k), float(K + 1));
            const float z = normcdfinvf(__fmaf_rn(d, c, ulo));
            tau[(k - 1) * kSelBlock] = __fmaf_rn(sigma, z, mu);
        }
    } else {
        for (int k = 1; k <= K; ++k)
            tau[(k - 1) * kSelBlock] = __fdiv_rn(float(K + 1 - k), float(K + 1));
    }
}

// Pass 2 of one pixel: Algorithm 1's state (Walk) with its own boundaries.
// thr is the larger of the next boundary and the last one (where the walk
// stops), -1 once it has stopped.
__device__ __forceinline__ void strat_event(Walk &w, float Tt, float a, uint32_t gid, int K, float stop,
                                            const float *tau, uint32_t *key, float *wts) {
    if (w.k < K && Tt < tau[w.k * kSelBlock]) {
        key[w.m * kSelBlock] = gid;
        wts[w.m * kSelBlock] = __fmul_rn(w.TQ, a);
        ++w.m;
        w.TQ = __fmul_rn(w.TQ, __fsub_rn(1.0f, a));
        do {
            ++w.k;
        } while (w.k < K && Tt < tau[w.k * kSelBlock]);
    }
    w.thr = Tt < stop ? -1.0f : w.k < K ? fmaxf(tau[w.k * kSelBlock], stop) : stop;
}

// The first entry from u on that takes T below thr (4: none).
__device__ __forceinline__ int strat_next(int u, float t0, float t1, float t2, float t3,
                                          const float (&a)[4], float thr) {
    if (u <= 0 && a[0] > 0.0f && t0 < thr) return 0;
    if (u <= 1 && a[1] > 0.0f && t1 < thr) return 1;
    if (u <= 2 && a[2] > 0.0f && t2 < thr) return 2;
    if (u <= 3 && a[3] > 0.0f && t3 < thr) return 3;
    return 4;
}

__global__ void __launch_bounds__(32, 24)
stratified_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
                  const float *__restrict__ rec_a, const float *__restrict__ rec_h,
                  const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
                  int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
                  float T_min, int32_t *__restrict__ ids, float *__restrict__ wout,
                  uint8_t *__restrict__ cnt, float *__restrict__ tau_out, int vec) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ SelStage st;
    extern __shared__ unsigned char s_dyn[];
    const int lane = threadIdx.x & 31;
    uint32_t *s_key = reinterpret_cast<uint32_t *>(s_dyn);           // [K][64]
    float *s_w = reinterpret_cast<float *>(s_key + K * kSelBlock);   // [K][64]
    float *s_tau = s_w + K * kSelBlock;                              // [K][64]
    pdl_wait();   // the predecessor's outputs are complete and visible
    const BlockAt at = block_at(int(blockIdx.x), tile_w, tiles_x);
    const int px = at.x0 + (lane & 7), py = at.y0 + 2 * (lane >> 3);
    const bool in0 = px < W && py < H, in1 = px < W && py + 1 < H;
    const uint2 range = ranges[at.tile];
    // ---- pass 1: transmittance statistics of the dense walk
    const float2 zero = make_float2(0.f, 0.f);
    float2 T = make_float2(1.0f, 1.0f);
    df2 s1{zero, zero}, s2{zero, zero};
    int n0 = 0, n1 = 0;
    auto stats = [&](int, const float (&a0)[4], const float (&a1)[4]) -> bool {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            T = sel_mul2(T, sel_add2(make_float2(1.0f, 1.0f), make_float2(-a0[u], -a1[u])));
            // a member that would take T below T_min is not blended, nor is any
            // after it (T never rises)
            const bool b0 = a0[u] > 0.0f && !(T.x < T_min), b1 = a1[u] > 0.0f && !(T.y < T_min);
            n0 += b0;
            n1 += b1;
            const float2 x = make_float2(b0 ? T.x : 0.0f, b1 ? T.y : 0.0f);
            s1 = df2_add_f(s1, x);
            s2 = df2_add(s2, two_prod2(x, x));
        }
        return !__all_sync(FULL, (T.x < T_min || !in0) && (T.y < T_min || !in1));
    };
    walk_block<false>(rec_m, rec_w, rec_a, rec_h, isect_gid, range, W, H, at.x0, at.y0, alpha_min, alpha_max,
                      st, stats);
    boundaries(df{s1.hi.x, s1.lo.x}, df{s2.hi.x, s2.lo.x}, n0, K, s_tau + lane);
    boundaries(df{s1.hi.y, s1.lo.y}, df{s2.hi.y, s2.lo.y}, n1, K, s_tau + 32 + lane);
    __syncwarp();
    // ---- pass 2: Algorithm 1 with the boundaries tau_k
    const float *tau0 = s_tau + lane, *tau1 = s_tau + 32 + lane;
    const float stop0 = tau0[(K - 1) * kSelBlock], stop1 = tau1[(K - 1) * kSelBlock];
    Walk w0{1.0f, 1.0f, in0 ? fmaxf(tau0[0], stop0) : -1.0f, 0, 0};
    Walk w1{1.0f, 1.0f, in1 ? fmaxf(tau1[0], stop1) : -1.0f, 0, 0};
    auto visit = [&](int j, const float (&a0)[4], const float (&a1)[4]) -> bool {
        float2 t[4];
        float2 T2 = make_float2(w0.T, w1.T);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            T2 = sel_mul2(T2, sel_add2(make_float2(1.0f, 1.0f), make_float2(-a0[u], -a1[u])));
            t[u] = T2;
        }
        w0.T = T2.x;
        w1.T = T2.y;
        int u0 = 0, u1 = 0;   // entries already settled
        while (__any_sync(FULL, (u0 < 4 && T2.x < w0.thr) || (u1 < 4 && T2.y < w1.thr))) {
            if (u0 < 4 && T2.x < w0.thr) {
                u0 = strat_next(u0, t[0].x, t[1].x, t[2].x, t[3].x, a0, w0.thr);
                if (u0 < 4) {
                    const float a = u0 == 0 ? a0[0] : u0 == 1 ? a0[1] : u0 == 2 ? a0[2] : a0[3];
                    const float Tt = u0 == 0 ? t[0].x : u0 == 1 ? t[1].x : u0 == 2 ? t[2].x : t[3].x;
                    strat_event(w0, Tt, a, st.g[j + u0], K, stop0, tau0, s_key + lane, s_w + lane);
                    ++u0;
                }
            }
            if (u1 < 4 && T2.y < w1.thr) {
                u1 = strat_next(u1, t[0].y, t[1].y, t[2].y, t[3].y, a1, w1.thr);
                if (u1 < 4) {
                    const float a = u1 == 0 ? a1[0] : u1 == 1 ? a1[1] : u1 == 2 ? a1[2] : a1[3];
                    const float Tt = u1 == 0 ? t[0].y : u1 == 1 ? t[1].y : u1 == 2 ? t[2].y : t[3].y;
                    strat_event(w1, Tt, a, st.g[j + u1], K, stop1, tau1, s_key + 32 + lane, s_w + 32 + lane);
                    ++u1;
                }
            }
        }
        return !__all_sync(FULL, w0.thr == -1.0f && w1.thr == -1.0f);
    };
    walk_block<false>(rec_m, rec_w, rec_a, rec_h, isect_gid, range, W, H, at.x0, at.y0, alpha_min, alpha_max,
                      st, visit);
    auto finish = [&](const Walk &w, uint32_t *key, float *wts) {
        const float D = __fsub_rn(1.0f, w.TQ);
        for (int j = 0; j < K; ++j) {
            if (j >= w.m) key[j * kSelBlock] = 0xFFFFFFFFu;
            wts[j * kSelBlock] = j < w.m ? __fdiv_rn(wts[j * kSelBlock], D) : 0.0f;
        }
    };
    finish(w0, s_key + lane, s_w + lane);
    finish(w1, s_key + 32 + lane, s_w + 32 + lane);
    __syncwarp();
    store_slots(W, H, at.x0, at.y0, K, vec != 0, reinterpret_cast<const int32_t *>(s_key), ids);
    store_slots(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_w, wout);
    if (tau_out) store_slots(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_tau, tau_out);
    if (in0) cnt[int64_t(py) * W + px] = uint8_t(w0.m);
    if (in1) cnt[int64_t(py + 1) * W + px] = uint8_t(w1.m);
}

}  // namespace

cudaError_t launch_select_rule(const qr_frame &f, int rule, int32_t *ids, float *w, uint8_t *cnt,
                               float *tau, cudaStream_t s) {
    const int tiles = num_tiles(f);
    if (tiles == 0) return cudaSuccess;
    const int K = f.params.K, G = (K + 3) / 4;
    // at most 24 KB of slots per warp
    const size_t dyn = size_t(kSelBlock) * 4 * (rule == kStratified ? 3 * K : 2 * K + 2 * G);
    const uintptr_t outs = reinterpret_cast<uintptr_t>(ids) | reinterpret_cast<uintptr_t>(w) |
                           reinterpret_cast<uintptr_t>(tau);
    const int vec = K % 4 == 0 && (outs & 15) == 0;
    auto go = [&](auto kern, auto... last) -> cudaError_t {
        return pdl_launch(kern, dim3(unsigned(tiles) * 4), dim3(32), dyn, s,
                          (const float4 *)slot<float4>(f, S_REC_M),
                          (const float4 *)slot<float4>(f, S_REC_C),
                          (const float *)slot<float>(f, S_REC_A),
                          (const float *)slot<float>(f, S_REC_H),
                          (const uint32_t *)slot<uint32_t>(f, S_IGID),
                          (const uint2 *)slot<uint2>(f, S_RANGES), f.camera.width,
                          f.camera.height, f.params.tile_w, f.tiles_x, K, f.params.alpha_min,
                          f.params.alpha_max, f.params.T_min, ids, w, cnt, last...);
    };
    const cudaError_t e = rule == kTopK ? go(topk_kernel, vec) : go(stratified_kernel, tau, vec);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace qr
