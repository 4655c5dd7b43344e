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
// GB300 design: one warp per 8 x 8 pixel block (or 8 x 4), on the
// selection's walk (walk_block in select_tile.cuh: the warp culls the list
// for its own block and takes the survivors four at a time), so a warp stops
// when its own 64 pixels have and no CTA barrier ties it to others.  alpha'
// and the transmittance are evaluated as the dense blend does, so the walks
// agree with it bit for bit.
//   * top-K (8 x 4 pixels, one per lane) keeps its candidates sorted in
//     registers: a strictly larger weight moves the smaller ones down and the
//     smallest (latest among equal) out.  Once fl(T alpha_max) is no larger
//     than the smallest kept weight, no later entry can enter (T only falls
//     and alpha' <= alpha_max), so the pixel stops early without changing the
//     result.  With more than 8 entries the insertions cost more than
//     replacing the smallest of K slots in shared memory (topk_slots_kernel),
//     unless the latency of a walk bounds the frame.
//   * Stratified-K sums T and T^2 in compensated double-FP32 arithmetic, both
//     pixels of a lane in one packed FP32x2 instruction stream (adding an
//     exact 0 where an entry is no member) and four entries at a time, forms
//     mu and sigma from them, and the boundaries with the FP32 normal CDF and
//     its inverse (normcdff, normcdfinvf); the boundaries sit in shared memory
//     for pass 2, which re-walks the list as the selection does.
// Bound by instruction issue (room) and by the longest lists' chains (object).
// Measured (CTAs of eight warps walking a tile in step, one pixel per lane ->
// now): Stratified-K, room VGA, K = 8: 183 -> 109 us; top-K, K = 8, room VGA
// 90 -> 73 us; top-K in slots: with its kernel.
#include "select_tile.cuh"

namespace qr {
namespace {

enum { kTopK = 1, kStratified = 2 };

// 8 x 8 blocks up to which, and capacity per tile from which, the chain of a
// walk rather than issue bounds top-K (launch_select_rule)
constexpr int kFewBlocks = 152 * 8;
constexpr int64_t kLongTopLists = 320;

// ------------------------------------------------------------------ top-K
constexpr int kTopPix = 32;        // pixels per warp: 8 x 4, one per lane
// The K largest weights of one pixel, kept sorted in registers: v descending,
// -0.5 in a free slot (every member enters), equal weights in list order, pos
// the list positions.  KT >= K slots are held; the first K are the rule's.
template <int KT>
struct Top {
    float v[KT];
    uint32_t pos[KT];
};

// Enters (x, at) where x > v[KT - 1]: slots below its place move down by one,
// the last one falls out (the smallest weight, the latest of equal ones).  All
// slots are written from the old values, so the 5 KT instructions are free of
// chains and of branches.
template <int KT>
__device__ __forceinline__ void top_insert(Top<KT> &t, float x, uint32_t at) {
#pragma unroll
    for (int j = KT - 1; j > 0; --j) {
        t.pos[j] = x > t.v[j - 1] ? t.pos[j - 1] : x > t.v[j] ? at : t.pos[j];
        t.v[j] = fmaxf(fminf(t.v[j - 1], x), t.v[j]);
    }
    t.pos[0] = x > t.v[0] ? at : t.pos[0];
    t.v[0] = fmaxf(t.v[0], x);
}

// Depth order (list position), the kept sum in that order, weights divided by
// it, Gaussian ids in place of positions, the rest padded.
__device__ __forceinline__ void top_finish(int m, int K, const uint32_t *__restrict__ isect_gid,
                                           uint32_t *key, float *w) {
    for (int i = 1; i < m; ++i) {
        const uint32_t kk = key[i * kTopPix];
        const float ww = w[i * kTopPix];
        int j = i;
        while (j > 0 && key[(j - 1) * kTopPix] > kk) {
            key[j * kTopPix] = key[(j - 1) * kTopPix];
            w[j * kTopPix] = w[(j - 1) * kTopPix];
            --j;
        }
        key[j * kTopPix] = kk;
        w[j * kTopPix] = ww;
    }
    float D = 0.0f;
    for (int j = 0; j < m; ++j) D = __fadd_rn(D, w[j * kTopPix]);
    for (int j = 0; j < K; ++j) {
        key[j * kTopPix] = j < m ? isect_gid[key[j * kTopPix]] : 0xFFFFFFFFu;
        w[j * kTopPix] = j < m ? __fdiv_rn(w[j * kTopPix], D) : 0.0f;
    }
}

// The K entries of a block's PX 32 pixels (entry-major, pixel (x, y) at
// (y % PX) 32 + (y / PX) 8 + x) written to the image.
template <int PX, typename T>
__device__ __forceinline__ void store_slots(int W, int H, int x0, int y0, int K, bool vec, const T *s,
                                            T *__restrict__ out) {
    constexpr int N = 32 * PX;
    const int lane = threadIdx.x & 31;
    const int per = vec ? 4 : 1;
    const int KP = K / per;
    const uint32_t inv = (65536u + uint32_t(KP) - 1u) / uint32_t(KP);   // e / KP, e < 64 KP <= 2048
    for (int e = lane; e < N * KP; e += 32) {
        const int pix = int((uint32_t(e) * inv) >> 16), j = (e - pix * KP) * per;
        const int x = pix & 7, y = pix >> 3;
        if (x0 + x >= W || y0 + y >= H) continue;
        const T *v = s + j * N + (y % PX) * 32 + (y / PX) * 8 + x;
        T *o = out + (int64_t(y0 + y) * W + x0 + x) * K + j;
        if (vec) {
            struct alignas(16) V4 { T a, b, c, d; };
            *reinterpret_cast<V4 *>(o) = V4{v[0], v[N], v[2 * N], v[3 * N]};
        } else {
            *o = *v;
        }
    }
}

struct BlockAt {
    int tile, x0, y0;
};
// Block of 8 x (4 PX) pixels, 8 / PX of them to a tile.
template <int PX>
__device__ __forceinline__ BlockAt block_at(int block, int tile_w, int tiles_x) {
    constexpr int N = 8 / PX;
    const int tile = block / N, part = block % N, across = tile_w >> 3;
    return {tile, (tile % tiles_x) * tile_w + (part % across) * 8,
            (tile / tiles_x) * (kSelPix / tile_w) + (part / across) * 4 * PX};
}

// One pixel per lane (8 x 4 pixels per warp): the kept entries stay in
// registers, and the chain of a long list is half as long as with two.  An
// entry that some pixel of the warp may keep costs the warp one top_insert,
// the others a vote.
template <int KT>
__global__ void __launch_bounds__(32, 24)
topk_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
            const float *__restrict__ rec_a, const float *__restrict__ rec_h,
            const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
            int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
            float T_min, int32_t *__restrict__ ids, float *__restrict__ wout,
            uint8_t *__restrict__ cnt, int vec) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ SelStage st;
    __shared__ uint32_t s_key[KT * kTopPix];   // entry-major
    __shared__ float s_w[KT * kTopPix];
    const int lane = threadIdx.x & 31;
    pdl_wait();   // the predecessor's outputs are complete and visible
    const BlockAt at = block_at<1>(int(blockIdx.x), tile_w, tiles_x);
    const int px = at.x0 + (lane & 7), py = at.y0 + (lane >> 3);
    const bool inside = px < W && py < H;
    Top<KT> top;
#pragma unroll
    for (int j = 0; j < KT; ++j) {
        top.v[j] = -0.5f;
        top.pos[j] = 0u;
    }
    float T = 1.0f;
    float wmin = inside ? -0.5f : INFINITY;   // the K-th largest; +inf once the pixel has stopped
    auto visit = [&](int j, const float (&a)[4][1]) -> bool {
        float w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            // weight T alpha' of a member, -1 of any other entry; a member that
            // would take T below T_min is not blended, nor is any after it (T
            // never rises)
            const float n = __fmul_rn(T, __fsub_rn(1.0f, a[u][0]));
            w[u] = a[u][0] > 0.0f && !(n < T_min) ? __fmul_rn(T, a[u][0]) : -1.0f;
            T = n;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = w[u] > wmin;
            if (!__any_sync(FULL, in)) continue;
            if (in) {
                top_insert(top, w[u], st.g[j + u]);
                if (KT > 4) {
#pragma unroll
                    for (int i = KT / 2; i < KT; ++i) wmin = i == K - 1 ? top.v[i] : wmin;
                } else {
#pragma unroll
                    for (int i = 0; i < KT; ++i) wmin = i == K - 1 ? top.v[i] : wmin;
                }
            }
        }
        // no later entry can enter once fl(T alpha_max) is no larger than wmin
        if (T < T_min || __fmul_rn(T, alpha_max) <= wmin) wmin = INFINITY;
        return !__all_sync(FULL, wmin == INFINITY);
    };
    walk_block<true, 1>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[at.tile], W, H, at.x0, at.y0,
                        alpha_min, alpha_max, st, visit);
    int m = 0;
#pragma unroll
    for (int j = 0; j < KT; ++j) {
        m += j < K && top.v[j] >= 0.0f;
        s_key[j * kTopPix + lane] = top.pos[j];
        s_w[j * kTopPix + lane] = top.v[j];
    }
    top_finish(m, K, isect_gid, s_key + lane, s_w + lane);
    __syncwarp();
    store_slots<1>(W, H, at.x0, at.y0, K, vec != 0, reinterpret_cast<const int32_t *>(s_key), ids);
    store_slots<1>(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_w, wout);
    if (inside) cnt[int64_t(py) * W + px] = uint8_t(m);
}

// ------------------------------------------------------------------ top-K, many entries
// A pixel's K slots (shared memory, entry-major: a lane's accesses fall in its
// own bank) stand in groups of four with the smallest of each group kept
// beside them, so replacing the smallest searches four slots and the groups,
// and only lanes whose entry enters take part.
// Bound by instruction issue (room) and by the longest lists' chains (object).
// K = 9 / 16 / 32, us (one CTA of eight warps per tile, the list staged for all
// of them and K slots searched on each replacement -> sorted registers, K <= 16
// -> this): room VGA 300k Gaussians 102 / 155 / 366 -> 135 / 181 -> 87 / 111 /
// 210; room VGA 1M 100 / 149 / 316 -> 142 / 188 -> 92 / 112 / 187; room 1M at 1296
// x 968 278 / 445 / 1037 -> 461 / 618 -> 275 / 339 / 584; object VGA 500k 358 / 474 /
// 1141 -> 250 / 303 -> 220 / 269 / 430; object 517 x 389 200k 235 / 332 / 717 -> 158 /
// 200 -> 143 / 178 / 274.  Two pixels per lane instead: that last K = 16 238.
struct Slots {
    uint32_t *key;   // [K][32]: list position
    float *w;        // [K][32]: weight
    float *gw;       // [G][32]: smallest weight of a group ...
    uint32_t *gk;    // [G][32]: ... and its slot
};
// Slot a goes before slot b: the smaller weight, the later entry of equal ones.
__device__ __forceinline__ bool slot_less(float wa, uint32_t a, float wb, uint32_t b, const uint32_t *key) {
    return wa < wb || (wa == wb && key[a * kTopPix] > key[b * kTopPix]);
}
__device__ __forceinline__ void rescan_group(const Slots &s, int g, int K) {
    const int j0 = 4 * g;
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = j0 + i < K ? s.w[(j0 + i) * kTopPix] : INFINITY;
    uint32_t at = uint32_t(j0);
    float b = v[0];
#pragma unroll
    for (int i = 1; i < 4; ++i)
        if (v[i] <= b && j0 + i < K && slot_less(v[i], uint32_t(j0 + i), b, at, s.key)) {
            at = uint32_t(j0 + i);
            b = v[i];
        }
    s.gw[g * kTopPix] = b;
    s.gk[g * kTopPix] = at;
}
// Keeps the member at list position pos with weight x > wmin: a free slot
// while there is one (wmin < 0), else the smallest's.
__device__ __forceinline__ void slot_insert(const Slots &s, int K, uint32_t pos, float x, int &m,
                                            uint32_t &smin, float &wmin) {
    const int G = (K + 3) >> 2;
    const uint32_t at = m < K ? uint32_t(m) : smin;
    s.key[at * kTopPix] = pos;
    s.w[at * kTopPix] = x;
    if (m < K) {
        if (++m < K) return;
        for (int g = 0; g < G; ++g) rescan_group(s, g, K);
    } else {
        rescan_group(s, int(at >> 2), K);
    }
    float b = s.gw[0];
    uint32_t bs = s.gk[0];
    for (int g = 1; g < G; ++g) {
        const float v = s.gw[g * kTopPix];
        const uint32_t vs = s.gk[g * kTopPix];
        if (v <= b && slot_less(v, vs, b, bs, s.key)) {
            b = v;
            bs = vs;
        }
    }
    wmin = b;
    smin = bs;
}

__global__ void __launch_bounds__(32, 24)
topk_slots_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
                  const float *__restrict__ rec_a, const float *__restrict__ rec_h,
                  const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
                  int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
                  float T_min, int32_t *__restrict__ ids, float *__restrict__ wout,
                  uint8_t *__restrict__ cnt, int vec) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ SelStage st;
    extern __shared__ unsigned char s_dyn[];
    const int lane = threadIdx.x & 31, G = (K + 3) >> 2;
    uint32_t *s_key = reinterpret_cast<uint32_t *>(s_dyn);
    float *s_w = reinterpret_cast<float *>(s_key + K * kTopPix);
    float *s_gw = s_w + K * kTopPix;
    const Slots s{s_key + lane, s_w + lane, s_gw + lane, reinterpret_cast<uint32_t *>(s_gw + G * kTopPix) + lane};
    pdl_wait();   // the predecessor's outputs are complete and visible
    const BlockAt at = block_at<1>(int(blockIdx.x), tile_w, tiles_x);
    const int px = at.x0 + (lane & 7), py = at.y0 + (lane >> 3);
    const bool inside = px < W && py < H;
    int m = 0;
    uint32_t smin = 0u;
    float T = 1.0f;
    float wmin = inside ? -0.5f : INFINITY;   // the smallest kept weight; +inf once the pixel has stopped
    auto visit = [&](int j, const float (&a)[4][1]) -> bool {
        float w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {   // as in topk_kernel
            const float n = __fmul_rn(T, __fsub_rn(1.0f, a[u][0]));
            w[u] = a[u][0] > 0.0f && !(n < T_min) ? __fmul_rn(T, a[u][0]) : -1.0f;
            T = n;
        }
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {   // the insertion's code once
            const float x = u == 0 ? w[0] : u == 1 ? w[1] : u == 2 ? w[2] : w[3];
            if (x > wmin) slot_insert(s, K, st.g[j + u], x, m, smin, wmin);
        }
        // no later entry can enter once fl(T alpha_max) is no larger than wmin
        if (T < T_min || __fmul_rn(T, alpha_max) <= wmin) wmin = INFINITY;
        return !__all_sync(FULL, wmin == INFINITY);
    };
    walk_block<true, 1>(rec_m, rec_w, rec_a, rec_h, isect_gid, ranges[at.tile], W, H, at.x0, at.y0,
                        alpha_min, alpha_max, st, visit);
    top_finish(m, K, isect_gid, s_key + lane, s_w + lane);
    __syncwarp();
    store_slots<1>(W, H, at.x0, at.y0, K, vec != 0, reinterpret_cast<const int32_t *>(s_key), ids);
    store_slots<1>(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_w, wout);
    if (inside) cnt[int64_t(py) * W + px] = uint8_t(m);
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
// s + (x[0] + .. + x[3]) + lo, the nonzero x not increasing: their sum runs in
// error-free steps (a running sum is 0 or no smaller than the next term, as
// the three-operation form wants), the errors, of 2^-24 of the terms, in plain
// ones: 22 operations a step where four compensated additions took 40.
__device__ __forceinline__ df2 df2_add4(df2 s, const float2 (&x)[4], float2 lo) {
    df2 r = fast_two_sum2(x[0], x[1]);
    float2 e = r.lo;
    r = fast_two_sum2(r.hi, x[2]);
    e = sel_add2(e, r.lo);
    r = fast_two_sum2(r.hi, x[3]);
    e = sel_add2(sel_add2(e, r.lo), lo);
    const df2 t = two_sum2(s.hi, r.hi);
    return fast_two_sum2(t.hi, sel_add2(t.lo, sel_add2(s.lo, e)));
}
__device__ __forceinline__ df2 two_prod2(float2 a, float2 b) {
    const float2 p = sel_mul2(a, b);
    return {p, sel_fma2(a, b, make_float2(-p.x, -p.y))};
}

// What the boundaries of a pixel are formed from (nb >= 2 blended entries).
struct Spread {
    float mu, sigma, ulo, d;
};
__device__ __forceinline__ Spread spread_of(df s1, df s2, int nb) {
    const df n = df_from(float(nb));
    const df mu2 = df_div(s1, n);
    const df var = df_sub(df_div(s2, n), df_mul(mu2, mu2));
    const float mu = mu2.hi;
    const float sigma = df_sqrt(var).hi;
    const float zlo = __fdiv_rn(-mu, sigma);
    const float zhi = __fdiv_rn(__fsub_rn(1.0f, mu), sigma);
    const float ulo = normcdff(zlo), uhi = normcdff(zhi);
    return {mu, sigma, ulo, __fsub_rn(uhi, ulo)};
}
__device__ __forceinline__ float boundary_of(const Spread &p, float c, int nb) {
    return nb >= 2 ? __fmaf_rn(p.sigma, normcdfinvf(__fmaf_rn(p.d, c, p.ulo)), p.mu) : c;
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
                                          const float (&a)[4][2], int i, float thr) {
    if (u <= 0 && a[0][i] > 0.0f && t0 < thr) return 0;
    if (u <= 1 && a[1][i] > 0.0f && t1 < thr) return 1;
    if (u <= 2 && a[2][i] > 0.0f && t2 < thr) return 2;
    if (u <= 3 && a[3][i] > 0.0f && t3 < thr) return 3;
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
    const BlockAt at = block_at<2>(int(blockIdx.x), tile_w, tiles_x);
    const int px = at.x0 + (lane & 7), py = at.y0 + 2 * (lane >> 3);
    const bool in0 = px < W && py < H, in1 = px < W && py + 1 < H;
    const uint2 range = ranges[at.tile];
    // ---- pass 1: transmittance statistics of the dense walk
    const float2 zero = make_float2(0.f, 0.f);
    float2 T = make_float2(1.0f, 1.0f);
    df2 s1{zero, zero}, s2{zero, zero};
    int n0 = 0, n1 = 0;
    auto stats = [&](int, const float (&a)[4][2]) -> bool {
        float2 x[4], y[4], lo = zero;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            T = sel_mul2(T, sel_add2(make_float2(1.0f, 1.0f), make_float2(-a[u][0], -a[u][1])));
            // a member that would take T below T_min is not blended, nor is any
            // after it (T never rises)
            const bool b0 = a[u][0] > 0.0f && !(T.x < T_min), b1 = a[u][1] > 0.0f && !(T.y < T_min);
            n0 += b0;
            n1 += b1;
            x[u] = make_float2(b0 ? T.x : 0.0f, b1 ? T.y : 0.0f);
            const df2 p = two_prod2(x[u], x[u]);
            y[u] = p.hi;
            lo = sel_add2(lo, p.lo);
        }
        s1 = df2_add4(s1, x, zero);
        s2 = df2_add4(s2, y, lo);
        return !__all_sync(FULL, (T.x < T_min || !in0) && (T.y < T_min || !in1));
    };
    walk_block<false, 2>(rec_m, rec_w, rec_a, rec_h, isect_gid, range, W, H, at.x0, at.y0, alpha_min, alpha_max,
                      st, stats);
    {
        Spread p[2];
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {   // the code once: it is long
            const Spread q = spread_of(i ? df{s1.hi.y, s1.lo.y} : df{s1.hi.x, s1.lo.x},
                                       i ? df{s2.hi.y, s2.lo.y} : df{s2.hi.x, s2.lo.x}, max(i ? n1 : n0, 1));
            if (i) p[1] = q; else p[0] = q;
        }
#pragma unroll 1
        for (int k = 1; k <= K; ++k) {   // both pixels' chains side by side
            const float c = __fdiv_rn(float(K + 1 - k), float(K + 1));
            s_tau[(k - 1) * kSelBlock + lane] = boundary_of(p[0], c, n0);
            s_tau[(k - 1) * kSelBlock + 32 + lane] = boundary_of(p[1], c, n1);
        }
    }
    __syncwarp();
    // ---- pass 2: Algorithm 1 with the boundaries tau_k
    const float *tau0 = s_tau + lane, *tau1 = s_tau + 32 + lane;
    const float stop0 = tau0[(K - 1) * kSelBlock], stop1 = tau1[(K - 1) * kSelBlock];
    Walk w0{1.0f, 1.0f, in0 ? fmaxf(tau0[0], stop0) : -1.0f, 0, 0};
    Walk w1{1.0f, 1.0f, in1 ? fmaxf(tau1[0], stop1) : -1.0f, 0, 0};
    auto visit = [&](int j, const float (&a)[4][2]) -> bool {
        float2 t[4];
        float2 T2 = make_float2(w0.T, w1.T);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            T2 = sel_mul2(T2, sel_add2(make_float2(1.0f, 1.0f), make_float2(-a[u][0], -a[u][1])));
            t[u] = T2;
        }
        w0.T = T2.x;
        w1.T = T2.y;
        int u0 = 0, u1 = 0;   // entries already settled
        while (__any_sync(FULL, (u0 < 4 && T2.x < w0.thr) || (u1 < 4 && T2.y < w1.thr))) {
            if (u0 < 4 && T2.x < w0.thr) {
                u0 = strat_next(u0, t[0].x, t[1].x, t[2].x, t[3].x, a, 0, w0.thr);
                if (u0 < 4) {
                    const float e = u0 == 0 ? a[0][0] : u0 == 1 ? a[1][0] : u0 == 2 ? a[2][0] : a[3][0];
                    const float Tt = u0 == 0 ? t[0].x : u0 == 1 ? t[1].x : u0 == 2 ? t[2].x : t[3].x;
                    strat_event(w0, Tt, e, st.g[j + u0], K, stop0, tau0, s_key + lane, s_w + lane);
                    ++u0;
                }
            }
            if (u1 < 4 && T2.y < w1.thr) {
                u1 = strat_next(u1, t[0].y, t[1].y, t[2].y, t[3].y, a, 1, w1.thr);
                if (u1 < 4) {
                    const float e = u1 == 0 ? a[0][1] : u1 == 1 ? a[1][1] : u1 == 2 ? a[2][1] : a[3][1];
                    const float Tt = u1 == 0 ? t[0].y : u1 == 1 ? t[1].y : u1 == 2 ? t[2].y : t[3].y;
                    strat_event(w1, Tt, e, st.g[j + u1], K, stop1, tau1, s_key + 32 + lane, s_w + 32 + lane);
                    ++u1;
                }
            }
        }
        return !__all_sync(FULL, w0.thr == -1.0f && w1.thr == -1.0f);
    };
    walk_block<false, 2>(rec_m, rec_w, rec_a, rec_h, isect_gid, range, W, H, at.x0, at.y0, alpha_min, alpha_max,
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
    store_slots<2>(W, H, at.x0, at.y0, K, vec != 0, reinterpret_cast<const int32_t *>(s_key), ids);
    store_slots<2>(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_w, wout);
    if (tau_out) store_slots<2>(W, H, at.x0, at.y0, K, vec != 0, (const float *)s_tau, tau_out);
    if (in0) cnt[int64_t(py) * W + px] = uint8_t(w0.m);
    if (in1) cnt[int64_t(py + 1) * W + px] = uint8_t(w1.m);
}

}  // namespace

cudaError_t launch_select_rule(const qr_frame &f, int rule, int32_t *ids, float *w, uint8_t *cnt,
                               float *tau, cudaStream_t s) {
    const int tiles = num_tiles(f);
    if (tiles == 0) return cudaSuccess;
    const int K = f.params.K;
    const uintptr_t outs = reinterpret_cast<uintptr_t>(ids) | reinterpret_cast<uintptr_t>(w) |
                           reinterpret_cast<uintptr_t>(tau);
    const int vec = K % 4 == 0 && (outs & 15) == 0;
    auto go = [&](auto kern, int blocks, size_t dyn, auto... last) -> cudaError_t {
        return pdl_launch(kern, dim3(unsigned(tiles) * blocks), dim3(32), dyn, s,
                          (const float4 *)slot<float4>(f, S_REC_M),
                          (const float4 *)slot<float4>(f, S_REC_C),
                          (const float *)slot<float>(f, S_REC_A),
                          (const float *)slot<float>(f, S_REC_H),
                          (const uint32_t *)slot<uint32_t>(f, S_IGID),
                          (const uint2 *)slot<uint2>(f, S_RANGES), f.camera.width,
                          f.camera.height, f.params.tile_w, f.tiles_x, K, f.params.alpha_min,
                          f.params.alpha_max, f.params.T_min, ids, w, cnt, last...);
    };
    // Top-K of 9 .. 16 entries in registers / in slots (us, K = 9, 16) where a
    // frame has few blocks: long lists, object 30k at 100 x 70 124, 131 / 157, 169,
    // object 200k at 320 x 240 149, 178 / 170, 206, room 100k at 160 x 120 (326
    // entries per tile) 46, 56 / 54, 66; short ones, room 100k at 320 x 240 (151) 60,
    // 78 / 48, 58, room 20k at 160 x 120 (65) 30, 34 / 33, 25.  With more blocks slots
    // are the faster ones throughout (topk_slots_kernel).
    const bool latency = tiles * 4 <= kFewBlocks && f.max_isect >= kLongTopLists * tiles;
    cudaError_t e;
    if (rule == kStratified) {
        e = go(stratified_kernel, 4, size_t(kSelBlock) * 4 * 3 * K, tau, vec);
    } else if (K <= 4) {
        e = go(topk_kernel<4>, 8, 0, vec);
    } else if (K <= 8) {
        e = go(topk_kernel<8>, 8, 0, vec);
    } else if (K <= 16 && latency) {
        e = go(topk_kernel<16>, 8, 0, vec);
    } else {
        e = go(topk_slots_kernel, 8, size_t(kTopPix) * 8 * (K + (K + 3) / 4), vec);
    }
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace qr
