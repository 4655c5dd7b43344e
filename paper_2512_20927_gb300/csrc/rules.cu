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
//     result.  Shared-memory slots with a replaced minimum, two pixels per
//     lane, took 238 us where this takes 187 (below).  With many entries the
//     insertions cost more than a search of slots: topk_tile_kernel.
//   * Stratified-K sums T and T^2 in compensated double-FP32 arithmetic, both
//     pixels of a lane in one packed FP32x2 instruction stream (adding an
//     exact 0 where an entry is no member) and four entries at a time, forms
//     mu and sigma from them, and the boundaries with the FP32 normal CDF and
//     its inverse (normcdff, normcdfinvf); the boundaries sit in shared memory
//     for pass 2, which re-walks the list as the selection does.
// Bound by instruction issue (room) and by the longest lists' chains (object).
// Measured (CTAs of eight warps walking a tile in step, one pixel per lane ->
// now): Stratified-K, room VGA, K = 8: 183 -> 109 us; top-K, object 517 x 389,
// 200k Gaussians, K = 16: 315 -> 187 us.
#include "select_tile.cuh"

namespace qr {
namespace {

enum { kTopK = 1, kStratified = 2 };

// 8 x 8 blocks up to which, and list capacity per tile from which, latency
// rather than issue bounds top-K's walk
constexpr int kFewBlocks = 152 * 8;
constexpr int64_t kLongTopLists = 768;

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
// One CTA per screen tile, one pixel per thread: the list is staged 256 records
// at a time and culled per warp, and a pixel's candidates sit in shared-memory
// slots whose smallest a replacement searches again.  With more entries an
// insertion into sorted registers costs more than that search, unless latency
// bounds the walk.
constexpr int kPix = 256;
constexpr int kThreads = 256;
constexpr int kTileBatch = 256;

struct Stage {
    float4 *m, *c;
    float *a, *h;
};

// Walks the tile's list for this thread's pixel: stages records, culls them
// per warp against the warp's pixel box and calls visit(pos, alpha') for
// every member entry (alpha' >= alpha_min) in list order until the pixel is
// done.  visit returns true when the pixel has finished its walk.  All
// threads of the CTA must call it.
template <typename Visit>
__device__ __forceinline__ void walk_list(const float4 *__restrict__ rec_m,
                                          const float4 *__restrict__ rec_w,
                                          const float *__restrict__ rec_a,
                                          const float *__restrict__ rec_h,
                                          const uint32_t *__restrict__ isect_gid, uint2 range,
                                          const Stage &st, float ux, float uy, float bx0,
                                          float bx1, float by0, float by1, float alpha_min,
                                          float alpha_max, bool &done, Visit visit) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (uint32_t b = range.x; b < range.y; b += kTileBatch) {
        if (__syncthreads_count(done) == kThreads) break;
        if (b + threadIdx.x < range.y) {
            const uint32_t g = isect_gid[b + threadIdx.x];
            st.m[threadIdx.x] = rec_m[g];
            st.c[threadIdx.x] = rec_w[g];
            st.a[threadIdx.x] = rec_a[g];
            st.h[threadIdx.x] = rec_h[g];
        }
        __syncthreads();
        const int nb = int(min(uint32_t(kTileBatch), range.y - b));
        for (int c0 = 0; c0 < nb; c0 += 32) {
            if (__all_sync(FULL, done)) break;
            const int jl = c0 + lane;
            bool pass = false;
            if (jl < nb)
                pass = !(box_min_half_q(st.m[jl], st.c[jl], bx0, bx1, by0, by1) * 0.999f >
                         st.h[jl] + 1e-3f);
            unsigned todo = __ballot_sync(FULL, pass);
            while (todo && !done) {
                const int j = c0 + __ffs(todo) - 1;
                todo &= todo - 1u;
                const PixelTerm pt = eval_half_q(ux, uy, st.m[j], st.c[j]);
                if (pt.half_q > st.h[j]) continue;
                const float a = eval_alpha(st.a[j], pt.half_q, alpha_max);
                if (a < alpha_min) continue;
                done = visit(b + uint32_t(j), a);
            }
        }
        __syncthreads();   // the stage is rewritten by the next batch
    }
}

__global__ void __launch_bounds__(kThreads)
topk_tile_kernel(const float4 *__restrict__ rec_m, const float4 *__restrict__ rec_w,
            const float *__restrict__ rec_a, const float *__restrict__ rec_h,
            const uint32_t *__restrict__ isect_gid, const uint2 *__restrict__ ranges, int W,
            int H, int tile_w, int tiles_x, int K, float alpha_min, float alpha_max,
            float T_min, int32_t *__restrict__ ids, float *__restrict__ wout,
            uint8_t *__restrict__ cnt) {
    pdl_wait();
    __shared__ float4 s_m[kTileBatch];
    __shared__ float4 s_c[kTileBatch];
    __shared__ float s_a[kTileBatch];
    __shared__ float s_h[kTileBatch];
    extern __shared__ unsigned char s_dyn[];
    const int KS = K | 1;   // odd stride: a thread's slots fall in their own banks
    uint32_t *s_key = reinterpret_cast<uint32_t *>(s_dyn);                 // [256][KS]
    float *s_w = reinterpret_cast<float *>(s_dyn) + KS * kPix;             // [256][KS]
    const Stage st{s_m, s_c, s_a, s_h};

    const int tile = blockIdx.x;
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    const int tile_h = kPix / tile_w;
    const int lx = threadIdx.x % tile_w, ly = threadIdx.x / tile_w;
    const int px = tx * tile_w + lx, py = ty * tile_h + ly;
    const bool inside = px < W && py < H;
    const float ux = float(px) + 0.5f, uy = float(py) + 0.5f;
    const uint2 range = ranges[tile];
    uint32_t *my_key = s_key + threadIdx.x * KS;
    float *my_w = s_w + threadIdx.x * KS;

    constexpr unsigned FULL = 0xffffffffu;
    float bx0 = ux, bx1 = ux, by0 = uy, by1 = uy;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        bx0 = fminf(bx0, __shfl_xor_sync(FULL, bx0, o));
        bx1 = fmaxf(bx1, __shfl_xor_sync(FULL, bx1, o));
        by0 = fminf(by0, __shfl_xor_sync(FULL, by0, o));
        by1 = fmaxf(by1, __shfl_xor_sync(FULL, by1, o));
    }

    int m = 0;          // kept entries
    float D = 0.0f;     // normaliser
    {
        // ---- one dense walk keeping the K largest weights
        float T = 1.0f, wmin = 0.0f;
        int smin = 0;
        bool done = !inside;
        walk_list(rec_m, rec_w, rec_a, rec_h, isect_gid, range, st, ux, uy, bx0, bx1, by0, by1,
                  alpha_min, alpha_max, done, [&](uint32_t pos, float a) -> bool {
                      const float Tt = __fmul_rn(T, __fsub_rn(1.0f, a));
                      if (T_min > 0.0f && Tt < T_min) return true;
                      const float w = __fmul_rn(T, a);
                      T = Tt;
                      if (m < K) {
                          my_key[m] = pos;
                          my_w[m] = w;
                          ++m;
                          if (m < K) return false;
                      } else if (w > wmin) {
                          my_key[smin] = pos;
                          my_w[smin] = w;
                      } else {
                          return __fmul_rn(T, alpha_max) <= wmin;
                      }
                      // the smallest kept weight, the latest entry among equal ones
                      smin = 0;
                      for (int j = 1; j < K; ++j)
                          if (my_w[j] < my_w[smin] ||
                              (my_w[j] == my_w[smin] && my_key[j] > my_key[smin]))
                              smin = j;
                      wmin = my_w[smin];
                      return __fmul_rn(T, alpha_max) <= wmin;
                  });
        // depth order (list position), then the kept sum in that order
        for (int i = 1; i < m; ++i) {
            const uint32_t kk = my_key[i];
            const float ww = my_w[i];
            int j = i;
            while (j > 0 && my_key[j - 1] > kk) {
                my_key[j] = my_key[j - 1];
                my_w[j] = my_w[j - 1];
                --j;
            }
            my_key[j] = kk;
            my_w[j] = ww;
        }
        for (int j = 0; j < m; ++j) D = __fadd_rn(D, my_w[j]);
        for (int j = 0; j < m; ++j) my_key[j] = isect_gid[my_key[j]];
    }

    // ---- outputs (a pixel outside the image writes nothing)
    if (inside) {
        const int64_t p = int64_t(py) * W + px;
        for (int j = 0; j < K; ++j) {
            const bool has = j < m;
            ids[p * K + j] = has ? int32_t(my_key[j]) : -1;
            wout[p * K + j] = has ? __fdiv_rn(my_w[j], D) : 0.0f;
        }
        cnt[p] = uint8_t(m);
    }
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
    // Top-K with registers / in the tile kernel (us): K = 8 room VGA 64 / 83, object
    // 517 x 389 101 / 216; K = 16 room VGA 169 / 141, object of 30k at VGA 176 / 139,
    // but where latency bounds the walk (few blocks, or long lists, for which
    // the capacity per tile stands) room 160 x 120 36 / 62, room 320 x 240 79 / 99,
    // object 517 x 389 191 / 325; K = 32 room 800 x 600 903 / 441, object VGA 806 /
    // 714.
    const bool latency = tiles * 4 <= kFewBlocks || f.max_isect >= kLongTopLists * tiles;
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
        const size_t dyn = size_t(K | 1) * kPix * 4 * 2;
        e = cudaFuncSetAttribute(topk_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(dyn));
        if (e != cudaSuccess) return e;
        e = pdl_launch(topk_tile_kernel, dim3(unsigned(tiles)), dim3(kThreads), dyn, s,
                       (const float4 *)slot<float4>(f, S_REC_M), (const float4 *)slot<float4>(f, S_REC_C),
                       (const float *)slot<float>(f, S_REC_A), (const float *)slot<float>(f, S_REC_H),
                       (const uint32_t *)slot<uint32_t>(f, S_IGID), (const uint2 *)slot<uint2>(f, S_RANGES),
                       f.camera.width, f.camera.height, f.params.tile_w, f.tiles_x, K, f.params.alpha_min,
                       f.params.alpha_max, f.params.T_min, ids, w, cnt);
    }
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace qr
