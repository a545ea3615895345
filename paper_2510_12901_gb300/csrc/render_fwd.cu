// render_fwd.cu -- camera compositing (Eq. 1, the response at tau_max as in
// render.cu) for frames that keep no state for a backward: images only, as
// rendered by a serving loop or a benchmark.  The work decomposition is
// k_render_camera's (persistent independent warps, tile lists split into
// segments merged by the last arriving warp, sub-block masks, live-ray
// staging) over 8x4 pixel sub-blocks; the rays are parameterised so that a
// (ray, Gaussian) pair costs fewer instructions, and no state for a backward
// (last composited entry, final sums) is tracked or written.
//
// Tangent-plane rays.  With d_T the tile's reference direction (double, split
// into two floats) and (e_1, e_2) an orthonormal basis of the plane normal to
// it, a pixel's unit direction d is written as d / (d . d_T) = d_T + u_1 e_1 +
// u_2 e_2, (u_1, u_2) computed once per camera in double.  D^2 does not depend
// on the length of the direction, and tau_max along d' = d / (d . d_T) is the
// distance along d times (d . d_T), so the distance is tau' |d'|.  With v =
// mu - o and f_k = s_k / (s_i s_j):
//   num_k = a_k + u_1 p_k1 + u_2 p_k2,  a_k = f_k M_k . (v x d_T),
//                                        p_kj = f_k M_k . (v x e_j)
//   den_k = b_k + u_1 m_k1 + u_2 m_k2,  b_k = M_k . d_T,  m_kj = M_k . e_j
//   (M v) . den = t_0 + u_1 t_1 + u_2 t_2
// so each of the seven is two FMAs per pair, against three with a 3-vector
// offset; a_k keeps the error-free moment of render.cu, and the u-terms are
// small corrections.
#include <math.h>

#include "pairs.cuh"
#include "render.cuh"

namespace sg {

constexpr int kFwdWarps = 4;        // warps per block of the persistent grid
// Blocks per SM (4 and 6: 80 registers; 8: 64, a few bytes of the merge spill).
// Few warps walk faster, and with few pairs the launch ends with the dense tiles'
// chain of merges and re-walks, the longer the fewer tiles there are; many warps
// hide more latency, which counts the more pairs there are.  Measured, 4 / 6 / 8
// blocks in us, pinhole street views, by pairs:
//   320x240    0.97M 224 / 238 / 267   3.9M 742 / 748 / 867     7.8M 834 / 793 / 871
//   640x480    1.1M 203 / 224 / 260    2.3M 298 / 333 / 375     4.5M 605 / 559 / 669
//              9.0M 1158 / 955 / 904
//   800x600    1.2M 199 / 218 / 263    2.5M 337 / 335 / 388     4.9M 713 / 595 / 670
//   1024x768   1.4M 226 / 239 / 275    2.7M 429 / 360 / 407     5.5M 902 / 756 / 724
//   1280x720   0.45M 111 / 119 / 132   1.5M 259 / 251 / 293     6.0M 1041 / 881 / 842
//   1280x960   0.42M 104 / 104 / 124   3.1M 541 / 456 / 476     6.3M 1136 / 960 / 915
//   1600x900   1.7M 335 / 289 / 340    3.4M 629 / 534 / 525
//   1920x1080  0.69M 193 / 156 / 188   2.0M 408 / 339 / 374     3.0M 582 / 492 / 482
// Renders that overlap with others fill each other's ends, and take 8: views of
// one call on streams of their own (both street views of 1M in steps queued one
// after another 4636 Mrays/s, 4392 with the rule for one view) and frames in
// capacity mode, which are a server's (12 requests 1595 and 1655 us).  Views that
// follow one another on one stream take the rule for one view (the same two views
// 1177 us with 8 blocks, 1113 with the rule).
constexpr int fwd_blocks(int64_t n_tiles, int64_t n_pairs, bool overlaps)
{
    if (overlaps) return 8;
    if (n_tiles < 4000 && n_pairs < 4500000 && n_pairs * n_tiles < 4500000000LL) return 4;
    return n_pairs < (n_tiles < 2000 ? 7000000 : n_tiles < 5000 ? 4300000 : 2700000) ? 6 : 8;
}
// List entries a warp scans at a time: kFwdPer per lane.  Those that reach a
// live ray of the sub-block (about a third on the street views) go to a queue
// and are staged 32 at a time, so that the staging pass, one entry per lane,
// runs with all its lanes busy whatever the window.  Measured (1920x1080
// pinhole, 2M Gaussians): 32 entries 636, 64 624, 96 628 us.
constexpr int kFwdPer = 2;
constexpr int kFwdWin = 32 * kFwdPer;
constexpr int kFwdStage = 32;         // staged entries held in shared memory at once
// the queue of entries to stage: a window's, after at most 31 left over
constexpr int kFwdQueue = 128;
static_assert(kFwdWin + 31 <= kFwdQueue && (kFwdQueue & (kFwdQueue - 1)) == 0, "staging queue");
// Segment length of this kernel's work items (frames that keep no backward
// state need not match the segments of a backward).  Measured on the street
// views (compositing alone fisheye / pinhole, two-view step): 128 entries
// 0.390 / 0.562 ms, 3102 Mrays/s; 256 0.363 / 0.513 ms, 3310; 384 0.367 /
// 0.503 ms, 3364; 512 0.381 / 0.508 ms, 3384.  Longer runs mean fewer
// merges; shorter ones split the densest tiles (the fisheye's) finer.
constexpr uint32_t kFwdSeg = 384;

// The tile's reference frame in world coordinates: d_T = dh + dl (from the
// double direction, as cam_tile_ref) and e_1, e_2 rotated in float.
__device__ __forceinline__ void fwd_tile_ref(const CamPose &P, const double *tile_dir,
                                             const float *tile_basis, int tile, float *s_ref)
{
    cam_tile_ref(P, tile_dir, tile, s_ref);
    const float *b = tile_basis + 6 * tile;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        s_ref[6 + i] = P.R[3 * i] * b[0] + P.R[3 * i + 1] * b[1] + P.R[3 * i + 2] * b[2];
        s_ref[9 + i] = P.R[3 * i] * b[3] + P.R[3 * i + 1] * b[4] + P.R[3 * i + 2] * b[5];
    }
}

__device__ __forceinline__ void cross3(const float a[3], const float b[3], float c[3])
{
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}

// The rays of a sub-block in the tangent plane, as a parallelogram that holds
// every valid one: centre (x, y), half-edges along the pixel rows and columns.
// s_reg: centre, row half-edge, column half-edge (2 floats each), a bound on
// |x| + |y| over it, and 1 if there is one (the four corner lanes have rays).
// Every lane calls it with its ray's coordinates.
constexpr int kRegion = 8;
__device__ __forceinline__ void fwd_region(float x, float y, bool has_ray, float *s_reg)
{
    constexpr uint32_t full = 0xffffffffu, corners = 0x81000081u;
    const uint32_t have = __ballot_sync(full, has_ray);
    const float x0 = __shfl_sync(full, x, 0), x7 = __shfl_sync(full, x, 7);
    const float x24 = __shfl_sync(full, x, 24), x31 = __shfl_sync(full, x, 31);
    const float y0 = __shfl_sync(full, y, 0), y7 = __shfl_sync(full, y, 7);
    const float y24 = __shfl_sync(full, y, 24), y31 = __shfl_sync(full, y, 31);
    const float xc = 0.25f * ((x0 + x7) + (x24 + x31)), yc = 0.25f * ((y0 + y7) + (y24 + y31));
    const float gx = 0.25f * ((x7 - x0) + (x31 - x24)), gy = 0.25f * ((y7 - y0) + (y31 - y24));
    const float hx = 0.25f * ((x24 - x0) + (x31 - x7)), hy = 0.25f * ((y24 - y0) + (y31 - y7));
    // the lanes' coordinates along the two half-edges; their largest values
    // (the lens curves the pixel grid) scale the parallelogram
    const float det = gx * hy - gy * hx, inv = 1.f / det;
    const float dx = x - xc, dy = y - yc;
    const float s = fabsf(dx * hy - dy * hx) * fabsf(inv), t = fabsf(gx * dy - gy * dx) * fabsf(inv);
    const float ks = 1.0001f * __uint_as_float(__reduce_max_sync(full, has_ray ? __float_as_uint(s) : 0u));
    const float kt = 1.0001f * __uint_as_float(__reduce_max_sync(full, has_ray ? __float_as_uint(t) : 0u));
    const bool ok = (have & corners) == corners && ks < 2.f && kt < 2.f;   // no for NaN, too
    if ((threadIdx.x & 31) == 0) {
        s_reg[0] = xc; s_reg[1] = yc;
        s_reg[2] = ks * gx; s_reg[3] = ks * gy;
        s_reg[4] = kt * hx; s_reg[5] = kt * hy;
        s_reg[6] = fabsf(xc) + fabsf(yc) + ks * (fabsf(gx) + fabsf(gy)) + kt * (fabsf(hx) + fabsf(hy));
        s_reg[7] = ok ? 1.f : 0.f;
    }
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Whether no ray of the sub-block composites the entry: alpha = sigma 2^-q
// with q = |num|^2 / |den|^2 stays below alpha_min wherever |num|^2 > c
// |den|^2, c = log2(sigma / alpha_min).  Over the parallelogram num is n_c + s
// A + t B, |s|, |t| <= 1.  For any vector u, |num| |u| >= u . n_c - |u . A| -
// |u . B|; u is taken as the point of the parallelogram nearest to 0 (by
// coordinate descent: a bad u only weakens the bound).  |den| is bounded per
// component.  Half of a pinhole street view's (entry, sub-block) pairs are left
// out (a box is mostly empty beside a long diagonal ellipse), a sixth of a
// fisheye view's; the test takes about 4 instructions a pair (a lane each, 32
// at once), the composited pair it saves about 50.  Measured, compositing:
// 1920x1080 pinhole of 2M Gaussians 938 -> 711 us; both street views of 1M in
// one step 1341 -> 1193 us; a 641x479 fisheye view (7% left out) 62 -> 64 us.
// The slack covers the rounding of the bound and of the pair
// evaluation: 4e-6 (about 30 ulp) of the size of the terms num is summed
// from, and 1e-3 relative on q.  False for any NaN.
__device__ __forceinline__ bool fwd_unseen(const float a[3], const float p1[3], const float p2[3],
                                           const float b[3], const float m1[3], const float m2[3],
                                           float sigma, float alpha_min, const float *s_reg)
{
    const float xc = s_reg[0], yc = s_reg[1], gx = s_reg[2], gy = s_reg[3];
    const float hx = s_reg[4], hy = s_reg[5];
    float n[3], A[3], B[3];
    float mag = 0.f, mp = 0.f, U2 = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        n[k] = a[k] + xc * p1[k] + yc * p2[k];
        A[k] = gx * p1[k] + gy * p2[k];
        B[k] = hx * p1[k] + hy * p2[k];
        mag += fabsf(a[k]);
        mp += fabsf(p1[k]) + fabsf(p2[k]);
        const float d = fabsf(b[k] + xc * m1[k] + yc * m2[k]) + fabsf(gx * m1[k] + gy * m2[k]) +
                        fabsf(hx * m1[k] + hy * m2[k]);
        U2 += d * d;
    }
    mag += s_reg[6] * mp;
    const float na = dot3(n, A), nb = dot3(n, B), ab = dot3(A, B);
    const float ia = __fdividef(1.f, dot3(A, A)), ib = __fdividef(1.f, dot3(B, B));
    float s = fmaxf(-1.f, fminf(1.f, -na * ia));
    float t = fmaxf(-1.f, fminf(1.f, -(nb + s * ab) * ib));
    s = fmaxf(-1.f, fminf(1.f, -(na + t * ab) * ia));
    t = fmaxf(-1.f, fminf(1.f, -(nb + s * ab) * ib));
    float u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = n[k] + s * A[k] + t * B[k];
    const float uu = dot3(u, u);
    const float low = dot3(u, n) - fabsf(dot3(u, A)) - fabsf(dot3(u, B)) - 4e-6f * mag * uu * rsqrt_approx(uu);
    const float c = 1.0002f * __log2f(__fdividef(sigma, alpha_min)) + 1e-3f;
    return low > 0.f && low * low > 1.001f * c * U2 * uu;
}

// A staged entry, 7 float4 (one per shared-memory plane):
//   k = 0..2 (a_k, b_k, p_k1, m_k1)   3 (p02, m02, p12, m12)   4 (p22, m22, t0, t1)
//   5 (t2, sigma, lane mask, c2)      6 (c0, c1, 0, 0)
// with p_kj = f_k M_k . (v x e_j) and m_kj = M_k . e_j.  The P terms (a, p)
// carry the response scale sqrt(log2(e) / 2), as in cam_pair_scaled, so that
// |num|^2 / |den|^2 is the exponent of 2.  ref: the tile's reference frame
// (dh, dl, e_1, e_2), in the warp's shared memory.
// Every lane calls it with an entry (live: one that counts).  The entries that
// some ray of the sub-block (s_reg) may composite go to the warp's planes s, in
// lane order, each with its lane mask; returns their number.  The test comes
// before the stores, so that nothing has to be moved up past the entries left
// out (moving them through shared memory took a tenth of the kernel's
// instructions: 671 -> 643 us); the features, which it does not need, are read
// after it.
__device__ __forceinline__ int fwd_entry(const GRec &r, const float4 *pfeat, bool live, const float o[3], const float *ref,
                                          const float *s_reg, float alpha_min, uint32_t lanes,
                                          float4 (*s)[kFwdStage])
{
    const float mu[3] = {r.mu_sigma.x, r.mu_sigma.y, r.mu_sigma.z}, sigma = r.mu_sigma.w;
    const float M[3][3] = {{r.m0.x, r.m0.y, r.m0.z}, {r.m1.x, r.m1.y, r.m1.z},
                           {r.m2.x, r.m2.y, r.m2.z}};
    const float f[3] = {kResponseScale * r.m0.w, kResponseScale * r.m1.w,
                        kResponseScale * r.m2.w};
    const float dh[3] = {ref[0], ref[1], ref[2]}, dl[3] = {ref[3], ref[4], ref[5]};
    const float e1[3] = {ref[6], ref[7], ref[8]}, e2[3] = {ref[9], ref[10], ref[11]};
    float w[3], vh[3], g1[3], g2[3];
    precise_moment(mu, o, dh, dl, w, vh);
    cross3(vh, e1, g1);
    cross3(vh, e2, g2);
    float a[3], p1[3], p2[3], b[3], m1[3], m2[3], mv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a[k] = f[k] * dot3(M[k], w);
        p1[k] = f[k] * dot3(M[k], g1);
        p2[k] = f[k] * dot3(M[k], g2);
        b[k] = dot3(M[k], dh);
        m1[k] = dot3(M[k], e1);
        m2[k] = dot3(M[k], e2);
        mv[k] = dot3(M[k], vh);
    }
    const float t0 = dot3(mv, b), t1 = dot3(mv, m1), t2 = dot3(mv, m2);
    const bool keep = live && (s_reg[7] == 0.f ||
                               !fwd_unseen(a, p1, p2, b, m1, m2, sigma, alpha_min, s_reg));
    const uint32_t kb = __ballot_sync(0xffffffffu, keep);
    if (keep) {
        const int t = __popc(kb & ((1u << (threadIdx.x & 31)) - 1u));
        const float4 feat = *pfeat;
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k][t] = make_float4(a[k], b[k], p1[k], m1[k]);
        s[3][t] = make_float4(p2[0], m2[0], p2[1], m2[1]);
        s[4][t] = make_float4(p2[2], m2[2], t0, t1);
        s[5][t] = make_float4(t2, sigma, __uint_as_float(lanes), feat.z);
        s[6][t] = make_float4(feat.x, feat.y, 0.f, 0.f);
    }
    return __popc(kb);
}

struct FwdAcc {
    float T, W, Z, c0, c1, c2;
};

// A ray that has stopped (or a lane without one) has T = -1: whatever alpha,
// T (1 - alpha) is then below t_min and nothing is added, so that the loop
// needs no flag of its own.
constexpr float kFwdStopped = -1.f;

// Composite the n staged entries into the lane's accumulator (ray with
// tangent-plane coordinates (x, y)).  At alpha = 0 the step changes nothing.
// The warps issue instructions in 70% of the cycles and shared memory returns
// data in 85%, so what counts is instructions an entry: numerator and
// denominator of a component go side by side through packed FMAs (1920x1080
// pinhole of 2M: 711 -> 698 us), the flag went into T, and two entries a pass
// share the loop (-> 671).
__device__ __forceinline__ void fwd_composite(const CamRender &P, float4 (*s)[kFwdStage], int n,
                                              float x, float y, FwdAcc &a)
{
    const uint32_t bit = 1u << (threadIdx.x & 31);
    const float2 xx = make_float2(x, x), yy = make_float2(y, y);
    float2 c01 = make_float2(a.c0, a.c1);
#pragma unroll 2
    for (int j = 0; j < n; ++j) {
        const float4 A = s[0][j], B = s[1][j], C = s[2][j], D = s[3][j], E = s[4][j];
        const float4 F = s[5][j], G = s[6][j];
        // (num_k, den_k) side by side
        const float2 q0 = fma2(lo2(D), yy, fma2(hi2(A), xx, lo2(A)));
        const float2 q1 = fma2(hi2(D), yy, fma2(hi2(B), xx, lo2(B)));
        const float2 q2 = fma2(lo2(E), yy, fma2(hi2(C), xx, lo2(C)));
        const float tn = fmaf(F.x, y, fmaf(E.w, x, E.z));
        const float2 q = fma2(q2, q2, fma2(q0, q0, mul2(q1, q1)));
        const float inv = __fdividef(1.f, q.y);
        const float rho = ex2_approx(-(q.x * inv));
        const float al = fminf(F.y * rho, P.alpha_max);
        const bool in = (__float_as_uint(F.z) & bit) != 0u;
        const float alpha = in && tn > 0.f && al >= P.alpha_min ? al : 0.f;
        const float w = alpha * a.T;
        const float Tn = __fsub_rn(a.T, w);
        const bool go = Tn >= P.t_min;
        const float wgt = go ? w : 0.f;
        a.T = go ? Tn : kFwdStopped;
        c01 = fma2(make_float2(wgt, wgt), lo2(G), c01);
        a.c2 += wgt * F.w;
        a.Z += wgt * (tn * inv);
        a.W += wgt;
    }
    a.c0 = c01.x;
    a.c1 = c01.y;
}

// Stage the n <= 32 entries waiting at the head of the warp's queue and
// composite the ones a ray of the sub-block may composite.
__device__ __forceinline__ void fwd_batch(const CamRender &P, const CamPose &pose,
                                          const GRec *__restrict__ rec, const float *ref,
                                          const uint2 *cand, uint32_t head, int n, float x, float y,
                                          float4 (*s)[kFwdStage], FwdAcc &a)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    // lanes without an entry take the first one's record and drop it
    const bool live = lane < n;
    const uint2 c = cand[(head + (live ? lane : 0)) % kFwdQueue];
    const int m = fwd_entry(rec[c.x], &rec[c.x].feat, live, pose.t, ref, ref + 12, P.alpha_min, c.y, s);
    __syncwarp();
    fwd_composite(P, s, m, x, y, a);
}

// Composite list entries [lo, hi) of a tile that can reach sub-block `sub`
// into the lane's accumulator.  Lanes whose ray is done take part in the
// staging and keep their state; only entries whose box holds a live ray are
// staged (their lane masks come from the column/row words, no record load).
// ref: the tile's reference frame, then the sub-block's region, which the
// first walk of an item (done = no ray) writes through `region`.  cand: the
// warp's queue of (Gaussian, lane mask) entries to stage, a ring; they are
// staged 32 at a time, so that every lane of a staging pass has one.
__device__ __forceinline__ void fwd_walk(const CamRender &P, const CamPose &pose,
                                         const GRec *__restrict__ rec,
                                         const uint32_t *__restrict__ ids,
                                         const uint32_t *__restrict__ crw, int sub, uint32_t lo,
                                         uint32_t hi, const float *ref, float x, float y,
                                         float4 (*s)[kFwdStage], uint2 *cand, FwdAcc &a,
                                         float *region = nullptr)
{
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    uint32_t head = 0u, tail = 0u;
    // the next window's column/row words and Gaussian ids (entries lane + 32 w
    // of it), loaded one window ahead
    uint32_t ncr[kFwdPer], nid[kFwdPer];
#pragma unroll
    for (int w = 0; w < kFwdPer; ++w) {
        const uint32_t i = lo + 32 * w + lane;
        ncr[w] = i < hi ? crw[i] : 0u;
        nid[w] = i < hi ? ids[i] : 0u;
    }
    if (region) fwd_region(x, y, a.T >= 0.f, region);    // while they arrive
    for (uint32_t base = lo; base < hi; base += kFwdWin) {
        const uint32_t act = __ballot_sync(0xffffffffu, a.T >= 0.f);
        if (act == 0u) return;
#pragma unroll
        for (int w = 0; w < kFwdPer; ++w) {
            const uint32_t lm = word_lanes(ncr[w], sub) & act;
            const uint32_t bw = __ballot_sync(0xffffffffu, lm != 0u);
            if (lm) cand[(tail + __popc(bw & below)) % kFwdQueue] = make_uint2(nid[w], lm);
            tail += __popc(bw);
            const uint32_t i = base + kFwdWin + 32 * w + lane;
            ncr[w] = 0u;
            if (i < hi) {
                ncr[w] = crw[i];
                nid[w] = ids[i];
            }
        }
        // after the last window, what is left over
        const uint32_t least = base + kFwdWin < hi ? 32u : 1u;
        while (tail - head >= least) {
            const uint32_t n = min(32u, tail - head);
            fwd_batch(P, pose, rec, ref, cand, head, (int)n, x, y, s, a);
            head += n;
        }
    }
}

// Partial slot layout, as k_render_camera's: (c0, c1, c2, W), (Z, T, 0,
// stopped flag), at pixel slot 32 sub + lane of the tile's 8x4 sub-block sub.
__device__ __forceinline__ void fwd_put(float4 *pq, const FwdAcc &a, bool stopped)
{
    pq[0] = make_float4(a.c0, a.c1, a.c2, a.W);
    pq[1] = make_float4(a.Z, a.T, 0.f, stopped ? 1.f : 0.f);
}

template <uint32_t kSeg, int kBlocks>
__global__ void __launch_bounds__(32 * kFwdWarps, kBlocks)
k_render_camera_fwd(CamRender P, const GRec *rec, const uint32_t *ids,
                    const uint2 *ranges, const uint2 *items,
                    const uint2 *tile_info, const uint32_t *counts,
                    const uint32_t *crw, uint32_t *counter,
                    uint32_t *arrive, float4 *partials,
                    const float4 *__restrict__ pix2, const double *__restrict__ tile_dir,
                    const float *__restrict__ tile_basis, const RenderDesc *D)
{
    after_previous();
    __shared__ float4 s_all[kFwdWarps][7][kFwdStage];
    __shared__ uint2 s_cand[kFwdWarps][kFwdQueue];
    __shared__ __align__(16) float s_refs[kFwdWarps][12 + kRegion];
    __shared__ CamPose s_pose;
    load_cam_pose(D, s_pose);
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float4(*s_e)[kFwdStage] = s_all[wib];
    uint2 *cand = s_cand[wib];
    float *s_ref = s_refs[wib];
    const uint32_t n_items = counts[0];
    while (true) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(counter, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        const uint2 it = items[item];
        const int tile = (int)it.x, seg = (int)(it.y >> 3), sub = (int)(it.y & 7);
        const uint2 ti = tile_info[tile];            // (segments, first partial slot)
        const int tx = tile % P.ntx, ty = tile / P.ntx;
        const int sbx = tx * kTile + 8 * (sub & 1), sby = ty * kTile + 4 * (sub >> 1);
        if (lane == 0) fwd_tile_ref(s_pose, tile_dir, tile_basis, tile, s_ref);
        __syncwarp();
        const int px = sbx + (lane & 7), py = sby + (lane >> 3);
        const bool inside = px < P.W && py < P.H;
        const int64_t pidx = inside ? (int64_t)py * P.W + px : -1;
        const float4 e = inside ? pix2[pidx] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool no_ray = !(inside && e.w > 0.f);
        const uint2 rg = ranges[tile];
        const uint32_t lo = rg.x + (uint32_t)seg * kSeg;
        const uint32_t hi = min(rg.y, lo + kSeg);
        FwdAcc a = {no_ray ? kFwdStopped : 1.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        fwd_walk(P, s_pose, rec, ids, crw, sub, lo, hi, s_ref, e.x, e.y, s_e, cand, a,
                 s_ref + 12);
        if (ti.x > 1) {
            // long tile: publish this run, and combine if it is the last one
            fwd_put(partials + ((size_t)(ti.y + seg) * 256 + sub * 32 + lane) * 2, a,
                    a.T < 0.f && !no_ray);
            __threadfence();
            __syncwarp();
            uint32_t prev = 0;
            if (lane == 0) prev = atomicAdd(&arrive[ti.y * 8 + sub], 1u);
            prev = __shfl_sync(0xffffffffu, prev, 0);
            if (prev != ti.x - 1) {
                __syncwarp();
                continue;
            }
            __threadfence();
            // combine the runs in list order, two runs' partials in flight at
            // a time and no walk in between: a ray that stops in run s > 0
            // keeps the state before it and its run number.  The re-walks of a
            // dense tile's sub-block (up to ~20 runs) are a serial chain of
            // the launch; keeping the partials' loads out of it shortens it ...
            const float4 *pq = partials + ((size_t)ti.y * 256 + sub * 32 + lane) * 2;
            const float4 u0 = __ldcg(pq), v0 = __ldcg(pq + 1);
            a = {v0.y, u0.w, v0.x, u0.x, u0.y, u0.z};
            bool fin = no_ray || v0.w != 0.f;
            uint32_t stop_run = 0u;
            for (uint32_t s0 = 1; s0 < ti.x; s0 += 2) {
                if (__all_sync(0xffffffffu, fin)) break;
                float4 u[2], v[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (s0 + k < ti.x) {
                        u[k] = __ldcg(pq + 512 * (s0 + k));
                        v[k] = __ldcg(pq + 512 * (s0 + k) + 1);
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (s0 + k >= ti.x) break;
                    const bool take = !fin && v[k].w == 0.f && a.T * v[k].y >= P.t_min;
                    if (take) {
                        a.c0 += a.T * u[k].x;
                        a.c1 += a.T * u[k].y;
                        a.c2 += a.T * u[k].z;
                        a.W += a.T * u[k].w;
                        a.Z += a.T * v[k].x;
                        a.T *= v[k].y;
                    } else if (!fin) {
                        stop_run = s0 + k;
                    }
                    fin = fin || !take;
                }
            }
            // ... then each run in which rays stop, walked again for them from
            // the true state before it, in list order
            bool pend = stop_run != 0u;
            while (true) {
                const uint32_t r = __reduce_min_sync(0xffffffffu, pend ? stop_run : 0xffffffffu);
                if (r == 0xffffffffu) break;
                const bool mine = pend && stop_run == r;
                const float T = a.T;
                if (!mine) a.T = kFwdStopped;
                const uint32_t l0 = rg.x + r * kSeg;
                fwd_walk(P, s_pose, rec, ids, crw, sub, l0, min(rg.y, l0 + kSeg), s_ref, e.x, e.y,
                         s_e, cand, a);
                if (!mine) a.T = T;
                pend = pend && !mine;
            }
        }
        if (pidx >= 0) {
            float *const out_rgb = D->out[0], *const out_alpha = D->out[1];
            float *const out_depth = D->out[2];
            if (out_rgb) {
                out_rgb[3 * pidx] = a.c0;
                out_rgb[3 * pidx + 1] = a.c1;
                out_rgb[3 * pidx + 2] = a.c2;
            }
            if (out_alpha) out_alpha[pidx] = a.W;
            // Z sums tau' along d'; the distance along the unit ray is tau' |d'|
            if (out_depth) out_depth[pidx] = a.W > 0.f ? a.Z * pix2[pidx].z / a.W : 0.f;
        }
        __syncwarp();
    }
}

bool camera_forward_only(const Camera &cam, const Frame &fr)
{
    return !fr.keep_state && fr.seg_len == kSegLen && cam.tangent_ok;
}

sg_status render_camera_fwd(const Camera &cam, const sg_render_opts &o, Frame &fr,
                            cudaStream_t st)
{
    const CamRender P = cam_render_params(cam, o);
    const int nt = cam.ntx * cam.nty;
    const int64_t K = fr.n_pairs;
    const WorkSize ws = work_size(nt, K, kFwdSeg, 8);
    sg_status s = ensure(fr.camwork, ws.work_bytes);
    if (s == SG_OK) s = ensure(fr.partials, ws.partial_bytes);
    if (s == SG_OK && fr.submask.bytes < 4 * (size_t)(K > 0 ? K : 1)) {
        set_error("internal: sub-block masks of the camera list missing");
        s = SG_ERR_INVALID;
    }
    if (s != SG_OK) return s;
    unsigned char *cw = (unsigned char *)fr.camwork.p;
    const uint2 *tile_info = (const uint2 *)cw;
    const uint2 *items = (const uint2 *)(cw + ws.info_bytes + ws.off_bytes);
    uint32_t *arrive = (uint32_t *)(cw + ws.info_bytes + ws.off_bytes + ws.items_bytes);
    const uint32_t *counts = (const uint32_t *)fr.scalars.p + 4;    // [0] items [1] slots
    uint32_t *counter = (uint32_t *)fr.scalars.p + 2;
    if ((s = launch_work_items(fr, ws, nullptr, nt, nt, 8, kFwdSeg, st)) != SG_OK) return s;
    const uint32_t *ids = (const uint32_t *)fr.pvals[fr.pair_buf].p;
    int dev = 0, sms = 0;
    SG_CUDA(cudaGetDevice(&dev));
    SG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t cap = (ws.max_items + kFwdWarps - 1) / kFwdWarps;
    const int nb = fwd_blocks(nt, K, fr.k_cap > 0 || fr.beside_others);
    int64_t grid = (int64_t)sms * nb;
    grid = grid < cap ? grid : cap;
    if (grid < 1) grid = 1;
    launch_after(nb > 6 ? k_render_camera_fwd<kFwdSeg, 8> : k_render_camera_fwd<kFwdSeg, 6>, (unsigned)grid, 32 * kFwdWarps, 0, st,
        P, (const GRec *)fr.rec.p, ids, (const uint2 *)fr.ranges.p, items, tile_info, counts,
        (const uint32_t *)fr.submask.p, counter, arrive, (float4 *)fr.partials.p, cam.d_pix2,
        cam.d_tile_dir, cam.d_tile_basis, (const RenderDesc *)fr.desc.p);
    SG_LAUNCHED();
    return SG_OK;
}

}  // namespace sg
