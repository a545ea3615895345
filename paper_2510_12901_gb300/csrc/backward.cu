// backward.cu -- gradients of the compositing (the differentiable renderer
// of Sec. 3.2 / 3.4) w.r.t. means, log-scales, quaternions, opacities and
// features.  The unscented transform only selects tiles (a piecewise-constant
// choice) and is not differentiated.
//
// The backward runs over the forward's own work items (segments of a tile
// list x sub-blocks for the camera, segments x LiDAR work items), with the
// forward's staging and pair arithmetic (pairs.cuh), so that the same
// entries contribute.  Each segment is walked front to back from the state
// the forward's merge left for it (transmittance T and the sums (F, Z, W)
// before the segment).  With Q = (F0, F1, F2, Z, W) = sum_i (c_i, tau_i, 1)
// alpha_i T_i and U = gQ . Q (gQ = dL/dQ), the gradient of a composited
// entry's alpha is
//   dL/dalpha_i = (gQ . q_i) T_i - (U - U_{<=i}) / (1 - alpha_i),
// where U comes from the ray's saved final (F, Z, W) and U_{<=i} is the
// prefix sum up to and including entry i; T_{i+1} = T_i (1 - alpha_i) is
// the forward's own product.  The closest approach gives the geometric
// gradients in a stable form: with q = M (o + tau d - mu) = (num x den) /
// |den|^2 (the closest point in the Gaussian's frame, no cancellation),
// p = M^-1 q and d = M^-1 den (envelope theorem at tau_max),
//   dD^2/dM = 2 q p^T,                        dD^2/dmu = -2 M^T q,
//   dtau/dM = -(den p^T + q d^T) / |den|^2,   dtau/dmu = M^T den / |den|^2.
// Every term of dL/dM is a product of q and den times M^-T, so with a = 2
// dL/dD^2, b = (dL/dtau) / |den|^2 and u = a q - b den,
//   dL/dM = S M^-T,  S = sum (u q^T - b q den^T)  (symmetric),
//   dL/dmu = -M^T sum u:
// 13 sums a Gaussian (6 of S, 3 of u, dL/dsigma, 3 of the features) that need neither M^-1 nor the ray's direction.  A last
// per-Gaussian kernel maps them to the raw parameters (M = S^-1 R^T, R of the
// normalised quaternion, SH colour at the direction from the camera to the
// mean).
//
// Two phases per 16 staged entries.  Lanes are rays first: each walks the
// entries in list order, as the forward, and leaves two numbers per pair in
// shared memory, w = alpha T and y = rho dL/dalpha, which is the pair's
// dL/dsigma (both 0 where the pair does not composite, y where alpha is clamped).  Then lanes are entries (two lanes each,
// half of the rays a lane): each evaluates its pairs' num and den again and
// adds the 13 terms in registers.  One shuffle a sum joins the two halves and
// four 16-byte atomics a Gaussian add them to its row.  The kernels are bound
// by instructions: summing 16 components over the warp for every (entry,
// warp), 16 shuffles with their selects and 16 atomics, and forming p and d
// per pair (three divisions) took about 280 instructions an entry, the second
// evaluation takes 75.  Measured: the 1M-Gaussian fisheye view 826 -> 594 us,
// the 2M-Gaussian LiDAR sweep 620 -> 410 us; two entries a pass (kBwPass) 583 and
// 382.  Both divide a ray's remainder as IEEE 754 rounds it and get dL/dsigma
// without a division, as the one-phase form did: 602 and 396 us (approximate
// divisions, within 2 ulp, gave the 583 and 382).
#include <math.h>

#include "pairs.cuh"
#include "render.cuh"

namespace sg {

constexpr int kG = 16;          // floats per Gaussian in the accumulator (13 used)
constexpr int kBwBatch = 16;    // staged entries a phase takes
constexpr int kBwQueue = 64;    // entries waiting to be staged: a window's, after at most 31
constexpr int kBwWarps = 4;     // warps per block of the camera's persistent grid
constexpr int kBwCamBlocks = 5;  // its blocks per SM (4: 648 us, 6: 633)
constexpr int kBwWarpsPosed = 2;   // of LiDAR's and the rolling shutter's (13 KB a warp; 3: 422 us)

// A ray's walk over its composited entries.
struct RayGrad {
    float gQ[5];     // dL/d(F0, F1, F2, Z, W)
    float T, U, Ut;  // transmittance and gQ . Q before the entry, gQ . Q of the ray
};

// Front-to-back step of one composited entry with features q: returns (w, y).
__device__ __forceinline__ float2 ray_step(RayGrad &r, const PairEval &pe, const float q[3])
{
    const float w = pe.alpha * r.T;
    const float gq = r.gQ[0] * q[0] + r.gQ[1] * q[1] + r.gQ[2] * q[2] + r.gQ[3] * pe.tau + r.gQ[4];
    const float Ua = r.U + gq * w, om = 1.f - pe.alpha;
    const float dLda = gq * r.T - (r.Ut - Ua) / om;
    r.U = Ua;
    r.T = r.T * om;
    return make_float2(w, pe.clamped ? 0.f : dLda * pe.rho);
}

// The sums of one Gaussian.
struct GaussSums {
    float S[6];      // 00 01 02 11 12 22
    float u[3];
    float y;
    float F[3];
};

__device__ __forceinline__ void clear(GaussSums &g)
{
#pragma unroll
    for (int k = 0; k < 6; ++k) g.S[k] = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) g.u[k] = g.F[k] = 0.f;
    g.y = 0.f;
}

// Add one pair: num scaled by 1 / nscale, den, sigma, (w, y) and the ray's
// upstream (gF, gZ).
__device__ __forceinline__ void add_pair(GaussSums &g, const float n[3], const float e[3],
                                         float nscale, float sigma, float2 wy, const float gF[3],
                                         float gZ)
{
    const float inv = __fdividef(1.f, e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);
    const float c = inv * nscale;
    const float q[3] = {(n[1] * e[2] - n[2] * e[1]) * c, (n[2] * e[0] - n[0] * e[2]) * c,
                        (n[0] * e[1] - n[1] * e[0]) * c};
    // a = 2 dL/dD^2 = -sigma y (dalpha/dD^2 = -sigma rho / 2); b = gZ w / |den|^2
    const float x = sigma * wy.y, b = gZ * wy.x * inv;
    float u[3], bq[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u[k] = -(x * q[k] + b * e[k]);
        bq[k] = b * q[k];
        g.u[k] += u[k];
        g.F[k] += gF[k] * wy.x;
    }
    g.y += wy.y;
    g.S[0] += u[0] * q[0] - bq[0] * e[0];
    g.S[1] += u[0] * q[1] - bq[0] * e[1];
    g.S[2] += u[0] * q[2] - bq[0] * e[2];
    g.S[3] += u[1] * q[1] - bq[1] * e[1];
    g.S[4] += u[1] * q[2] - bq[1] * e[2];
    g.S[5] += u[2] * q[2] - bq[2] * e[2];
}

// Join the halves of an entry's rays (lanes L and L ^ 16) and add the sums to
// the Gaussian's row: S 0..5, u 6..8, sum y 9, F 10..12.  Every lane calls it;
// `use`: the entry has a composited pair.
__device__ __forceinline__ void add_sums(GaussSums &g, bool use, float *row)
{
#pragma unroll
    for (int k = 0; k < 6; ++k) g.S[k] += __shfl_xor_sync(0xffffffffu, g.S[k], 16);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        g.u[k] += __shfl_xor_sync(0xffffffffu, g.u[k], 16);
        g.F[k] += __shfl_xor_sync(0xffffffffu, g.F[k], 16);
    }
    g.y += __shfl_xor_sync(0xffffffffu, g.y, 16);
    if (!use) return;
    if (threadIdx.x & 16) {
        atomicAdd(reinterpret_cast<float4 *>(row) + 2,
                  make_float4(g.u[2], g.y, g.F[0], g.F[1]));
        atomicAdd(row + 12, g.F[2]);
    } else {
        atomicAdd(reinterpret_cast<float4 *>(row), make_float4(g.S[0], g.S[1], g.S[2], g.S[3]));
        atomicAdd(reinterpret_cast<float4 *>(row) + 1,
                  make_float4(g.S[4], g.S[5], g.u[0], g.u[1]));
    }
}

// Upstream of (F0, F1, F2, Z, W) for a camera ray from dL/d(rgb, alpha,
// depth), depth = Z / W.
__device__ __forceinline__ void camera_gQ(const float *g_rgb, const float *g_alpha,
                                          const float *g_depth, int64_t r, float W, float Z,
                                          float gQ[5])
{
    gQ[0] = g_rgb ? g_rgb[3 * r] : 0.f;
    gQ[1] = g_rgb ? g_rgb[3 * r + 1] : 0.f;
    gQ[2] = g_rgb ? g_rgb[3 * r + 2] : 0.f;
    const float gd = g_depth ? g_depth[r] : 0.f, ga = g_alpha ? g_alpha[r] : 0.f;
    gQ[3] = W > 0.f ? gd / W : 0.f;
    gQ[4] = ga - (W > 0.f ? gd * Z / (W * W) : 0.f);
}

// The start of a segment's walk: the state the forward's merge left before it
// (partial slot of two float4), the ray's totals and its upstream gQ.
__device__ __forceinline__ void start_ray(RayGrad &r, const float4 *slot, const float gQ[5],
                                          const float4 F, float Z, float W)
{
    float Q[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    r.T = 1.f;
    if (slot) {
        const float4 u = slot[0], v = slot[1];
        Q[0] = u.x; Q[1] = u.y; Q[2] = u.z; Q[3] = v.x; Q[4] = u.w;
        r.T = v.y;
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) r.gQ[k] = gQ[k];
    r.Ut = gQ[0] * F.x + gQ[1] * F.y + gQ[2] * F.z + gQ[3] * Z + gQ[4] * W;
    r.U = gQ[0] * Q[0] + gQ[1] * Q[1] + gQ[2] * Q[2] + gQ[3] * Q[3] + gQ[4] * Q[4];
}

// Entries that the lanes as rays evaluate before they take the steps in turn:
// the evaluations overlap (with approximate divisions, 1M-Gaussian fisheye view: 1
// entry 601, 2 586 us; the camera's last step, 16 rays an entry, unrolled by 8 583;
// street sweep of 2M: 1 entry 407, 2 382, 3 382 us).
constexpr int kBwPass = 2;

// ------------------------------------------------------------------ camera
struct BwCam {                     // a warp's shared memory
    float4 e[8][32];               // staged entries (cam_entry's planes 0..7)
    float2 wy[kBwBatch][33];       // (w, y) per (entry, ray); rows an odd number of banks apart
    float4 ray[2][32];             // (dd, gZ), (gF, 0)
    EntryQueue<kBwQueue> q;
    uint32_t pos[32], lanes[32], gid[32];
    float ref[6];
};

// Stage the n <= 32 entries at the queue's head and add their gradients.
__device__ __forceinline__ void bw_batch(const CamRender &P, const CamPose &pose,
                                         const GRec *__restrict__ rec, BwCam &S, uint32_t head,
                                         int n, const float dh[3], const float dl[3],
                                         const float dd[3], uint32_t last, RayGrad &r,
                                         float *__restrict__ gacc)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < n) {
        const uint2 c = S.q.cand[(head + lane) % kBwQueue];
        float4 ent[9];
        cam_entry(rec[c.x], pose.t, dh, dl, ent, kResponseScale);
#pragma unroll
        for (int k = 0; k < 8; ++k) S.e[k][lane] = ent[k];
        S.lanes[lane] = c.y;
        S.pos[lane] = S.q.pos[(head + lane) % kBwQueue];
        S.gid[lane] = c.x;
    }
    __syncwarp();
    for (int b0 = 0; b0 < n; b0 += kBwBatch) {
        const int nb = min(kBwBatch, n - b0);
        uint32_t used = 0u;        // entries with a composited pair
        for (int j0 = 0; j0 < nb; j0 += kBwPass) {
            PairEval pe[kBwPass];
            bool ok[kBwPass];
#pragma unroll
            for (int k = 0; k < kBwPass; ++k) {
                const int i = min(b0 + j0 + k, n - 1);
                ok[k] = cam_pair_scaled(S.e[0][i], S.e[1][i], S.e[2][i], S.e[3][i], S.e[4][i],
                                        S.e[5][i], S.e[6][i], (S.lanes[i] >> lane) & 1u, dd,
                                        P.alpha_min, P.alpha_max, pe[k]);
                ok[k] = ok[k] && S.pos[i] <= last && j0 + k < nb;
            }
#pragma unroll
            for (int k = 0; k < kBwPass; ++k) {
                const int i = min(b0 + j0 + k, n - 1);
                float2 wy = make_float2(0.f, 0.f);
                if (ok[k]) {
                    const float4 col = S.e[7][i];
                    const float q[3] = {col.x, col.y, col.z};
                    wy = ray_step(r, pe[k], q);
                }
                if (kBwPass == 1 || j0 + k < kBwBatch) S.wy[j0 + k][lane] = wy;
                used |= (__any_sync(0xffffffffu, ok[k]) ? 1u : 0u) << (j0 + k);
            }
        }
        __syncwarp();
        if (used == 0u) continue;
        // lanes as entries: lane & 15 of the batch, rays 16 (lane >> 4) ..
        const int j = lane & 15, i = b0 + j, r0 = lane & 16;
        const bool use = (used >> j) & 1u;
        GaussSums g;
        clear(g);
        const int il = use ? i : b0;
        const float4 e0 = S.e[0][il], e1 = S.e[1][il], e2 = S.e[2][il];
        const float4 e3 = S.e[3][il], e4 = S.e[4][il], e5 = S.e[5][il];
        const float sigma = S.e[6][il].w;
#pragma unroll 8
        for (int k = 0; k < 16; ++k) {
            const float4 d = S.ray[0][r0 + k], f = S.ray[1][r0 + k];
            const float2 wy = use ? S.wy[j][r0 + k] : make_float2(0.f, 0.f);
            if (wy.x == 0.f) continue;      // not composited
            const float2 xx = make_float2(d.x, d.x), yy = make_float2(d.y, d.y);
            const float2 zz = make_float2(d.z, d.z);
            const float2 v0 = fma2(hi2(e3), zz, fma2(lo2(e3), yy, fma2(hi2(e0), xx, lo2(e0))));
            const float2 v1 = fma2(hi2(e4), zz, fma2(lo2(e4), yy, fma2(hi2(e1), xx, lo2(e1))));
            const float2 v2 = fma2(hi2(e5), zz, fma2(lo2(e5), yy, fma2(hi2(e2), xx, lo2(e2))));
            const float num[3] = {v0.x, v1.x, v2.x}, den[3] = {v0.y, v1.y, v2.y};
            const float gF[3] = {f.x, f.y, f.z};
            add_pair(g, num, den, 1.f / kResponseScale, sigma, wy, gF, d.w);
        }
        add_sums(g, use, gacc + (int64_t)S.gid[il] * kG);
        __syncwarp();
    }
}

__global__ void __launch_bounds__(32 * kBwWarps, kBwCamBlocks)
k_backward_camera(CamRender P, const GRec *rec, const uint32_t *ids,
                  const uint2 *ranges, const uint2 *items,
                  const uint2 *tile_info, const uint32_t *counts,
                  const uint32_t *crw, uint32_t *counter,
                  const float4 *partials, const float4 *__restrict__ pix,
                  const double *__restrict__ tile_dir, const RenderDesc *D,
                  const float4 *ray_state, const float4 *ray_feat,
                  const uint32_t *n_contrib, const float *g_rgb,
                  const float *g_alpha, const float *g_depth,
                  float *gacc)
{
    after_previous();
    __shared__ BwCam s_all[kBwWarps];
    __shared__ CamPose s_pose;
    load_cam_pose(D, s_pose);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    BwCam &S = s_all[threadIdx.x >> 5];
    const uint32_t n_items = counts[0];
    while (true) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(counter, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        const uint2 it = items[item];
        const int tile = (int)it.x, seg = (int)(it.y >> 3), sub = (int)(it.y & 7);
        const uint2 ti = tile_info[tile];
        const int tx = tile % P.ntx, ty = tile / P.ntx;
        const int sbx = tx * kTile + 8 * (sub & 1), sby = ty * kTile + 4 * (sub >> 1);
        const int px = sbx + (lane & 7), py = sby + (lane >> 3);
        const bool inside = px < P.W && py < P.H;
        const int64_t pidx = (int64_t)py * P.W + px;
        const float4 e = inside ? pix[pidx] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool ray_ok = inside && e.w > 0.f;
        const uint32_t last = ray_ok ? n_contrib[pidx] : 0u;
        const uint2 rg = ranges[tile];
        const uint32_t lo = rg.x + (uint32_t)seg * kSegLen;
        uint32_t hi = min(rg.y, lo + kSegLen);
        // entries idx < rg.x + last may contribute
        hi = min(hi, rg.x + __reduce_max_sync(0xffffffffu, last));
        if (hi <= lo) continue;                        // nothing of this segment composited
        if (lane == 0) cam_tile_ref(s_pose, tile_dir, tile, S.ref);
        __syncwarp();
        const float dh[3] = {S.ref[0], S.ref[1], S.ref[2]};
        const float dl[3] = {S.ref[3], S.ref[4], S.ref[5]};
        float dd[3];
        cam_ray_offset(s_pose, e, dd);
        RayGrad r;
        {
            float gQ[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            float4 st = make_float4(0.f, 0.f, 0.f, 0.f), F = st;
            if (ray_ok) {
                st = ray_state[pidx];
                F = ray_feat[pidx];
                camera_gQ(g_rgb, g_alpha, g_depth, pidx, st.y, st.z, gQ);
            }
            start_ray(r, seg > 0 ? partials + ((size_t)(ti.y + seg) * 256 + sub * 32 + lane) * 2 : nullptr,
                      gQ, F, st.z, st.y);
        }
        S.ray[0][lane] = make_float4(dd[0], dd[1], dd[2], r.gQ[3]);
        S.ray[1][lane] = make_float4(r.gQ[0], r.gQ[1], r.gQ[2], 0.f);
        // the next window's column/row word and id, loaded one window ahead
        uint32_t ncr = 0u, nid = 0u, head = 0u, tail = 0u;
        if (lo + lane < hi) {
            ncr = crw[lo + lane];
            nid = ids[lo + lane];
        }
        for (uint32_t base = lo; base < hi; base += 32) {
            // lanes whose composited entries reach this window: an entry that
            // reaches none of them contributes to no ray and is not staged
            const uint32_t act = __ballot_sync(0xffffffffu, rg.x + last > base);
            const uint32_t idx = base + lane;
            push(S.q, tail, nid, word_lanes(ncr, sub) & act, idx + 1 - rg.x);
            ncr = 0u;
            if (idx + 32 < hi) {
                ncr = crw[idx + 32];
                nid = ids[idx + 32];
            }
            const uint32_t least = base + 32 < hi ? 32u : 1u;     // at the end, what is left
            while (tail - head >= least) {
                const uint32_t n = min(32u, tail - head);
                bw_batch(P, s_pose, rec, S, head, (int)n, dh, dl, dd, last, r, gacc);
                head += n;
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ posed rays
// LiDAR items and rolling-shutter sub-blocks, whose rays lie in up to four
// slots (columns, pixel rows) with a pose each: entries are staged as by the
// forward (lidar_entry), 16 at a time, two lanes an entry, each for two of its
// slots.
struct BwPosed {                   // a warp's shared memory
    float4 s[(3 * 32 + kBwBatch * kLidEntryStride + 31) / 32][32];
    float2 wy[kBwBatch][33];
    float4 ray[3][32];             // (dd, gZ), (d, slot), (gF, 0)
    EntryQueue<kBwQueue> q;
    uint32_t pos[kBwBatch], lanes[kBwBatch], gid[kBwBatch];
};

__device__ __forceinline__ void posed_stage(const GRec *__restrict__ rec, BwPosed &S, uint32_t head,
                                            int n, const float *poses, int first, int slots,
                                            const float dh[3], const float dl[3])
{
    const int lane = threadIdx.x & 31, j = lane & 15, half = lane >> 4;
    __syncwarp();
    if (j < n) {
        const uint2 c = S.q.cand[(head + j) % kBwQueue];
        lidar_entry_slots(rec[c.x], poses, first, 2 * half, min(slots, 2 * half + 2), dh, dl, S.s, j);
        if (half == 0) {
            S.lanes[j] = c.y;
            S.pos[j] = S.q.pos[(head + j) % kBwQueue];
            S.gid[j] = c.x;
        }
    }
    __syncwarp();
}

// Phase 2 of one pair: entry j, ray k (rows of M in m).
__device__ __forceinline__ void posed_pair(GaussSums &g, BwPosed &S, int j, int k, const float4 m[3],
                                           float2 wy)
{
    if (wy.x == 0.f) return;     // not composited
    const float4 a = S.ray[0][k], d = S.ray[1][k], f = S.ray[2][k];
    const int sl = __float_as_int(d.w);
    const float4 q0 = lid_col(S.s, j, 0, sl), q1 = lid_col(S.s, j, 1, sl), q2 = lid_col(S.s, j, 2, sl);
    const float num[3] = {q0.w + q0.x * a.x + q0.y * a.y + q0.z * a.z,
                          q1.w + q1.x * a.x + q1.y * a.y + q1.z * a.z,
                          q2.w + q2.x * a.x + q2.y * a.y + q2.z * a.z};
    float den[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) den[i] = m[i].x * d.x + m[i].y * d.y + m[i].z * d.z;
    const float gF[3] = {f.x, f.y, f.z};
    add_pair(g, num, den, 1.f, m[0].w, wy, gF, a.w);
}

// ------------------------------------------------------------------ rolling shutter
// The camera backward with a pose per pixel row.
__global__ void __launch_bounds__(32 * kBwWarpsPosed)
k_backward_camera_rs(CamRender P, const GRec *rec, const uint32_t *ids,
                     const uint2 *ranges, const uint2 *items,
                     const uint2 *tile_info, const uint32_t *counts,
                     const uint32_t *crw, uint32_t *counter,
                     const float4 *partials, const float4 *__restrict__ pix,
                     const double *__restrict__ tile_dir, const float *__restrict__ poses,
                     const float4 *ray_state, const float4 *ray_feat,
                     const uint32_t *n_contrib, const float *g_rgb,
                     const float *g_alpha, const float *g_depth,
                     float *gacc)
{
    after_previous();
    __shared__ BwPosed s_all[kBwWarpsPosed];
    const int lane = threadIdx.x & 31;
    BwPosed &S = s_all[threadIdx.x >> 5];
    const uint32_t n_items = counts[0];
    while (true) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(counter, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        const uint2 it = items[item];
        const int tile = (int)it.x, seg = (int)(it.y >> 3), sub = (int)(it.y & 7);
        const uint2 ti = tile_info[tile];
        const int tx = tile % P.ntx, ty = tile / P.ntx;
        const int sbx = tx * kTile + 8 * (sub & 1), sby = ty * kTile + 4 * (sub >> 1);
        const int px = sbx + (lane & 7), py = sby + (lane >> 3);
        const bool inside = px < P.W && py < P.H;
        const int64_t pidx = (int64_t)py * P.W + px;
        const float4 e = inside ? pix[pidx] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool ray_ok = inside && e.w > 0.f;
        const uint32_t last = ray_ok ? n_contrib[pidx] : 0u;
        const uint2 rg = ranges[tile];
        const uint32_t lo = rg.x + (uint32_t)seg * kSegLen;
        uint32_t hi = min(rg.y, lo + kSegLen);
        hi = min(hi, rg.x + __reduce_max_sync(0xffffffffu, last));
        if (hi <= lo) continue;
        const int nrows = min(4, P.H - sby);
        const int row = py < P.H ? py : sby;
        const int sb = 3 + 4 * (row - sby);
        float dh[3], dl[3], dd[3], d[3];
        {
            const double *u = tile_dir + 3 * tile;
            sensor_ray(poses + 12 * sby, u[0], u[1], u[2], poses + 12 * row, e, dh, dl, dd, d);
        }
        RayGrad r;
        {
            float gQ[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            float4 st = make_float4(0.f, 0.f, 0.f, 0.f), F = st;
            if (ray_ok) {
                st = ray_state[pidx];
                F = ray_feat[pidx];
                camera_gQ(g_rgb, g_alpha, g_depth, pidx, st.y, st.z, gQ);
            }
            start_ray(r, seg > 0 ? partials + ((size_t)(ti.y + seg) * 256 + sub * 32 + lane) * 2 : nullptr,
                      gQ, F, st.z, st.y);
        }
        S.ray[0][lane] = make_float4(dd[0], dd[1], dd[2], r.gQ[3]);
        S.ray[1][lane] = make_float4(d[0], d[1], d[2], __int_as_float(row - sby));
        S.ray[2][lane] = make_float4(r.gQ[0], r.gQ[1], r.gQ[2], 0.f);
        uint32_t ncr = 0u, nid = 0u, head = 0u, tail = 0u;    // as in k_backward_camera
        if (lo + lane < hi) {
            ncr = crw[lo + lane];
            nid = ids[lo + lane];
        }
        for (uint32_t base = lo; base < hi; base += 32) {
            const uint32_t act = __ballot_sync(0xffffffffu, rg.x + last > base);
            const uint32_t idx = base + lane;
            push(S.q, tail, nid, word_lanes(ncr, sub) & act, idx + 1 - rg.x);
            ncr = 0u;
            if (idx + 32 < hi) {
                ncr = crw[idx + 32];
                nid = ids[idx + 32];
            }
            const uint32_t least = base + 32 < hi ? (uint32_t)kBwBatch : 1u;
            while (tail - head >= least) {
                const int nb = (int)min((uint32_t)kBwBatch, tail - head);
                posed_stage(rec, S, head, nb, poses, sby, nrows, dh, dl);
                head += nb;
                uint32_t used = 0u;
                for (int j = 0; j < nb; ++j) {
                    PairEval pe;
                    bool ok = lidar_pair_in(S.s, j, sb, (S.lanes[j] >> lane) & 1u, dd, d,
                                            P.alpha_min, P.alpha_max, pe);
                    ok = ok && S.pos[j] <= last;
                    float2 wy = make_float2(0.f, 0.f);
                    if (ok) {
                        const float q[3] = {S.s[1][j].w, S.s[2][j].w, lid_u(S.s, j, sb).w};
                        wy = ray_step(r, pe, q);
                    }
                    S.wy[j][lane] = wy;
                    used |= (__any_sync(0xffffffffu, ok) ? 1u : 0u) << j;
                }
                __syncwarp();
                if (used == 0u) continue;
                const int j = lane & 15, r0 = lane & 16;
                const bool use = (used >> j) & 1u;
                const int jl = use ? j : 0;
                const float4 m[3] = {S.s[0][jl], S.s[1][jl], S.s[2][jl]};
                GaussSums g;
                clear(g);
#pragma unroll 2
                for (int k = 0; k < 16; ++k)
                    posed_pair(g, S, jl, r0 + k, m,
                               use ? S.wy[j][r0 + k] : make_float2(0.f, 0.f));
                add_sums(g, use, gacc + (int64_t)S.gid[jl] * kG);
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ LiDAR
// Phase 1 by column groups, as the forward (the lanes of one column walk the
// entries whose box holds a ray of it, side by side with the other columns');
// phase 2 over the rays in each entry's own box (6 of 32 on the street sweep).
__global__ void __launch_bounds__(32 * kBwWarpsPosed)
k_backward_lidar(LidRender P, const LidarItem *__restrict__ items,
                 const uint32_t *__restrict__ item_rays, const float4 *__restrict__ ray_e,
                 const double *__restrict__ item_u, const float *__restrict__ poses,
                 const uint2 *__restrict__ tile_items, const uint32_t *lmask,
                 int64_t lmask_stride, const GRec *rec,
                 const uint32_t *ids,
                 const uint2 *ranges, const uint2 *work,
                 const uint2 *unit_info, const uint32_t *counts,
                 uint32_t *counter, const float4 *partials,
                 const float4 *ray_state, const float4 *ray_feat,
                 const uint32_t *n_contrib, const float *g_range,
                 const float *g_int, const float *g_drop,
                 const float *g_alpha, float *gacc)
{
    after_previous();
    __shared__ BwPosed s_all[kBwWarpsPosed];
    const int lane = threadIdx.x & 31;
    BwPosed &S = s_all[threadIdx.x >> 5];
    const uint32_t n_work = counts[0];
    while (true) {
        uint32_t wi = 0;
        if (lane == 0) wi = atomicAdd(counter, 1u);
        wi = __shfl_sync(0xffffffffu, wi, 0);
        if (wi >= n_work) break;
        const uint2 w = work[wi];
        const int item_id = (int)w.x;
        const uint32_t seg = w.y;
        const uint2 ui = unit_info[item_id];
        const LidarItem it = items[item_id];
        const uint32_t ray = item_rays[it.ray_off + lane];
        const bool valid = ray != 0xffffffffu;
        const uint32_t last = valid ? n_contrib[ray] : 0u;
        const uint2 rg = ranges[it.tile];
        const uint32_t lo = rg.x + seg * kSegLen;
        uint32_t hi = min(rg.y, lo + kSegLen);
        hi = min(hi, rg.x + __reduce_max_sync(0xffffffffu, last));
        if (hi <= lo) continue;
        const int c = valid ? (int)(ray % (uint32_t)P.n_cols) : it.col0;
        const int sb = 3 + 4 * (c - it.col0);
        const uint32_t gm = __match_any_sync(0xffffffffu, sb);   // lanes of this lane's column
        float dh[3], dl[3], dd[3], d[3];
        lidar_ray(it, item_u, item_id, poses, ray_e[it.ray_off + lane], c, dh, dl, dd, d);
        // the item's ray masks of the list entries (the forward's own)
        const uint32_t *lm = lmask + (int64_t)(item_id - (int)tile_items[it.tile].x) * lmask_stride;
        RayGrad r;
        {
            float gQ[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            float4 st = make_float4(0.f, 0.f, 0.f, 0.f), F = st;
            if (valid) {
                st = ray_state[ray];
                F = ray_feat[ray];
                const float W = st.y, Z = st.z, drop = st.w;
                const float gr = g_range ? g_range[ray] : 0.f;
                const float gi = g_int ? g_int[ray] : 0.f;
                const float gp = g_drop ? g_drop[ray] : 0.f;
                const float ga = g_alpha ? g_alpha[ray] : 0.f;
                // drop = softmax(F1, F2)[drop] = 1 / (1 + exp(F1 - F2))
                const float dd_ = drop * (1.f - drop);
                gQ[0] = gi;
                gQ[1] = -gp * dd_;
                gQ[2] = gp * dd_;
                gQ[3] = W > 0.f ? gr / W : 0.f;
                gQ[4] = ga - (W > 0.f ? gr * Z / (W * W) : 0.f);
            }
            start_ray(r, seg > 0 ? partials + ((size_t)(ui.y + seg) * 32 + lane) * 2 : nullptr, gQ, F,
                      st.z, st.y);
        }
        __syncwarp();
        S.ray[0][lane] = make_float4(dd[0], dd[1], dd[2], r.gQ[3]);
        S.ray[1][lane] = make_float4(d[0], d[1], d[2], __int_as_float(c - it.col0));
        S.ray[2][lane] = make_float4(r.gQ[0], r.gQ[1], r.gQ[2], 0.f);
        uint32_t nid = 0u, nm = 0u, head = 0u, tail = 0u;   // one window ahead
        if (lo + lane < hi) {
            nid = ids[lo + lane];
            nm = lm[lo + lane];
        }
        for (uint32_t base = lo; base < hi; base += 32) {
            const uint32_t act = __ballot_sync(0xffffffffu, rg.x + last > base);
            const uint32_t idx = base + lane;
            push(S.q, tail, nid, nm & act, idx + 1 - rg.x);
            nm = 0u;
            if (idx + 32 < hi) {
                nid = ids[idx + 32];
                nm = lm[idx + 32];
            }
            const uint32_t least = base + 32 < hi ? (uint32_t)kBwBatch : 1u;
            while (tail - head >= least) {
                const int nb = (int)min((uint32_t)kBwBatch, tail - head);
                posed_stage(rec, S, head, nb, poses, it.col0, it.ncols, dh, dl);
                head += nb;
                // the staged entries that reach a ray of this lane's column
                const uint32_t lj = lane < nb ? S.lanes[lane] : 0u;
                uint32_t G = 0u;
                for (uint32_t rest = 0xffffffffu; rest;) {
                    const uint32_t gm_g = __shfl_sync(0xffffffffu, gm, __ffs(rest) - 1);
                    const uint32_t Gg = __ballot_sync(0xffffffffu, (lj & gm_g) != 0u);
                    G = gm == gm_g ? Gg : G;
                    rest &= ~gm_g;
                }
                uint32_t used = 0u;      // entries this lane's ray composites
                while (__any_sync(0xffffffffu, G != 0u)) {
                    PairEval pe[kBwPass];
                    int jj[kBwPass];
                    bool in[kBwPass], ok[kBwPass];
#pragma unroll
                    for (int k = 0; k < kBwPass; ++k) {
                        const bool has = G != 0u;
                        const int j = has ? __ffs(G) - 1 : 0;
                        G &= G - 1u;
                        jj[k] = j;
                        in[k] = has && ((S.lanes[j] >> lane) & 1u);
                        ok[k] = lidar_pair_in(S.s, j, sb, in[k], dd, d, P.alpha_min, P.alpha_max,
                                              pe[k]) &&
                                S.pos[j] <= last;
                    }
#pragma unroll
                    for (int k = 0; k < kBwPass; ++k) {
                        const int j = jj[k];
                        float2 wy = make_float2(0.f, 0.f);
                        if (ok[k]) {
                            const float q[3] = {S.s[1][j].w, S.s[2][j].w, lid_u(S.s, j, sb).w};
                            wy = ray_step(r, pe[k], q);
                            used |= 1u << j;
                        }
                        if (in[k]) S.wy[j][lane] = wy;
                    }
                }
                used = __reduce_or_sync(0xffffffffu, used);
                __syncwarp();
                if (used == 0u) continue;
                const int j = lane & 15, r0 = lane & 16;
                const bool use = (used >> j) & 1u;
                const int jl = use ? j : 0;
                const float4 m[3] = {S.s[0][jl], S.s[1][jl], S.s[2][jl]};
                uint32_t rays = use ? (S.lanes[jl] >> r0) & 0xffffu : 0u;
                GaussSums g;
                clear(g);
                while (rays) {
                    const int k = r0 + __ffs(rays) - 1;
                    rays &= rays - 1u;
                    posed_pair(g, S, jl, k, m, S.wy[jl][k]);
                }
                __syncwarp();
                add_sums(g, use, gacc + (int64_t)S.gid[jl] * kG);
            }
        }
    }
}

// ------------------------------------------------------------------ parameters
// Y_k(d) and its gradient w.r.t. d (as a polynomial in d), k = 0 .. (kDeg + 1)^2 - 1.
template <int kDeg>
__device__ __forceinline__ void sh_basis(float x, float y, float z, float Y[(kDeg + 1) * (kDeg + 1)])
{
    const float xx = x * x, yy = y * y, zz = z * z;
    Y[0] = 0.28209479177387814f;
    if constexpr (kDeg >= 1) {
        const float c = 0.48860251190291992f;
        Y[1] = -c * y;
        Y[2] = c * z;
        Y[3] = -c * x;
    }
    if constexpr (kDeg >= 2) {
        const float a = 1.0925484305920792f, b = 0.31539156525252005f, h = 0.54627421529603959f;
        Y[4] = a * x * y;
        Y[5] = -a * y * z;
        Y[6] = b * (2.f * zz - xx - yy);
        Y[7] = -a * x * z;
        Y[8] = h * (xx - yy);
    }
    if constexpr (kDeg >= 3) {
        const float c0 = 0.59004358992664352f, c1 = 2.8906114426405538f;
        const float c2 = 0.45704579946446572f, c3 = 0.37317633259011540f;
        const float c5 = 1.4453057213202769f;
        Y[9] = -c0 * y * (3.f * xx - yy);
        Y[10] = c1 * x * y * z;
        Y[11] = -c2 * y * (4.f * zz - xx - yy);
        Y[12] = c3 * z * (2.f * zz - 3.f * xx - 3.f * yy);
        Y[13] = -c2 * x * (4.f * zz - xx - yy);
        Y[14] = c5 * z * (xx - yy);
        Y[15] = -c0 * x * (xx - 3.f * yy);
    }
}

// sum_k h_k grad Y_k(d).
template <int kDeg>
__device__ __forceinline__ void sh_basis_grad(float x, float y, float z,
                                              const float h[(kDeg + 1) * (kDeg + 1)], float g[3])
{
    const float xx = x * x, yy = y * y, zz = z * z;
    g[0] = g[1] = g[2] = 0.f;
    if constexpr (kDeg >= 1) {
        const float c = 0.48860251190291992f;
        g[0] -= c * h[3];
        g[1] -= c * h[1];
        g[2] += c * h[2];
    }
    if constexpr (kDeg >= 2) {
        const float a = 1.0925484305920792f, b = 0.31539156525252005f, c = 0.54627421529603959f;
        g[0] += a * y * h[4] - 2.f * b * x * h[6] - a * z * h[7] + 2.f * c * x * h[8];
        g[1] += a * x * h[4] - a * z * h[5] - 2.f * b * y * h[6] - 2.f * c * y * h[8];
        g[2] += -a * y * h[5] + 4.f * b * z * h[6] - a * x * h[7];
    }
    if constexpr (kDeg >= 3) {
        const float c0 = 0.59004358992664352f, c1 = 2.8906114426405538f;
        const float c2 = 0.45704579946446572f, c3 = 0.37317633259011540f;
        const float c5 = 1.4453057213202769f;
        g[0] += -6.f * c0 * x * y * h[9] + c1 * y * z * h[10] + 2.f * c2 * x * y * h[11] -
                6.f * c3 * x * z * h[12] - c2 * (4.f * zz - 3.f * xx - yy) * h[13] +
                2.f * c5 * x * z * h[14] - c0 * (3.f * xx - 3.f * yy) * h[15];
        g[1] += -c0 * (3.f * xx - 3.f * yy) * h[9] + c1 * x * z * h[10] -
                c2 * (4.f * zz - xx - 3.f * yy) * h[11] - 6.f * c3 * y * z * h[12] +
                2.f * c2 * x * y * h[13] - 2.f * c5 * y * z * h[14] + 6.f * c0 * x * y * h[15];
        g[2] += c1 * x * y * h[10] - 8.f * c2 * y * z * h[11] +
                c3 * (6.f * zz - 3.f * xx - 3.f * yy) * h[12] - 8.f * c2 * x * z * h[13] +
                c5 * (xx - yy) * h[14];
    }
}

constexpr int kPgThreads = 128;     // Gaussians per block of k_param_grads

// Write zeros (s NULL) or the block's rows of C floats, staged at s + row *
// stride, to out (rows g0 .. g0 + ng - 1 of [n, C]).
template <int C>
__device__ __forceinline__ void put_rows(float *__restrict__ out, int64_t g0, int ng,
                                         const float *s, int stride)
{
    if (!out) return;
    float *p = out + g0 * C;
    const int tot = ng * C;
    const int v4 = ((uintptr_t)out & 15u) == 0 ? tot / 4 : 0;   // then p is aligned, too
    auto at = [&](int i) { return s ? s[(i / C) * stride + i % C] : 0.f; };
    for (int j = threadIdx.x; j < v4; j += kPgThreads)
        reinterpret_cast<float4 *>(p)[j] =
            make_float4(at(4 * j), at(4 * j + 1), at(4 * j + 2), at(4 * j + 3));
    for (int j = 4 * v4 + threadIdx.x; j < tot; j += kPgThreads) p[j] = at(j);
}

// Add the block's rows of C floats, staged at s + row * stride, to out (rows
// g0 .. g0 + ng - 1 of [n, C]); a group of four floats is skipped if no row in
// it has a gradient (any: a bit a row).
template <int C>
__device__ __forceinline__ void add_rows(float *__restrict__ out, int64_t g0, int ng,
                                         const float *s, int stride, const uint32_t *any)
{
    if (!out) return;
    float *p = out + g0 * C;
    const int tot = ng * C;
    const int v4 = ((uintptr_t)out & 15u) == 0 ? tot / 4 : 0;   // then p is aligned, too
    auto has = [&](int row) { return (any[row >> 5] >> (row & 31)) & 1u; };
#pragma unroll 2
    for (int j = threadIdx.x; j < v4; j += kPgThreads) {
        int r[4];
        bool some = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            r[k] = (4 * j + k) / C;
            some = some || has(r[k]);
        }
        if (!some) continue;
        float4 v = reinterpret_cast<float4 *>(p)[j];
        v.x += s[r[0] * stride + 4 * j - r[0] * C];
        v.y += s[r[1] * stride + 4 * j + 1 - r[1] * C];
        v.z += s[r[2] * stride + 4 * j + 2 - r[2] * C];
        v.w += s[r[3] * stride + 4 * j + 3 - r[3] * C];
        reinterpret_cast<float4 *>(p)[j] = v;
    }
    for (int j = 4 * v4 + threadIdx.x; j < tot; j += kPgThreads)
        if (has(j / C)) p[j] += s[(j / C) * stride + j % C];
}

// The 13 sums of each Gaussian (add_sums) to the raw parameters; the rows read
// are cleared for the next backward.  kDeg: degree of the SH features, or -1
// for three features used as they are.  SH origin: (ox, oy, oz) for cameras;
// for LiDAR SH^l features and rolling shutters, the origin of the pose that
// saw the mean, whose index the projection left in the record's feat.w.
//
// Bound by HBM: 64 bytes of sums, 236 of parameters and, read and written,
// 236 of gradients for a Gaussian with one (degree 3).  The gradients are AoS
// rows, staged in shared memory and added with 16-byte accesses: one thread
// adding its own 192-byte row 4 bytes at a time, with the SH planes read twice
// and the basis in local memory, took 365 us for 1M Gaussians, now 182 (LiDAR
// features, 2M: 136 -> 96).  kWrite: the arrays' old contents do not count and
// every row is written, nothing read: 95 and 68 us, and the caller's fills (39 and
// 22 us) are gone.
template <int kDeg, bool kWrite>
__global__ void __launch_bounds__(kPgThreads)
k_param_grads(const float *__restrict__ planes, int64_t pitch, int64_t n, int lidar, float ox,
              float oy, float oz, const GRec *rec, const float *__restrict__ poses,
              ActorParams A, float beam, int posed_origin, float *gacc,
              float *gm, float *gls, float *gq,
              float *gop, float *gf)
{
    after_previous();
    constexpr int nc = kDeg < 0 ? 1 : (kDeg + 1) * (kDeg + 1), F = 3 * nc;
    constexpr int fs = F | 1;            // odd: a thread's row in banks of its own
    __shared__ float s_f[kPgThreads * fs], s_p[kPgThreads * 11];
    __shared__ uint32_t s_any[kPgThreads / 32];
    const int t = threadIdx.x;
    const int64_t g0 = (int64_t)blockIdx.x * kPgThreads, g = g0 + t;
    const int ng = n - g0 < kPgThreads ? (int)(n - g0) : kPgThreads;
    float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0, a2 = a0;
    float a3 = 0.f;
    if (t < ng) {
        const float4 *row = reinterpret_cast<const float4 *>(gacc + g * kG);
        a0 = row[0];
        a1 = row[1];
        a2 = row[2];
        a3 = row[3].x;
    }
    const bool any = a0.x != 0.f || a0.y != 0.f || a0.z != 0.f || a0.w != 0.f || a1.x != 0.f ||
                     a1.y != 0.f || a1.z != 0.f || a1.w != 0.f || a2.x != 0.f || a2.y != 0.f ||
                     a2.z != 0.f || a2.w != 0.f || a3 != 0.f;
    const uint32_t bits = __ballot_sync(0xffffffffu, any);
    if ((t & 31) == 0) s_any[t >> 5] = bits;
    if (!__syncthreads_or(any)) {
        if constexpr (kWrite) {
            put_rows<F>(gf, g0, ng, nullptr, 0);
            put_rows<3>(gm, g0, ng, nullptr, 0);
            put_rows<3>(gls, g0, ng, nullptr, 0);
            put_rows<4>(gq, g0, ng, nullptr, 0);
            put_rows<1>(gop, g0, ng, nullptr, 0);
        }
        return;
    }
    float *fo = s_f + t * fs, *po = s_p + t * 11;     // means 3, log-scales 3, quaternion 4, opacity
    if (!any) {
#pragma unroll
        for (int k = 0; k < F; ++k) fo[k] = 0.f;
#pragma unroll
        for (int k = 0; k < 11; ++k) po[k] = 0.f;
    } else {
        float4 *row = reinterpret_cast<float4 *>(gacc + g * kG);
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        row[0] = zero;
        row[1] = zero;
        row[2] = zero;
        row[3] = zero;
        const float S[9] = {a0.x, a0.y, a0.z, a0.y, a0.w, a1.x, a0.z, a1.x, a1.y};
        const float u[3] = {a1.z, a1.w, a2.x};
        const float gc[3] = {a2.z, a2.w, a3};
        // an actor's Gaussian (M_w = S^-1 (Ra R)^T, mu_w = Ra mu + t): in its own
        // frame dL/dM_k becomes Ra^T dL/dM_k and dL/dmu becomes Ra^T dL/dmu
        float Ra[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f}, ta[3] = {0.f, 0.f, 0.f};
        const int ak = A.of ? A.of[g] : -1;
        const bool actor = ak >= 0 && ak < A.n;
        if (actor) {
            const float *P = A.poses + 12 * ak;
            for (int i = 0; i < 3; ++i) {
                for (int j = 0; j < 3; ++j) Ra[3 * i + j] = P[4 * i + j];
                ta[i] = P[4 * i + 3];
            }
        }
        float mu[3], sc[3], q[4];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            mu[k] = planes[(Scene::kMean + k) * pitch + g];
            sc[k] = expf(planes[(Scene::kLogScale + k) * pitch + g]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = planes[(Scene::kQuat + k) * pitch + g];
        const float qn = sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
        const float w = q[0] / qn, x = q[1] / qn, y = q[2] / qn, z = q[3] / qn;
        const float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z),
                            2.f * (x * z + w * y), 2.f * (x * y + w * z),
                            1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                            2.f * (x * z - w * y), 2.f * (y * z + w * x),
                            1.f - 2.f * (x * x + y * y)};
        // mu in the world, for the origins of beam divergence and SH
        const float mw[3] = {Ra[0] * mu[0] + Ra[1] * mu[1] + Ra[2] * mu[2] + ta[0],
                             Ra[3] * mu[0] + Ra[4] * mu[1] + Ra[5] * mu[2] + ta[1],
                             Ra[6] * mu[0] + Ra[7] * mu[1] + Ra[8] * mu[2] + ta[2]};
        float gmu[3], gs[3], gR[9];
        if (beam > 0.f) {
            // Beam divergence (Eq. 6): the record holds M of the smoothed
            // covariance, on which the loss depends through A = M^T M =
            // Sigma_hat^-1: dL/dSigma_hat = H = -M^T S M / 2.  Sigma_hat =
            // Sigma + beam^2 (|v|^2 I - v v^T), v = mu - o, adds beam^2 (2 v
            // tr(H) - 2 H v) to dL/dmu.
            const GRec &rc = rec[g];
            const float m[9] = {rc.m0.x, rc.m0.y, rc.m0.z, rc.m1.x, rc.m1.y, rc.m1.z,
                                rc.m2.x, rc.m2.y, rc.m2.z};
            float H[9], T[9], gw[3];
            for (int k = 0; k < 3; ++k)
                for (int j = 0; j < 3; ++j)
                    T[3 * k + j] = S[3 * k] * m[j] + S[3 * k + 1] * m[3 + j] + S[3 * k + 2] * m[6 + j];
            for (int i = 0; i < 3; ++i)
                for (int j = 0; j < 3; ++j)
                    H[3 * i + j] = -0.5f * (m[i] * T[j] + m[3 + i] * T[3 + j] + m[6 + i] * T[6 + j]);
            const float *P = poses + 12 * __float_as_uint(rc.feat.w);
            const float v[3] = {mw[0] - P[3], mw[1] - P[7], mw[2] - P[11]};
            const float tr = H[0] + H[4] + H[8], b2 = beam * beam;
            for (int i = 0; i < 3; ++i)
                gw[i] = -(m[i] * u[0] + m[3 + i] * u[1] + m[6 + i] * u[2]) +
                        b2 * (2.f * v[i] * tr -
                              2.f * (H[3 * i] * v[0] + H[3 * i + 1] * v[1] + H[3 * i + 2] * v[2]));
            // in the Gaussian's own frame: Ra^T gw, Ra^T H Ra
            for (int i = 0; i < 3; ++i) gmu[i] = Ra[i] * gw[0] + Ra[3 + i] * gw[1] + Ra[6 + i] * gw[2];
            if (actor) {
                for (int i = 0; i < 3; ++i)
                    for (int j = 0; j < 3; ++j)
                        T[3 * i + j] = H[3 * i] * Ra[j] + H[3 * i + 1] * Ra[3 + j] + H[3 * i + 2] * Ra[6 + j];
                for (int i = 0; i < 3; ++i)
                    for (int j = 0; j < 3; ++j)
                        H[3 * i + j] = Ra[i] * T[j] + Ra[3 + i] * T[3 + j] + Ra[6 + i] * T[6 + j];
            }
            // Sigma = sum_k s_k^2 r_k r_k^T: dL/dls_k = 2 s_k^2 r_k^T H r_k,
            // dL/dr_k = 2 s_k^2 H r_k
            for (int k = 0; k < 3; ++k) {
                const float s2 = sc[k] * sc[k], rk[3] = {R[k], R[3 + k], R[6 + k]};
                float Hr[3];
                for (int i = 0; i < 3; ++i)
                    Hr[i] = H[3 * i] * rk[0] + H[3 * i + 1] * rk[1] + H[3 * i + 2] * rk[2];
                gs[k] = 2.f * s2 * (rk[0] * Hr[0] + rk[1] * Hr[1] + rk[2] * Hr[2]);
                for (int i = 0; i < 3; ++i) gR[3 * i + k] = 2.f * s2 * Hr[i];
            }
        } else {
            // M_k = r_k / s_k (r_k = column k of R, orthonormal), dL/dM_k = sum_j
            // S_kj s_j r_j: dL/dls_k = -dL/dM_k . M_k = -S_kk, dL/dr_k = dL/dM_k /
            // s_k, dL/dmu = -sum_k u_k r_k / s_k
            const float is[3] = {1.f / sc[0], 1.f / sc[1], 1.f / sc[2]};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                gs[k] = -S[3 * k + k];
                const float c0 = S[3 * k] * sc[0] * is[k], c1 = S[3 * k + 1] * sc[1] * is[k];
                const float c2 = S[3 * k + 2] * sc[2] * is[k];
                gmu[k] = -(u[0] * is[0] * R[3 * k] + u[1] * is[1] * R[3 * k + 1] +
                           u[2] * is[2] * R[3 * k + 2]);
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    gR[3 * i + k] = c0 * R[3 * i] + c1 * R[3 * i + 1] + c2 * R[3 * i + 2];
            }
        }
        // partial derivatives of R(w,x,y,z) (entries row-major), times 2
        const float gw_ = 2.f * (-z * gR[1] + y * gR[2] + z * gR[3] - x * gR[5] - y * gR[6] + x * gR[7]);
        const float gx_ = 2.f * (y * gR[1] + z * gR[2] + y * gR[3] - 2.f * x * gR[4] - w * gR[5] +
                                 z * gR[6] + w * gR[7] - 2.f * x * gR[8]);
        const float gy_ = 2.f * (-2.f * y * gR[0] + x * gR[1] + w * gR[2] + x * gR[3] + z * gR[5] -
                                 w * gR[6] + z * gR[7] - 2.f * y * gR[8]);
        const float gz_ = 2.f * (-2.f * z * gR[0] - w * gR[1] + x * gR[2] + w * gR[3] -
                                 2.f * z * gR[4] + y * gR[5] + x * gR[6] + y * gR[7]);
        const float dot = gw_ * w + gx_ * x + gy_ * y + gz_ * z, iq = 1.f / qn;
        po[3] = gs[0]; po[4] = gs[1]; po[5] = gs[2];
        po[6] = (gw_ - w * dot) * iq;
        po[7] = (gx_ - x * dot) * iq;
        po[8] = (gy_ - y * dot) * iq;
        po[9] = (gz_ - z * dot) * iq;
        po[10] = a2.y;
        if constexpr (kDeg < 0) {
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) fo[ch] = gc[ch];
        } else {
            if (lidar || posed_origin) {
                const float *P = poses + 12 * __float_as_uint(rec[g].feat.w);
                ox = P[3];
                oy = P[7];
                oz = P[11];
            }
            // the view direction, in the Gaussian's own frame (Ra^T (mu_w - o))
            const float wx = mw[0] - ox, wy = mw[1] - oy, wz = mw[2] - oz;
            const float mx = actor ? Ra[0] * wx + Ra[3] * wy + Ra[6] * wz : wx;
            const float my = actor ? Ra[1] * wx + Ra[4] * wy + Ra[7] * wz : wy;
            const float mz = actor ? Ra[2] * wx + Ra[5] * wy + Ra[8] * wz : wz;
            const float inv = 1.f / sqrtf(mx * mx + my * my + mz * mz);
            const float dx = mx * inv, dy = my * inv, dz = mz * inv;
            float Y[nc], h[nc], gdir[3];
            sh_basis<(kDeg < 0 ? 0 : kDeg)>(dx, dy, dz, Y);
#pragma unroll
            for (int k = 0; k < nc; ++k) h[k] = 0.f;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                float f[nc], acc = 0.f;
#pragma unroll
                for (int k = 0; k < nc; ++k) f[k] = planes[(Scene::kFeat + 3 * k + ch) * pitch + g];
#pragma unroll
                for (int k = 0; k < nc; ++k) acc += Y[k] * f[k];
                const float gch = !lidar && acc + 0.5f < 0.f ? 0.f : gc[ch];   // clamped channel
#pragma unroll
                for (int k = 0; k < nc; ++k) {
                    fo[3 * k + ch] = Y[k] * gch;
                    h[k] += gch * f[k];
                }
            }
            sh_basis_grad<(kDeg < 0 ? 0 : kDeg)>(dx, dy, dz, h, gdir);
            const float dd = gdir[0] * dx + gdir[1] * dy + gdir[2] * dz;
            gmu[0] += (gdir[0] - dx * dd) * inv;
            gmu[1] += (gdir[1] - dy * dd) * inv;
            gmu[2] += (gdir[2] - dz * dd) * inv;
        }
        po[0] = gmu[0]; po[1] = gmu[1]; po[2] = gmu[2];
    }
    __syncthreads();
    if constexpr (kWrite) {
        put_rows<F>(gf, g0, ng, s_f, fs);
        put_rows<3>(gm, g0, ng, s_p, 11);
        put_rows<3>(gls, g0, ng, s_p + 3, 11);
        put_rows<4>(gq, g0, ng, s_p + 6, 11);
        put_rows<1>(gop, g0, ng, s_p + 10, 11);
    } else {
        add_rows<F>(gf, g0, ng, s_f, fs, s_any);
        add_rows<3>(gm, g0, ng, s_p, 11, s_any);
        add_rows<3>(gls, g0, ng, s_p + 3, 11, s_any);
        add_rows<4>(gq, g0, ng, s_p + 6, 11, s_any);
        add_rows<1>(gop, g0, ng, s_p + 10, 11, s_any);
    }
}

template <bool kWrite>
static auto param_kernel(const Scene &sc)
{
    if (!sh_features(sc.feature_kind)) return k_param_grads<-1, kWrite>;
    return sc.sh_degree == 0   ? k_param_grads<0, kWrite>
           : sc.sh_degree == 1 ? k_param_grads<1, kWrite>
           : sc.sh_degree == 2 ? k_param_grads<2, kWrite>
                               : k_param_grads<3, kWrite>;
}

static sg_status finish(const Scene &sc, Frame &fr, const float o[3], float beam,
                        const sg_grads &g, bool write, cudaStream_t st)
{
    if (sc.n == 0) return SG_OK;
    auto kern = write ? param_kernel<true>(sc) : param_kernel<false>(sc);
    launch_after(kern, (unsigned)((sc.n + kPgThreads - 1) / kPgThreads), kPgThreads, 0, st,
        sc.d_planes, sc.pitch, sc.n, sc.feature_kind == SG_FEATURES_LIDAR_SH ? 1 : 0, o[0], o[1],
        o[2], (const GRec *)fr.rec.p, fr.d_lidar_poses, actor_params(sc), beam,
        fr.kind == 2 ? 1 : 0, (float *)fr.gacc.p, g.d_g_means, g.d_g_log_scales, g.d_g_quats,
        g.d_g_opacity, g.d_g_features);
    SG_LAUNCHED();
    fr.gacc_clear = true;
    return SG_OK;
}

// The accumulator, all zero: k_param_grads clears the rows it reads, so only
// a new buffer, or one whose last backward did not get that far, is cleared here.
static sg_status clear_sums(Frame &fr, int64_t n, cudaStream_t st)
{
    const void *had = fr.gacc.p;
    const size_t bytes = fr.gacc.bytes;
    sg_status s = ensure(fr.gacc, sizeof(float) * kG * (n > 0 ? n : 1));
    if (s != SG_OK) return s;
    if (fr.gacc.p != had || fr.gacc.bytes != bytes || !fr.gacc_clear)
        SG_CUDA(cudaMemsetAsync(fr.gacc.p, 0, fr.gacc.bytes, st));
    fr.gacc_clear = false;
    return SG_OK;
}

static int blocks_per_sm(const void *kern, int threads)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, 0) != cudaSuccess ||
        nb < 1)
        nb = 4;
    return nb;
}

static sg_status persistent_grid(const void *kern, int warps, int64_t max_items, int64_t &grid)
{
    int dev = 0, sms = 0;
    SG_CUDA(cudaGetDevice(&dev));
    SG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t cap = (max_items + warps - 1) / warps;
    grid = (int64_t)sms * blocks_per_sm(kern, 32 * warps);
    grid = grid < cap ? grid : cap;
    if (grid < 1) grid = 1;
    return SG_OK;
}

sg_status backward_camera(const Scene &sc, const Camera &cam, Frame &fr, const float *g_rgb,
                          const float *g_alpha, const float *g_depth, const sg_grads &g,
                          bool write, cudaStream_t st)
{
    if (fr.seg_len != kSegLen) {
        set_error("sg_backward_camera: the frame's render used another list segment length");
        return SG_ERR_INVALID;
    }
    sg_status s = clear_sums(fr, sc.n, st);
    if (s != SG_OK) return s;
    const CamRender P = cam_render_params(cam, fr.opts);
    const int nt = cam.ntx * cam.nty;
    const WorkSize ws = work_size(nt, fr.n_pairs, kSegLen, 8);
    const unsigned char *cw = (const unsigned char *)fr.camwork.p;
    uint32_t *counter = (uint32_t *)fr.scalars.p + 6;
    SG_CUDA(cudaMemsetAsync(counter, 0, sizeof(uint32_t), st));
    int64_t grid = 0;
    if (fr.kind == 2) {     // rolling shutter: poses per pixel row
        if ((s = persistent_grid((const void *)k_backward_camera_rs, kBwWarpsPosed, ws.max_items,
                                 grid)) != SG_OK)
            return s;
        launch_after(k_backward_camera_rs, (unsigned)grid, 32 * kBwWarpsPosed, 0, st,
            P, (const GRec *)fr.rec.p, (const uint32_t *)fr.pvals[fr.pair_buf].p,
            (const uint2 *)fr.ranges.p, (const uint2 *)(cw + ws.info_bytes + ws.off_bytes),
            (const uint2 *)cw, (const uint32_t *)fr.scalars.p + 4, (const uint32_t *)fr.submask.p,
            counter, (const float4 *)fr.partials.p, cam.d_pix, cam.d_tile_dir, fr.d_lidar_poses,
            (const float4 *)fr.ray_state.p, (const float4 *)fr.ray_feat.p,
            (const uint32_t *)fr.n_contrib.p, g_rgb, g_alpha, g_depth, (float *)fr.gacc.p);
        SG_LAUNCHED();
        const float o[3] = {0.f, 0.f, 0.f};
        return finish(sc, fr, o, 0.f, g, write, st);
    }
    if ((s = persistent_grid((const void *)k_backward_camera, kBwWarps, ws.max_items, grid)) != SG_OK)
        return s;
    launch_after(k_backward_camera, (unsigned)grid, 32 * kBwWarps, 0, st,
        P, (const GRec *)fr.rec.p, (const uint32_t *)fr.pvals[fr.pair_buf].p,
        (const uint2 *)fr.ranges.p, (const uint2 *)(cw + ws.info_bytes + ws.off_bytes),
        (const uint2 *)cw, (const uint32_t *)fr.scalars.p + 4, (const uint32_t *)fr.submask.p,
        counter, (const float4 *)fr.partials.p, cam.d_pix, cam.d_tile_dir,
        (const RenderDesc *)fr.desc.p, (const float4 *)fr.ray_state.p,
        (const float4 *)fr.ray_feat.p, (const uint32_t *)fr.n_contrib.p, g_rgb, g_alpha,
        g_depth, (float *)fr.gacc.p);
    SG_LAUNCHED();
    const float o[3] = {fr.c2w[3], fr.c2w[7], fr.c2w[11]};
    return finish(sc, fr, o, 0.f, g, write, st);
}

sg_status backward_lidar(const Scene &sc, const Lidar &L, Frame &fr, const float *g_range,
                         const float *g_int, const float *g_drop, const float *g_alpha,
                         const sg_grads &g, bool write, cudaStream_t st)
{
    sg_status s = clear_sums(fr, sc.n, st);
    if (s != SG_OK) return s;
    const LidRender P = lidar_render_params(L, fr.opts);
    if (L.n_items > 0) {
        const WorkSize ws = work_size(L.n_items, fr.n_pairs * L.max_items_per_tile, kSegLen, 1);
        const unsigned char *cw = (const unsigned char *)fr.camwork.p;
        uint32_t *counter = (uint32_t *)fr.scalars.p + 6;
        SG_CUDA(cudaMemsetAsync(counter, 0, sizeof(uint32_t), st));
        int64_t grid = 0;
        if ((s = persistent_grid((const void *)k_backward_lidar, kBwWarpsPosed, ws.max_items, grid)) !=
            SG_OK)
            return s;
        launch_after(k_backward_lidar, (unsigned)grid, 32 * kBwWarpsPosed, 0, st,
            P, L.d_items, L.d_item_rays, L.d_ray_e, L.d_tile_u, fr.d_lidar_poses,
            L.d_tile_items, (const uint32_t *)fr.lmask.p, fr.lmask_stride,
            (const GRec *)fr.rec.p, (const uint32_t *)fr.pvals[fr.pair_buf].p,
            (const uint2 *)fr.ranges.p, (const uint2 *)(cw + ws.info_bytes + ws.off_bytes),
            (const uint2 *)cw, (const uint32_t *)fr.scalars.p + 4, counter,
            (const float4 *)fr.partials.p, (const float4 *)fr.ray_state.p,
            (const float4 *)fr.ray_feat.p, (const uint32_t *)fr.n_contrib.p, g_range, g_int,
            g_drop, g_alpha, (float *)fr.gacc.p);
        SG_LAUNCHED();
    }
    const float o[3] = {0.f, 0.f, 0.f};
    return finish(sc, fr, o, fr.opts.beam_divergence, g, write, st);
}

}  // namespace sg
