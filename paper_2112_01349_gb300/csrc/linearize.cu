// linearize.cu -- residuals, analytic Jacobians and the Hessian blocks
// (Alg. 1: residual/Jacobian step and linear-system step; Sec. 3 Eq. 2).
//
// * camera_table_kernel: per camera, R(w) and the rotation-Jacobian factor M
//   in FP64 (rounded to T for the FP32-mixed form).
// * lin_point_kernel: point-major; per observation e, Jc, Jp and the IRLS
//   weight W, stored sqrt(W)-scaled as structure-of-arrays in point-major order
//   (the layout every later pass streams); per point C = sum Jp~^T Jp~ and
//   w = -sum Jp~^T e~ reduced in shared memory in a fixed order.
// * lin_camera_kernel: camera-major chunks; recomputes Jc (cheaper than
//   re-reading it in another order) and reduces B = sum Jc~^T Jc~ and
//   v = -sum Jc~^T e~ per chunk; cam_finalize sums the chunks of each camera
//   in order.
// * cost kernels: F = 1/2 sum rho(|e|^2) in FP64 for accept/reject.
#include "ff.cuh"
#include "mba_internal.cuh"

namespace mba {

namespace {

inline unsigned grid_for(int64_t n, int per = kBlock) {
    int64_t g = (n + per - 1) / per;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)(g < 1 ? 1 : g);
}

// Camera constants of the factored FP32 product, from the FP64 table row.
// stat: f, k1, k2, sqrt(2) times the unit quaternion of R (half-angle form, so
// that x + w c + v x c with c = v x x rotates x), t.  ctr: the 9 x 3 transform
// between a camera vector (rotation, translation, intrinsics) and the three
// triples a row holds: R M for the rotation, the identity for the translation,
// (1, 0, 0; k1, f, 0; k2, 0, f)^T for f, k1, k2 (the Jacobian of f d(r^2) is
// d, f r^2, f r^4 = the row (1, k1, k2) / (0, f, 0) / (0, 0, f) applied to
// (1, r^2, r^4)).
__device__ __forceinline__ void factored_camera(const double *row, const double *quat, float *stat, float *ctr) {
    const double root2 = 1.4142135623730951;
    stat[0] = (float)row[21];
    stat[1] = (float)row[22];
    stat[2] = (float)row[23];
#pragma unroll
    for (int q = 0; q < 4; ++q) stat[3 + q] = (float)(root2 * quat[q]);
    stat[7] = (float)row[18];
    stat[8] = (float)row[19];
    stat[9] = (float)row[20];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            ctr[3 * a + b] = (float)(row[3 * b] * row[9 + a] + row[3 * b + 1] * row[12 + a] + row[3 * b + 2] * row[15 + a]);
            ctr[9 + 3 * a + b] = a == b ? 1.f : 0.f;
        }
    const float in[9] = {1.f, stat[1], stat[2], 0.f, stat[0], 0.f, 0.f, 0.f, stat[0]};
#pragma unroll
    for (int q = 0; q < 9; ++q) ctr[18 + q] = in[q];
}

// The same transform of the block-owned FP64 product, whose rows are in the
// world frame: M for the rotation, R for the translation.
__device__ __forceinline__ void own_camera(const double *row, double *ctr) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            ctr[3 * a + b] = row[9 + 3 * b + a];
            ctr[9 + 3 * a + b] = row[3 * a + b];
        }
    const double in[9] = {1.0, row[22], row[23], 0.0, row[21], 0.0, 0.0, 0.0, row[21]};
#pragma unroll
    for (int q = 0; q < 9; ++q) ctr[18 + q] = in[q];
}

// HALF: from the half angle, where the analytic products (block-owned, gathered)
// read the table; dual numbers and a stored FP64 Jacobian keep the full angle.
template <typename T, bool HALF>
__global__ void camera_table_kernel(const double *__restrict__ cams, int32_t nc, T *__restrict__ tab,
                                    double *__restrict__ tab64, float2 *__restrict__ tabff,
                                    float *__restrict__ stat, float *__restrict__ ctr, double *__restrict__ ctr64,
                                    const DevState *st, int gate) {
    if (gate == 1 && (st->done || !st->relin)) return;
    if (gate == 2 && st->done) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nc; i += gridDim.x * blockDim.x) {
        double row[kCamTab];
        double quat[4];
        camera_table_row<HALF>(cams + 9 * (int64_t)i, row, quat);
        if (tab)
#pragma unroll
            for (int q = 0; q < kCamTab; ++q) tab[(int64_t)i * kCamTab + q] = (T)row[q];
        if (ctr64) own_camera(row, ctr64 + (int64_t)i * kCtr);
        if (ctr) factored_camera(row, quat, stat + (int64_t)i * kCamStat, ctr + (int64_t)i * kCtr);
        if (tab64)
#pragma unroll
            for (int q = 0; q < kCamTab; ++q) tab64[(int64_t)i * kCamTab + q] = row[q];
        if (tabff) {  // R, t, f, k1, k2 as float-float
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const ff v = ff_from(row[q]);
                tabff[16 * (int64_t)i + q] = make_float2(v.hi, v.lo);
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const ff v = ff_from(row[18 + q]);
                tabff[16 * (int64_t)i + 9 + q] = make_float2(v.hi, v.lo);
            }
        }
    }
}

__global__ void split_points_kernel(const double *__restrict__ pts, int64_t m, float2 *__restrict__ out,
                                    const DevState *st, int gate) {
    if (gate && st->done) return;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        const ff v = ff_from(pts[k]);
        out[k] = make_float2(v.hi, v.lo);
    }
}

// FP32 copy of the pixels for the FP32-mixed linearisation (made once).
__global__ void uv32_kernel(const double2 *__restrict__ uv, int64_t n, float2 *__restrict__ out) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const double2 v = uv[k];
        out[k] = make_float2((float)v.x, (float)v.y);
    }
}

// FP32 copy of the current points for the FP32-mixed linearisation; runs where
// the linearisation runs (same gate).  One float4 per
// point, in sorted order in the factored form.
__global__ void point_table_kernel(const double *__restrict__ pts, const int32_t *__restrict__ sp_pt, int32_t np,
                                   float4 *__restrict__ out, const DevState *st, int gate) {
    if (gate && (st->done || !st->relin)) return;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < np; s += gridDim.x * blockDim.x) {
        const int64_t j = sp_pt ? sp_pt[s] : s;
        out[s] = make_float4((float)pts[3 * j], (float)pts[3 * j + 1], (float)pts[3 * j + 2], 0.f);
    }
}

__global__ void point_table64_kernel(const double *__restrict__ pts, const int32_t *__restrict__ sp_pt, int32_t np,
                                     double *__restrict__ out, const DevState *st, int gate) {
    if (gate && (st->done || !st->relin)) return;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < np; s += gridDim.x * blockDim.x) {
        const int64_t j = sp_pt[s];
        double2 *o = (double2 *)(out + 4 * (int64_t)s);
        o[0] = make_double2(pts[3 * j], pts[3 * j + 1]);
        o[1] = make_double2(pts[3 * j + 2], 0.0);
    }
}

__global__ void split_uv_kernel(const double2 *__restrict__ uv, int64_t n, float4 *__restrict__ out) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const ff u = ff_from(uv[k].x), v = ff_from(uv[k].y);
        out[k] = make_float4(u.hi, u.lo, v.hi, v.lo);
    }
}

// F = 1/2 sum rho(|e|^2) in float-float (ff.cuh): the BAL projection of each
// observation from the float-float camera table, point and pixel, the loss in
// FP64 where Huber's square root is needed, per-thread sums in float-float.
__global__ void __launch_bounds__(kBlock) cost_partial_ff_kernel(Prob P, double *__restrict__ partial, int gate) {
    __shared__ double sred[kWarps];
    if (gate && P.st->done) return;
    const double d2 = P.delta * P.delta;
    ff acc = ff_from(0.f);
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < P.n; o += (int64_t)gridDim.x * blockDim.x) {
        const int cam = P.pm_cam[o], pt = P.pm_pt[o];
        const float2 *c = P.camff + 16 * (int64_t)cam;
        const float2 *xp = P.ptsff + 3 * (int64_t)pt;
        ff R[9], t[3], X[3];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float2 v = __ldg(c + q);
            R[q] = {v.x, v.y};
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float2 v = __ldg(c + 9 + q), x = __ldg(xp + q);
            t[q] = {v.x, v.y};
            X[q] = {x.x, x.y};
        }
        ff Pc[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
            Pc[r] = ff_add(ff_add(ff_mul(R[3 * r], X[0]), ff_mul(R[3 * r + 1], X[1])),
                           ff_add(ff_mul(R[3 * r + 2], X[2]), t[r]));
        const ff iz = ff_rcp(Pc[2]);
        const ff px = ff_neg(ff_mul(Pc[0], iz)), py = ff_neg(ff_mul(Pc[1], iz));
        const float2 fv = __ldg(c + 12), k1v = __ldg(c + 13), k2v = __ldg(c + 14);
        const ff f = {fv.x, fv.y}, k1 = {k1v.x, k1v.y}, k2 = {k2v.x, k2v.y};
        const ff r2 = ff_add(ff_mul(px, px), ff_mul(py, py));
        const ff d = ff_add(ff_from(1.f), ff_mul(r2, ff_add(k1, ff_mul(k2, r2))));
        const ff fd = ff_mul(f, d);
        const float4 uv = __ldg(P.uvff + o);
        const ff e0 = ff_sub(ff_mul(fd, px), ff{uv.x, uv.y});
        const ff e1 = ff_sub(ff_mul(fd, py), ff{uv.z, uv.w});
        const ff sq = ff_add(ff_mul(e0, e0), ff_mul(e1, e1));
        if (P.loss == MBA_LOSS_HUBER && ff_to_double(sq) > d2) {
            const double r = sqrt(ff_to_double(sq));
            acc = ff_add(acc, ff_from(2.0 * P.delta * r - d2));
        } else {
            acc = ff_add(acc, sq);
        }
    }
    const double s = block_sum(ff_to_double(acc), sred);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// Per observation of a point-major warp chunk: residual and Jacobians, the
// stored per-observation data, and the nine point-block terms q (packed
// Jp~^T Jp~, then -Jp~^T e~).
template <typename T, bool AD>
__device__ __forceinline__ void lin_point_obs(const Prob &P, int64_t o, int cam, int pt, T *q) {
    const T *__restrict__ camtab = (const T *)P.camtab;
    T *__restrict__ J = (T *)P.J;
    T *__restrict__ res = (T *)P.res;
    const int64_t np_ = P.npad;
    T X0, X1, X2, u0, u1;
    load_point<T>(P, pt, X0, X1, X2);
    load_uv<T>(P.pm_uv, P.pm_uv32, o, u0, u1);
    T e[2], Jc[18], Jp[6];
    edge_eval<T, AD>(camtab + (int64_t)cam * kCamTab, X0, X1, X2, u0, u1, e, Jc, Jp);
    zero_fixed_columns<T>(P, cam, pt, Jc, Jp);
    T rho, W;
    loss_weight<T>(P.loss, (T)P.delta, e[0] * e[0] + e[1] * e[1], &rho, &W);
    const T sw = sqrt(W);
#pragma unroll
    for (int k = 0; k < 18; ++k) Jc[k] *= sw;
#pragma unroll
    for (int k = 0; k < 6; ++k) Jp[k] *= sw;
#pragma unroll
    for (int k = 0; k < 18; ++k) J[k * np_ + o] = Jc[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) J[(18 + k) * np_ + o] = Jp[k];
    e[0] *= sw;
    e[1] *= sw;
    res[o] = e[0];
    res[np_ + o] = e[1];
    q[0] = Jp[0] * Jp[0] + Jp[3] * Jp[3];
    q[1] = Jp[0] * Jp[1] + Jp[3] * Jp[4];
    q[2] = Jp[0] * Jp[2] + Jp[3] * Jp[5];
    q[3] = Jp[1] * Jp[1] + Jp[4] * Jp[4];
    q[4] = Jp[1] * Jp[2] + Jp[4] * Jp[5];
    q[5] = Jp[2] * Jp[2] + Jp[5] * Jp[5];
    q[6] = -(Jp[0] * e[0] + Jp[3] * e[1]);
    q[7] = -(Jp[1] * e[0] + Jp[4] * e[1]);
    q[8] = -(Jp[2] * e[0] + Jp[5] * e[1]);
}

// Point-major linearisation over warp chunks (whole points, <= 32 observations,
// one per lane; or one point with a longer track): every observation's data,
// and per point C = sum Jp~^T Jp~ and w = -sum Jp~^T e~ by a segmented shuffle
// scan in a fixed order, with no shared memory or CTA barrier.
template <typename T, bool AD>
__global__ void __launch_bounds__(kBlock, 4) lin_point_kernel(Prob P, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    for (int w = blockIdx.x * nwarp + (threadIdx.x >> 5); w < P.n_wchunks; w += gridDim.x * nwarp) {
        const int2 c0 = P.wchunk[w], c1 = P.wchunk[w + 1];
        const int o0 = c0.y, m = c1.y - c0.y;
        T q[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) q[k] = T(0);
        if (m <= 32) {
            const bool act = lane < m;
            const int64_t o = (int64_t)o0 + (act ? lane : 0);
            const int npts = c1.x - c0.x;
            const int rs = lane < npts ? __ldg(P.pt_ptr + c0.x + lane) - o0 : 32;
            const unsigned starts = __reduce_or_sync(full, rs < 32 ? (1u << rs) : 0u);
            const int pt = act ? c0.x + __popc(starts & (0xffffffffu >> (31 - lane))) - 1 : -1 - lane;
            if (act) lin_point_obs<T, AD>(P, o, __ldg(P.pm_cam + o), pt, q);
            // inclusive segmented scan keyed by point; the last lane of each point writes
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int kp = __shfl_up_sync(full, pt, d);
                T v[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) v[k] = __shfl_up_sync(full, q[k], d);
                if (lane >= d && kp == pt) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) q[k] += v[k];
                }
            }
            const int nxt = __shfl_down_sync(full, pt, 1);
            if (act && (lane == m - 1 || nxt != pt)) {
#pragma unroll
                for (int k = 0; k < 6; ++k) P.Hll[6 * (int64_t)pt + k] = (double)q[k];
#pragma unroll
                for (int k = 0; k < 3; ++k) P.w[3 * (int64_t)pt + k] = (double)q[6 + k];
            }
        } else {
            // one point with a long track: 32-observation slices, then a tree
            const int pt = c0.x;
            for (int base = 0; base < m; base += 32) {
                if (base + lane < m) {
                    const int64_t o = (int64_t)o0 + base + lane;
                    T qq[9];
                    lin_point_obs<T, AD>(P, o, __ldg(P.pm_cam + o), pt, qq);
#pragma unroll
                    for (int k = 0; k < 9; ++k) q[k] += qq[k];
                }
            }
#pragma unroll
            for (int k = 0; k < 9; ++k)
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) q[k] += __shfl_xor_sync(full, q[k], d);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < 6; ++k) P.Hll[6 * (int64_t)pt + k] = (double)q[k];
#pragma unroll
                for (int k = 0; k < 3; ++k) P.w[3 * (int64_t)pt + k] = (double)q[6 + k];
            }
        }
    }
}

// H = W Jp^T Jp, g = W Jp^T p and r2 of one observation (h = W Jp), as pairs, to its
// places in the slices and in the runs.
__device__ __forceinline__ void store_hg(const Prob &P, int64_t slot, const double *h, const double *Jp, const double *pz) {
    const double2 v[5] = {make_double2(fma(h[0], Jp[0], h[3] * Jp[3]), fma(h[0], Jp[1], h[3] * Jp[4])),
                          make_double2(fma(h[0], Jp[2], h[3] * Jp[5]), fma(h[1], Jp[1], h[4] * Jp[4])),
                          make_double2(fma(h[1], Jp[2], h[4] * Jp[5]), fma(h[2], Jp[2], h[5] * Jp[5])),
                          make_double2(fma(h[0], pz[0], h[3] * pz[1]), fma(h[1], pz[0], h[4] * pz[1])),
                          make_double2(fma(h[2], pz[0], h[5] * pz[1]), fma(pz[0], pz[0], pz[1] * pz[1]))};
    double2 *r = P.r_hg + __ldg(P.sl2r + slot);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        P.sl_hg[slot + q * P.slot_cap] = v[q];
        r[q * P.rslot_cap] = v[q];
    }
}

// Point-major linearisation of the factored form over slices: per observation
// (px, py, 1/P_z) and, with a loss, W; per point C = sum W Jp^T Jp and w = -sum
// W Jp^T e, summed in the point's lanes.
// SMEM: the CTA first copies R, t, f, k1, k2 of every camera into shared memory
// (stride kRowS), so that the per-observation camera read is four 16-byte
// shared loads instead of a gather through L1.
// FP64: H = W Jp^T Jp, g = W Jp^T p, r2 (and W) per observation for the
// block-owned product; the table has 15 doubles per camera (odd: few conflicts).
template <typename T, bool SMEM>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 1024 : 512, 1) lin_slices_kernel(Prob P, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    constexpr int TS = sizeof(T) == 4 ? kRowS : 15;
    extern __shared__ __align__(16) unsigned char s_raw[];
    T *s_tab = (T *)s_raw;
    const T *__restrict__ camtab = (const T *)P.camtab;
    if (SMEM) {
        for (int e = threadIdx.x; e < 16 * P.nc; e += blockDim.x) {
            const int cam = e >> 4, q = e & 15;
            if (q < 15) s_tab[cam * TS + q] = __ldg(camtab + (int64_t)cam * kCamTab + (q < 9 ? q : q + 9));
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    const T delta = (T)P.delta;
    for (int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < P.n_slices; w += gridDim.x * nwarp) {
        const int4 sl = __ldg(P.slice + w);
        const int K = sl.w & 0xffff, lg = sl.w >> 16, in = lane >> lg;
        const int count = sl.y & 0xff;
        const int s = sl.x + (in < count ? in : 0);
        T X0, X1, X2;
        if constexpr (sizeof(T) == 4) {
            const float4 X = __ldg(P.sp_X + s);
            X0 = X.x, X1 = X.y, X2 = X.z;
        } else {
            X0 = __ldg(P.sp_X64 + 4 * (int64_t)s), X1 = __ldg(P.sp_X64 + 4 * (int64_t)s + 1);
            X2 = __ldg(P.sp_X64 + 4 * (int64_t)s + 2);
        }
        T q[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) q[k] = T(0);
        for (int k = 0; k < K; ++k) {
            const int64_t slot = (int64_t)sl.z + 32 * k + lane;
            const int cam = __ldg(P.sl_cam + slot);
            if (cam < 0) continue;
            T ct[kCamTab];
            if constexpr (sizeof(T) == 8) {
                const T *src = SMEM ? s_tab + cam * TS : camtab + (int64_t)cam * kCamTab;
#pragma unroll
                for (int r = 0; r < 9; ++r) ct[r] = src[r];
#pragma unroll
                for (int r = 0; r < 6; ++r) ct[18 + r] = src[(SMEM ? 9 : 18) + r];
            } else {
                const float4 *src = (const float4 *)(SMEM ? s_tab + cam * TS : camtab + (int64_t)cam * kCamTab);
                const float4 a = src[0], b = src[1], c = src[2], d = src[SMEM ? 3 : 4];
                ct[0] = a.x, ct[1] = a.y, ct[2] = a.z, ct[3] = a.w, ct[4] = b.x, ct[5] = b.y, ct[6] = b.z, ct[7] = b.w;
                ct[8] = c.x;
                if (SMEM) {
                    ct[18] = c.y, ct[19] = c.z, ct[20] = c.w, ct[21] = d.x, ct[22] = d.y, ct[23] = d.z;
                } else {
                    const float4 f = src[5];
                    ct[18] = d.z, ct[19] = d.w, ct[20] = f.x, ct[21] = f.y, ct[22] = f.z, ct[23] = f.w;
                }
            }
            T u0, u1;
            if constexpr (sizeof(T) == 4) {
                const float2 uv = __ldg(P.sl_uv32 + slot);
                u0 = uv.x, u1 = uv.y;
            } else {
                const double2 uv = __ldg(P.sl_uv + slot);
                u0 = uv.x, u1 = uv.y;
            }
            T e[2], Jc[18], Jp[6], pz[3];
            project<T, true>(ct, X0, X1, X2, u0, u1, e, Jc, Jp, pz);
            T rho, W;
            loss_weight<T>(P.loss, delta, e[0] * e[0] + e[1] * e[1], &rho, &W);
            T h[6];
#pragma unroll
            for (int r = 0; r < 6; ++r) h[r] = W * Jp[r];
            if constexpr (sizeof(T) == 4) {
                P.sl_px[slot] = make_float4(__int_as_float(cam), pz[0], pz[1], pz[2]);
                if (P.sl_w) P.sl_w[slot] = W;
            } else {
                store_hg(P, slot, h, Jp, pz);
                if (P.sl_w64) P.sl_w64[slot] = W;
            }
            q[0] += h[0] * Jp[0] + h[3] * Jp[3];
            q[1] += h[0] * Jp[1] + h[3] * Jp[4];
            q[2] += h[0] * Jp[2] + h[3] * Jp[5];
            q[3] += h[1] * Jp[1] + h[4] * Jp[4];
            q[4] += h[1] * Jp[2] + h[4] * Jp[5];
            q[5] += h[2] * Jp[2] + h[5] * Jp[5];
            q[6] -= h[0] * e[0] + h[3] * e[1];
            q[7] -= h[1] * e[0] + h[4] * e[1];
            q[8] -= h[2] * e[0] + h[5] * e[1];
        }
        for (int d = 1; d < (1 << lg); d <<= 1) {
#pragma unroll
            for (int k = 0; k < 9; ++k) q[k] += __shfl_xor_sync(full, q[k], d);
        }
        if (in < count && (lane & ((1 << lg) - 1)) == 0) {
            const int64_t pt = __ldg(P.sp_pt + s);
            const bool fixed = P.has_fixed && P.pt_fixed[pt];  // its Jacobian columns are zero
#pragma unroll
            for (int k = 0; k < 6; ++k) P.Hll[6 * pt + k] = fixed ? 0.0 : (double)q[k];
#pragma unroll
            for (int k = 0; k < 3; ++k) P.w[3 * pt + k] = fixed ? 0.0 : (double)q[6 + k];
        }
    }
}

// One warp per camera chunk: each lane accumulates the 54 block terms of its
// observations, then one shuffle tree per chunk (a CTA-wide reduction per
// chunk of a few hundred observations cost as much as the Jacobians).
// The FP32 instance is held to two CTAs per SM (128 registers); the FP64 one is
// bound by the FP64 pipe and keeps its registers.
template <typename T, bool AD>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? 2 : 1) lin_camera_kernel(Prob P, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    __shared__ T ctabs[kWarps][kCamTab];
    const T *__restrict__ camtab = (const T *)P.camtab;
    const T delta = (T)P.delta;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T *ctab = ctabs[wid];
    for (int c = blockIdx.x * kWarps + wid; c < P.n_cchunks; c += gridDim.x * kWarps) {
        const int cam = P.cchunk_cam[c];
        const int b0 = P.cchunk_beg[c], b1 = P.cchunk_beg[c + 1];
        __syncwarp();
        if (lane < kCamTab) ctab[lane] = camtab[(int64_t)cam * kCamTab + lane];
        __syncwarp();
        T acc[54];
#pragma unroll
        for (int q = 0; q < 54; ++q) acc[q] = T(0);
        // two-deep pipeline over this lane's observations (the point index two
        // ahead, the point and pixels one ahead), so that the dependent point
        // gather is in flight while the previous observation is worked
        int s = b0 + lane;
        int pa = s < b1 ? P.cm_pt[s] : 0;
        int pb = s + 32 < b1 ? P.cm_pt[s + 32] : 0;
        T Xa0 = T(0), Xa1 = T(0), Xa2 = T(0), ua0 = T(0), ua1 = T(0);
        if (s < b1) {
            load_point<T>(P, pa, Xa0, Xa1, Xa2);
            load_uv<T>(P.cm_uv, P.cm_uv32, s, ua0, ua1);
        }
        for (; s < b1; s += 32) {
            const int pt = pa;
            const T X0 = Xa0, X1 = Xa1, X2 = Xa2, u0 = ua0, u1 = ua1;
            const int pc = s + 64 < b1 ? P.cm_pt[s + 64] : 0;
            if (s + 32 < b1) {
                load_point<T>(P, pb, Xa0, Xa1, Xa2);
                load_uv<T>(P.cm_uv, P.cm_uv32, s + 32, ua0, ua1);
            }
            pa = pb;
            pb = pc;
            T e[2], Jc[18], Jp[6];
            edge_eval<T, AD, true, false>(ctab, X0, X1, X2, u0, u1, e, Jc, Jp);
            zero_fixed_columns<T>(P, cam, pt, Jc, (T *)nullptr);
            T rho, W;
            loss_weight<T>(P.loss, delta, e[0] * e[0] + e[1] * e[1], &rho, &W);
            const T sw = sqrt(W);
#pragma unroll
            for (int q = 0; q < 18; ++q) Jc[q] *= sw;
            e[0] *= sw;
            e[1] *= sw;
            // what the PCG camera pass reads in camera-major order
            if (P.JcmT) {
#pragma unroll
                for (int q = 0; q < 18; ++q) ((T *)P.JcmT)[(int64_t)q * P.npad + s] = Jc[q];
            }
            int idx = 0;
#pragma unroll
            for (int a = 0; a < 9; ++a)
#pragma unroll
                for (int b = a; b < 9; ++b) acc[idx++] += Jc[a] * Jc[b] + Jc[9 + a] * Jc[9 + b];
#pragma unroll
            for (int a = 0; a < 9; ++a) acc[45 + a] -= Jc[a] * e[0] + Jc[9 + a] * e[1];
        }
        // lane q (and q - 32) ends with sum q
        double mine0 = 0.0, mine1 = 0.0;
#pragma unroll
        for (int q = 0; q < 54; ++q) {
            T v = acc[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == (q & 31)) {
                if (q < 32) mine0 = (double)v;
                else mine1 = (double)v;
            }
        }
        P.cpart[54 * (int64_t)c + lane] = mine0;
        if (lane < 22) P.cpart[54 * (int64_t)c + 32 + lane] = mine1;
    }
}

// ---------------------------------------------------------------------------
// Camera blocks of the block-owned FP64 form.  In the camera frame a residual row of
// the Jacobian is ctr applied to (Y x d, d, p (1, r2, r2^2)), d a row of D =
// d(pixel)/dP and Y = R X, or X on the first-order rotation branch, where ctr has I
// in place of R M.  So B = ctr (sum W raw^T raw) ctr^T per camera, and the sum has
// 44 distinct entries: H = W D^T D (6), Y x H (9), Y x H x Y (6), g and Y x g with
// g = W D^T p (9 each, times 1, r2, r2^2), W r2 (1 .. r2^4) (5); with v's nine, 53
// sums of about 130 FP64 instructions where J^T W J from the nine columns takes 170
// beside forming them.  The 53 lane sums of a chunk are reduced by exchanging
// halves, 62 additions instead of 5 x 54.  Both matter because the FP64 pipe bounds
// the kernel (nine columns: 3.34 ms for 5.0M observations).
// The product's H and g are in the world frame, where these sums were before.  Rotated
// to the camera frame, such sums lose the entries of the viewing direction, |p|^2 of
// the others in H: an error of 3.0e-13 of S x (16 cameras, 2.0M observations)
// instead of 4.7e-14.  They are left to the point side, which has them at hand: a
// linearisation of 5.0M observations took 2.93 ms, now 2.86.
// ---------------------------------------------------------------------------
constexpr int kRawSums = 53;
__device__ __forceinline__ int raw_index(int a, int b) {  // raw components a <= b of 0..8 (rotation, translation, intrinsics)
    const int ga = a / 3, gb = b / 3, i = a - 3 * ga, k = b - 3 * gb;
    if (ga == 0) return gb == 0 ? 15 + sym3(i, k) : (gb == 1 ? 6 + 3 * i + k : 30 + 3 * k + i);
    if (ga == 1) return gb == 1 ? sym3(i, k) : 21 + 3 * k + i;
    return 39 + i + k;
}

__global__ void __launch_bounds__(kBlock, 1) lin_camera64_kernel(Prob P, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    __shared__ double ctabs[kWarps][kCamTab];
    const double *__restrict__ camtab = (const double *)P.camtab;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double *ctab = ctabs[wid];
    for (int c = blockIdx.x * kWarps + wid; c < P.n_cchunks; c += gridDim.x * kWarps) {
        const int cam = P.cchunk_cam[c];
        const int b0 = P.cchunk_beg[c], b1 = P.cchunk_beg[c + 1];
        __syncwarp();
        if (lane < kCamTab) ctab[lane] = camtab[(int64_t)cam * kCamTab + lane];
        __syncwarp();
        const bool small = __double2hiint(ctab[24]) != 0;
        double acc[64];
#pragma unroll
        for (int q = 0; q < 64; ++q) acc[q] = 0.0;
        int s = b0 + lane;
        int pn = s < b1 ? __ldg(P.cm_sp + s) : 0;
        for (; s < b1; s += 32) {
            const int64_t pt = pn;
            if (s + 32 < b1) pn = __ldg(P.cm_sp + s + 32);
            const double2 xa = __ldg((const double2 *)(P.sp_X64 + 4 * pt)), uv = __ldg(P.cm_uv + s);
            const double X0 = xa.x, X1 = xa.y, X2 = __ldg(P.sp_X64 + 4 * pt + 2);
            double e[2], Jc[18], Jp[6], pz[3];
            project<double, true>(ctab, X0, X1, X2, uv.x, uv.y, e, Jc, Jp, pz);
            double Y[3];  // R X as in project
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double y = ctab[3 * k] * X0 + ctab[3 * k + 1] * X1 + ctab[3 * k + 2] * X2;
                Y[k] = small ? (k == 0 ? X0 : (k == 1 ? X1 : X2)) : y;
            }
            double hd[4], W = 1.0;  // W D (its first two columns)
            const double D[4] = {Jc[3], Jc[4], Jc[12], Jc[13]};
            if (P.loss != MBA_LOSS_NONE) {
                double rho;
                loss_weight<double>(P.loss, P.delta, e[0] * e[0] + e[1] * e[1], &rho, &W);
#pragma unroll
                for (int q = 0; q < 4; ++q) hd[q] = W * D[q];
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) hd[q] = D[q];
            }
            const double px = pz[0], py = pz[1], r2 = fma(px, px, py * py);
            // the third entries from the first two, D's third column being D_xy p
            double H[6], g[3];
            H[0] = fma(hd[0], D[0], hd[2] * D[2]);
            H[1] = fma(hd[0], D[1], hd[2] * D[3]);
            H[3] = fma(hd[1], D[1], hd[3] * D[3]);
            H[2] = fma(px, H[0], py * H[1]);
            H[4] = fma(px, H[1], py * H[3]);
            H[5] = fma(px, H[2], py * H[4]);
            g[0] = fma(hd[0], px, hd[2] * py);
            g[1] = fma(hd[1], px, hd[3] * py);
            g[2] = fma(px, g[0], py * g[1]);
#pragma unroll
            for (int q = 0; q < 6; ++q) acc[q] += H[q];
            // U = Y x H (column k), then U x Y
            double U[3][3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double h0 = H[k], h1 = H[k == 0 ? 1 : 2 + k], h2 = H[k == 0 ? 2 : 3 + k];
                U[0][k] = fma(Y[1], h2, -Y[2] * h1);
                U[1][k] = fma(Y[2], h0, -Y[0] * h2);
                U[2][k] = fma(Y[0], h1, -Y[1] * h0);
#pragma unroll
                for (int i = 0; i < 3; ++i) acc[6 + 3 * i + k] += U[i][k];
            }
            acc[15] = fma(Y[1], U[0][2], fma(-Y[2], U[0][1], acc[15]));
            acc[16] = fma(Y[2], U[0][0], fma(-Y[0], U[0][2], acc[16]));
            acc[17] = fma(Y[0], U[0][1], fma(-Y[1], U[0][0], acc[17]));
            acc[18] = fma(Y[2], U[1][0], fma(-Y[0], U[1][2], acc[18]));
            acc[19] = fma(Y[0], U[1][1], fma(-Y[1], U[1][0], acc[19]));
            acc[20] = fma(Y[0], U[2][1], fma(-Y[1], U[2][0], acc[20]));
            const double yg[3] = {fma(Y[1], g[2], -Y[2] * g[1]), fma(Y[2], g[0], -Y[0] * g[2]), fma(Y[0], g[1], -Y[1] * g[0])};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double a1 = r2 * g[k], c1 = r2 * yg[k];
                acc[21 + k] += g[k];
                acc[24 + k] += a1;
                acc[27 + k] = fma(r2, a1, acc[27 + k]);
                acc[30 + k] += yg[k];
                acc[33 + k] += c1;
                acc[36 + k] = fma(r2, c1, acc[36 + k]);
            }
            const double q0 = P.loss != MBA_LOSS_NONE ? W * r2 : r2, q1 = q0 * r2, q2 = q1 * r2, q3 = q2 * r2;
            acc[39] += q0;
            acc[40] += q1;
            acc[41] += q2;
            acc[42] += q3;
            acc[43] = fma(q3, r2, acc[43]);
            const double y0 = fma(hd[0], e[0], hd[2] * e[1]), y1 = fma(hd[1], e[0], hd[3] * e[1]), y2 = fma(px, y0, py * y1);
            acc[44] -= y0;
            acc[45] -= y1;
            acc[46] -= y2;
            acc[47] = fma(-Y[1], y2, fma(Y[2], y1, acc[47]));
            acc[48] = fma(-Y[2], y0, fma(Y[0], y2, acc[48]));
            acc[49] = fma(-Y[0], y1, fma(Y[1], y0, acc[49]));
            double t = fma(px, e[0], py * e[1]);
            if (P.loss != MBA_LOSS_NONE) t *= W;
            const double t1 = r2 * t;
            acc[50] -= t;
            acc[51] -= t1;
            acc[52] = fma(-r2, t1, acc[52]);
        }
        __syncwarp();
        double *out = P.cpart + 54 * (int64_t)c;
#pragma unroll
        for (int w = 32; w >= 2; w >>= 1) {
            const bool up = lane & (w >> 1);
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const double send = up ? acc[q] : acc[q + w], keep = up ? acc[q + w] : acc[q];
                acc[q] = keep + __shfl_xor_sync(full, send, w >> 1);
            }
        }
        const int idx = 2 * lane;  // bit 4 chose 32, ..., bit 0 chose 2
        if (idx < kRawSums) out[idx] = acc[0];
        if (idx + 1 < kRawSums) out[idx + 1] = acc[1];
    }
}

// The factored FP32 form's camera blocks in the same way, in the camera frame:
// raw rows (RX x d, d, p (1, r2, r2^2)) with d the rows of D = d(pixel)/dP, so
// neither Jp nor M enters the loop, and the 53 sums are reduced by exchanging
// halves.  Bound by issue and by the points' gathers and the runs' 16-byte
// scatter: 184 -> 120 us for 5.0M observations, 106 -> 82 us for 3.5M.
__global__ void __launch_bounds__(kBlock, 2) lin_camera32_kernel(Prob P, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    const float *__restrict__ camtab = (const float *)P.camtab;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float delta = (float)P.delta;
    for (int c = blockIdx.x * kWarps + wid; c < P.n_cchunks; c += gridDim.x * kWarps) {
        const float *ct = camtab + (int64_t)P.cchunk_cam[c] * kCamTab;
        const int b0 = P.cchunk_beg[c], b1 = P.cchunk_beg[c + 1];
        const float R0 = __ldg(ct), R1 = __ldg(ct + 1), R2 = __ldg(ct + 2), R3 = __ldg(ct + 3), R4 = __ldg(ct + 4),
                    R5 = __ldg(ct + 5), R6 = __ldg(ct + 6), R7 = __ldg(ct + 7), R8 = __ldg(ct + 8);
        const float t0 = __ldg(ct + 18), t1 = __ldg(ct + 19), t2 = __ldg(ct + 20), f = __ldg(ct + 21),
                    k1 = __ldg(ct + 22), k2 = __ldg(ct + 23);
        float acc[64];
#pragma unroll
        for (int q = 0; q < 64; ++q) acc[q] = 0.f;
        // the point index two observations ahead, the point and pixels one ahead
        int s = b0 + lane;
        int pa = s < b1 ? __ldg(P.cm_sp + s) : 0, pb = s + 32 < b1 ? __ldg(P.cm_sp + s + 32) : 0;
        float4 Xn = make_float4(0.f, 0.f, 0.f, 0.f);
        float2 un = make_float2(0.f, 0.f);
        if (s < b1) Xn = __ldg(P.sp_X + pa), un = __ldg(P.cm_uv32 + s);
        for (; s < b1; s += 32) {
            const float4 X = Xn;
            const float2 uv = un;
            if (s + 32 < b1) {
                Xn = __ldg(P.sp_X + pb);
                un = __ldg(P.cm_uv32 + s + 32);
                if (s + 64 < b1) pb = __ldg(P.cm_sp + s + 64);
            }
            const float X0 = R0 * X.x + R1 * X.y + R2 * X.z, X1 = R3 * X.x + R4 * X.y + R5 * X.z,
                        X2 = R6 * X.x + R7 * X.y + R8 * X.z;
            const float P0 = X0 + t0, P1 = X1 + t1, P2 = X2 + t2;
            const float iz = rcp_rn(P2), px = -P0 * iz, py = -P1 * iz;
            const float r2 = px * px + py * py, d = 1.f + k1 * r2 + k2 * r2 * r2;
            const float e0 = f * d * px - uv.x, e1 = f * d * py - uv.y;
            float rho, W;
            loss_weight<float>(P.loss, delta, e0 * e0 + e1 * e1, &rho, &W);
            {
                const int64_t o = P.own ? (int64_t)P.cm2r[s] : (int64_t)s;
                (P.own ? P.r_rx : P.RXcm)[o] = make_float4(X0, X1, X2, iz);
                if (P.loss != MBA_LOSS_NONE) (P.own ? P.r_w : P.cm_w)[o] = W;
            }
            const float fd = f * d, fdd = f * (2.f * k1 + 4.f * k2 * r2), gx = fdd * px;
            const float a00 = fd + gx * px, a01 = gx * py, a11 = fd + fdd * py * py;
            float D[6], h[6];
            D[0] = -a00 * iz, D[1] = -a01 * iz, D[2] = px * D[0] + py * D[1];
            D[3] = D[1], D[4] = -a11 * iz, D[5] = px * D[3] + py * D[4];
#pragma unroll
            for (int q = 0; q < 6; ++q) h[q] = W * D[q];
            const float H[6] = {h[0] * D[0] + h[3] * D[3], h[0] * D[1] + h[3] * D[4], h[0] * D[2] + h[3] * D[5],
                                h[1] * D[1] + h[4] * D[4], h[1] * D[2] + h[4] * D[5], h[2] * D[2] + h[5] * D[5]};
            const float g[3] = {h[0] * px + h[3] * py, h[1] * px + h[4] * py, h[2] * px + h[5] * py};
#pragma unroll
            for (int q = 0; q < 6; ++q) acc[q] += H[q];
            float U[3][3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float h0 = H[k], h1 = H[k == 0 ? 1 : 2 + k], h2 = H[k == 0 ? 2 : 3 + k];
                U[0][k] = X1 * h2 - X2 * h1;
                U[1][k] = X2 * h0 - X0 * h2;
                U[2][k] = X0 * h1 - X1 * h0;
#pragma unroll
                for (int i = 0; i < 3; ++i) acc[6 + 3 * i + k] += U[i][k];
            }
            acc[15] += X1 * U[0][2] - X2 * U[0][1];
            acc[16] += X2 * U[0][0] - X0 * U[0][2];
            acc[17] += X0 * U[0][1] - X1 * U[0][0];
            acc[18] += X2 * U[1][0] - X0 * U[1][2];
            acc[19] += X0 * U[1][1] - X1 * U[1][0];
            acc[20] += X0 * U[2][1] - X1 * U[2][0];
            const float xg[3] = {X1 * g[2] - X2 * g[1], X2 * g[0] - X0 * g[2], X0 * g[1] - X1 * g[0]};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float a1 = r2 * g[k], c1 = r2 * xg[k];
                acc[21 + k] += g[k];
                acc[24 + k] += a1;
                acc[27 + k] += r2 * a1;
                acc[30 + k] += xg[k];
                acc[33 + k] += c1;
                acc[36 + k] += r2 * c1;
            }
            const float q0 = W * r2, q1 = q0 * r2, q2 = q1 * r2, q3 = q2 * r2;
            acc[39] += q0;
            acc[40] += q1;
            acc[41] += q2;
            acc[42] += q3;
            acc[43] += q3 * r2;
            const float y0 = h[0] * e0 + h[3] * e1, y1 = h[1] * e0 + h[4] * e1, y2 = h[2] * e0 + h[5] * e1;
            acc[44] -= y0;
            acc[45] -= y1;
            acc[46] -= y2;
            acc[47] -= X1 * y2 - X2 * y1;
            acc[48] -= X2 * y0 - X0 * y2;
            acc[49] -= X0 * y1 - X1 * y0;
            const float t = W * (px * e0 + py * e1), tr = r2 * t;
            acc[50] -= t;
            acc[51] -= tr;
            acc[52] -= r2 * tr;
        }
        __syncwarp();
        double *out = P.cpart + 54 * (int64_t)c;
#pragma unroll
        for (int w = 32; w >= 2; w >>= 1) {
            const bool up = lane & (w >> 1);
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const float send = up ? acc[q] : acc[q + w], keep = up ? acc[q + w] : acc[q];
                acc[q] = keep + __shfl_xor_sync(full, send, w >> 1);
            }
        }
        const int idx = 2 * lane;
        if (idx < kRawSums) out[idx] = (double)acc[0];
        if (idx + 1 < kRawSums) out[idx + 1] = (double)acc[1];
    }
}

// One camera per 64 threads: the chunk sums in order, then B = ctr raw ctr^T and
// v = ctr raw, with ctr as in factored_camera (FP64: from the table row; I for R M on
// the first-order branch, whose sums have X in place of R X).
template <typename T>
__global__ void __launch_bounds__(64) cam_finalize_raw_kernel(Prob P, const int32_t *__restrict__ cfirst, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    __shared__ double raw[54], ct[27];
    const int i = blockIdx.x, t = threadIdx.x;
    const bool fixed = P.has_fixed && P.cam_fixed[i];  // its Jacobian columns are zero
    if (t < kRawSums) {
        double s = 0.0;
        for (int c = cfirst[i]; c < cfirst[i + 1]; ++c) s += P.cpart[54 * (int64_t)c + t];
        raw[t] = fixed ? 0.0 : s;
    }
    if (t < 27) {
        if constexpr (sizeof(T) == 4) {
            ct[t] = (double)P.ctr[(int64_t)i * kCtr + t];
        } else {
            const double *row = (const double *)P.camtab + (int64_t)i * kCamTab;
            const int g = t / 9, a = (t - 9 * g) / 3, b = t % 3;
            const double rm = fma(row[3 * b], row[9 + a], fma(row[3 * b + 1], row[12 + a], row[3 * b + 2] * row[15 + a]));
            const double f = row[21], kb = row[21 + b], unit = a == b ? 1.0 : 0.0;
            const bool first_order = row[24] != 0.0;
            ct[t] = g == 0 && !first_order ? rm : (g == 2 && a == b && a > 0 ? f : (g == 2 && a == 0 && b > 0 ? kb : unit));
        }
    }
    __syncthreads();
    if (t >= 54) return;
    double r = 0.0;
    if (t < 45) {
        int a = 0, f = t;
        while (f >= 9 - a) f -= 9 - a, ++a;
        const int b = a + f, ga = a / 3 * 3, gb = b / 3 * 3;
        for (int k = 0; k < 3; ++k) {
            double m = 0.0;
            for (int l = 0; l < 3; ++l) {
                const int p = ga + k, q = gb + l;
                m = fma(raw[p <= q ? raw_index(p, q) : raw_index(q, p)], ct[3 * b + l], m);
            }
            r = fma(ct[3 * a + k], m, r);
        }
    } else {
        const int a = t - 45, g = a / 3, at = g == 0 ? 47 : (g == 1 ? 44 : 50);
        for (int k = 0; k < 3; ++k) r = fma(ct[3 * a + k], raw[at + k], r);
    }
    if (t < 45) P.Hpp[45 * (int64_t)i + t] = r;
    else P.v[9 * (int64_t)i + (t - 45)] = r;
}

__global__ void cam_finalize_kernel(Prob P, const int32_t *__restrict__ cfirst, int force) {
    if (!force && (P.st->done || !P.st->relin)) return;
    const int64_t total = (int64_t)P.nc * 54;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / 54), q = (int)(t % 54);
        double s = 0.0;
        for (int c = cfirst[i]; c < cfirst[i + 1]; ++c) s += P.cpart[54 * (int64_t)c + q];
        if (q < 45) P.Hpp[45 * (int64_t)i + q] = s;
        else P.v[9 * (int64_t)i + (q - 45)] = s;
    }
}

// FP64 cost over the point-major observations; fixed grid and order.
template <bool AD>
__global__ void __launch_bounds__(kBlock) cost_partial_kernel(Prob P, const double *__restrict__ pts,
                                                               double *__restrict__ partial, int gate) {
    __shared__ double sred[kWarps];
    if (gate && P.st->done) return;
    double acc = 0.0;
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < P.n; o += (int64_t)gridDim.x * blockDim.x) {
        const int cam = P.pm_cam[o], pt = P.pm_pt[o];
        const double2 uv = P.pm_uv[o];
        double e[2];
        edge_residual<double, AD>(P.camtab64 + (int64_t)cam * kCamTab, pts[3 * (int64_t)pt],
                                  pts[3 * (int64_t)pt + 1], pts[3 * (int64_t)pt + 2], uv.x, uv.y, e);
        double rho, W;
        loss_weight<double>(P.loss, P.delta, e[0] * e[0] + e[1] * e[1], &rho, &W);
        acc += rho;
    }
    const double s = block_sum(acc, sred);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// The same over slices (analytic problems): the point stays in registers over
// its observations and the cameras' R, t, f, k1, k2 sit in shared memory (SMEM;
// 15 doubles, an odd stride).  Bound by the FP64 pipe: 21 instructions and a
// reciprocal per observation, written as fused chains from the constant term:
// 367 -> 246 us for 5.0M observations of 1,700 cameras, 2.08 -> 1.94 ms for 29M of
// 13,000 (the table read from L2, Huber's square roots).
template <bool SMEM>
__global__ void __launch_bounds__(512, SMEM ? 1 : 2) cost_slices_kernel(Prob P, const double *__restrict__ pts,
                                                                      double *__restrict__ partial, int gate) {
    __shared__ double sred[32];
    if (gate && P.st->done) return;
    extern __shared__ __align__(16) double s_ct[];
    if (SMEM) {
        for (int e = threadIdx.x; e < 16 * P.nc; e += blockDim.x) {
            const int cam = e >> 4, q = e & 15;
            if (q < 15) s_ct[15 * cam + q] = __ldg(P.camtab64 + (int64_t)cam * kCamTab + (q < 9 ? q : q + 9));
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    double acc = 0.0;
    for (int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < P.n_slices; w += gridDim.x * nwarp) {
        const int4 sl = __ldg(P.slice + w);
        const int K = sl.w & 0xffff, in = lane >> (sl.w >> 16);
        const int64_t pt = __ldg(P.sp_pt + sl.x + (in < (sl.y & 0xff) ? in : 0));
        const double X0 = __ldg(pts + 3 * pt), X1 = __ldg(pts + 3 * pt + 1), X2 = __ldg(pts + 3 * pt + 2);
        int64_t slot = (int64_t)sl.z + lane;
        int cn = __ldg(P.sl_cam + slot);
        double2 un = __ldg(P.sl_uv + slot);
        for (int k = 0; k < K; ++k) {
            const int cam = cn;
            const double2 uv = un;
            slot += 32;
            if (k + 1 < K) {
                cn = __ldg(P.sl_cam + slot);
                un = __ldg(P.sl_uv + slot);
            }
            if (cam < 0) continue;
            double c[15];
            if (SMEM) {
#pragma unroll
                for (int q = 0; q < 15; ++q) c[q] = s_ct[15 * cam + q];
            } else {
                const double2 *row = (const double2 *)(P.camtab64 + (int64_t)cam * kCamTab);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const double2 v = __ldg(row + q);
                    c[2 * q] = v.x, c[2 * q + 1] = v.y;
                }
                c[8] = __ldg(row + 4).x;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const double2 v = __ldg(row + 9 + q);
                    c[9 + 2 * q] = v.x, c[10 + 2 * q] = v.y;
                }
            }
            const double P0 = fma(c[0], X0, fma(c[1], X1, fma(c[2], X2, c[9])));
            const double P1 = fma(c[3], X0, fma(c[4], X1, fma(c[5], X2, c[10])));
            const double P2 = fma(c[6], X0, fma(c[7], X1, fma(c[8], X2, c[11])));
            const double iz = fast_rcp(P2);
            const double px = -P0 * iz, py = -P1 * iz;
            const double r2 = fma(px, px, py * py);
            const double fd = c[12] * fma(r2, fma(c[14], r2, c[13]), 1.0);
            const double e0 = fma(fd, px, -uv.x), e1 = fma(fd, py, -uv.y);
            const double s = fma(e0, e0, e1 * e1);
            if (P.loss == MBA_LOSS_NONE) {
                acc += s;
            } else {
                acc += s > P.delta * P.delta ? fma(2.0 * P.delta, fast_sqrt(s), -P.delta * P.delta) : s;  // Huber
            }
        }
    }
    const double s = block_sum(acc, sred);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void cost_final_kernel(const double *__restrict__ partial, int nb, double *out, double *out2,
                                  const DevState *st, int gate) {
    __shared__ double sred[kWarps];
    if (gate && st->done) return;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += partial[i];
    const double s = block_sum(acc, sred);
    if (threadIdx.x == 0) {
        *out = 0.5 * s;
        if (out2) *out2 = 0.5 * s;
    }
}

template <typename T, bool AD>
__global__ void __launch_bounds__(kBlock) evaluate_slice_kernel(Prob P, const int32_t *__restrict__ ci,
                                                                 const int32_t *__restrict__ pi,
                                                                 const double2 *__restrict__ uvs, int64_t m,
                                                                 double *__restrict__ eo, double *__restrict__ jco,
                                                                 double *__restrict__ jpo) {
    const T *__restrict__ camtab = (const T *)P.camtab;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        const int cam = ci[k], pt = pi[k];
        const double2 uv = uvs[k];
        T e[2], Jc[18], Jp[6];
        edge_eval<T, AD>(camtab + (int64_t)cam * kCamTab, (T)P.pts[3 * (int64_t)pt], (T)P.pts[3 * (int64_t)pt + 1],
                         (T)P.pts[3 * (int64_t)pt + 2], (T)uv.x, (T)uv.y, e, Jc, Jp);
        eo[2 * k] = (double)e[0];
        eo[2 * k + 1] = (double)e[1];
#pragma unroll
        for (int q = 0; q < 18; ++q) jco[18 * k + q] = (double)Jc[q];
#pragma unroll
        for (int q = 0; q < 6; ++q) jpo[6 * k + q] = (double)Jp[q];
    }
}

}  // namespace

int cost_grid(const Prob &P) { return (int)grid_for(P.n); }

template <typename T>
static cudaError_t launch_table(const Prob &P, const double *cams, T *tab, double *tab64, float2 *tabff, float *stat,
                                float *ctr, double *ctr64, int gate, cudaStream_t s) {
    const unsigned g = grid_for(P.nc, 128);
    if (P.own || P.fact)
        camera_table_kernel<T, true><<<g, 128, 0, s>>>(cams, P.nc, tab, tab64, tabff, stat, ctr, ctr64, P.st, gate);
    else
        camera_table_kernel<T, false><<<g, 128, 0, s>>>(cams, P.nc, tab, tab64, tabff, stat, ctr, ctr64, P.st, gate);
    return cudaGetLastError();
}

cudaError_t launch_camera_tables(const Prob &P, const double *cams, bool for_lin, cudaStream_t s) {
    if (!for_lin)
        return launch_table<double>(P, cams, nullptr, P.camtab64, P.camff, nullptr, nullptr, nullptr, 2, s);
    if (P.fp32) return launch_table(P, cams, (float *)P.camtab, nullptr, nullptr, P.camstat, P.ctr, nullptr, 1, s);
    return launch_table(P, cams, (double *)P.camtab, nullptr, nullptr, nullptr, nullptr, P.ctr64, 1, s);
}

cudaError_t launch_camera_tables_forced(const Prob &P, const double *cams, cudaStream_t s) {
    if (P.fp32) return launch_table(P, cams, (float *)P.camtab, P.camtab64, P.camff, P.camstat, P.ctr, nullptr, 0, s);
    return launch_table(P, cams, (double *)P.camtab, P.camtab64, nullptr, nullptr, nullptr, P.ctr64, 0, s);
}

cudaError_t launch_split_observations(const Prob &P, cudaStream_t s) {
    if (P.uvff) split_uv_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P.pm_uv, P.n, P.uvff);
    if (P.pm_uv32) uv32_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P.pm_uv, P.n, P.pm_uv32);
    if (P.cm_uv32) uv32_kernel<<<grid_for(P.n), kBlock, 0, s>>>(P.cm_uv, P.n, P.cm_uv32);
    return cudaGetLastError();
}

template <typename T, bool AD>
static cudaError_t launch_lin_pair(const Prob &P, int force, cudaStream_t s) {
    if (!AD && P.n_slices > 0) {
        // one CTA per SM, with as many warps as there are slices for it
        const int smem = P.nc * (sizeof(T) == 4 ? kRowS * 4 : 15 * 8);
        const SliceGrid g = slice_grid(P, sizeof(T) == 4 ? 1024 : 512);
        if (smem <= 220 * 1024) {
            if (cudaError_t e = allow_smem((const void *)lin_slices_kernel<T, true>)) return e;
            lin_slices_kernel<T, true><<<g.ctas, g.threads, smem, s>>>(P, force);
        } else {
            lin_slices_kernel<T, false><<<g.ctas, g.threads, 0, s>>>(P, force);
        }
    } else {
        int nbp = (P.n_wchunks + kWarps - 1) / kWarps;
        if (nbp > 152 * 16) nbp = 152 * 16;
        lin_point_kernel<T, AD><<<nbp < 1 ? 1 : nbp, kBlock, 0, s>>>(P, force);
    }
    int nbc = (P.n_cchunks + kWarps - 1) / kWarps;
    if (nbc > 152 * 16) nbc = 152 * 16;
    const unsigned nb = (unsigned)(nbc < 1 ? 1 : nbc);
    if constexpr (sizeof(T) == 4 && !AD) {
        lin_camera32_kernel<<<nb, kBlock, 0, s>>>(P, force);
    } else {
        if (!AD && P.own) lin_camera64_kernel<<<nb, kBlock, 0, s>>>(P, force);
        else lin_camera_kernel<T, AD><<<nb, kBlock, 0, s>>>(P, force);
    }
    return cudaGetLastError();
}

cudaError_t launch_linearize_impl(const Prob &P, const int32_t *cfirst, int force, cudaStream_t s) {
    cudaError_t e;
    if (P.fp32) {
        point_table_kernel<<<grid_for(P.np), kBlock, 0, s>>>(P.pts, P.fact ? P.sp_pt : nullptr, P.np,
                                                             P.fact ? P.sp_X : P.pts32, P.st, force ? 0 : 1);
        e = P.autodiff ? launch_lin_pair<float, true>(P, force, s) : launch_lin_pair<float, false>(P, force, s);
    } else {
        if (P.own)
            point_table64_kernel<<<grid_for(P.np), kBlock, 0, s>>>(P.pts, P.sp_pt, P.np, P.sp_X64, P.st, force ? 0 : 1);
        e = P.autodiff ? launch_lin_pair<double, true>(P, force, s) : launch_lin_pair<double, false>(P, force, s);
    }
    if (e != cudaSuccess) return e;
    if (P.fact) cam_finalize_raw_kernel<float><<<P.nc, 64, 0, s>>>(P, cfirst, force);
    else if (P.own) cam_finalize_raw_kernel<double><<<P.nc, 64, 0, s>>>(P, cfirst, force);
    else cam_finalize_kernel<<<grid_for((int64_t)P.nc * 54), kBlock, 0, s>>>(P, cfirst, force);
    return cudaGetLastError();
}

cudaError_t launch_cost_impl(const Prob &P, const double *pts, double *partial, double *out, double *out2, int gate,
                             cudaStream_t s, bool ff) {
    int nb = cost_grid(P);
    if (ff && P.camff && P.uvff && P.ptsff) {
        split_points_kernel<<<grid_for(3 * (int64_t)P.np), kBlock, 0, s>>>(pts, 3 * (int64_t)P.np, P.ptsff, P.st, gate);
        cost_partial_ff_kernel<<<nb, kBlock, 0, s>>>(P, partial, gate);
        cost_final_kernel<<<1, kBlock, 0, s>>>(partial, nb, out, out2, P.st, gate);
        return cudaGetLastError();
    }
    if (P.sorted) {
        const int smem = P.nc * 15 * 8;
        SliceGrid g = slice_grid(P, 512);
        if (smem <= 220 * 1024) {
            if (cudaError_t e = allow_smem((const void *)cost_slices_kernel<true>)) return e;
            cost_slices_kernel<true><<<g.ctas, g.threads, smem, s>>>(P, pts, partial, gate);
        } else {
            g.ctas *= 2;
            cost_slices_kernel<false><<<g.ctas, g.threads, 0, s>>>(P, pts, partial, gate);
        }
        nb = g.ctas;
    } else if (P.autodiff) cost_partial_kernel<true><<<nb, kBlock, 0, s>>>(P, pts, partial, gate);
    else cost_partial_kernel<false><<<nb, kBlock, 0, s>>>(P, pts, partial, gate);
    cost_final_kernel<<<1, kBlock, 0, s>>>(partial, nb, out, out2, P.st, gate);
    return cudaGetLastError();
}

cudaError_t launch_evaluate_slice(const Prob &P, const int32_t *ci, const int32_t *pi, const double2 *uv, int64_t m,
                                  double *e, double *jc, double *jp, cudaStream_t s) {
    const unsigned g = grid_for(m);
    if (P.fp32) {
        if (P.autodiff) evaluate_slice_kernel<float, true><<<g, kBlock, 0, s>>>(P, ci, pi, uv, m, e, jc, jp);
        else evaluate_slice_kernel<float, false><<<g, kBlock, 0, s>>>(P, ci, pi, uv, m, e, jc, jp);
    } else {
        if (P.autodiff) evaluate_slice_kernel<double, true><<<g, kBlock, 0, s>>>(P, ci, pi, uv, m, e, jc, jp);
        else evaluate_slice_kernel<double, false><<<g, kBlock, 0, s>>>(P, ci, pi, uv, m, e, jc, jp);
    }
    return cudaGetLastError();
}

}  // namespace mba
