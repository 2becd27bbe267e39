// pcg.cu -- damping and block inversions, the persistent PCG on the reduced
// camera system (Alg. 2) with the implicit Schur product (Alg. 3), and the
// point back-substitution (Sec. 3 Eq. 4) with the linear model decrease.
//
// Implicit product S p = B~ p - E C~^-1 E^T p, a point pass and a camera pass
// per PCG iteration:
//   per observation  t_k = Jc~_k p_i(k),  u_k = Jp~_k^T t_k        (E^T p)
//   per point        b_j = C~_j^-1 sum_k u_k                       (C~^-1)
//   per observation  y_k = Jc~_k^T (Jp~_k b_j) added into camera i(k) (E b)
// The camera-side work (B~ p, the preconditioner B~^-1 r, dot products,
// axpys) is FP64 in both precisions, spread over all CTAs, three cameras per
// warp, with bounded grid barriers between the phases.
#include <type_traits>

#include "mba_internal.cuh"

namespace mba {

namespace {

// ---------------------------------------------------------------------------
// damping: B~ = B + mu D_B, C~ = C + mu D_C (D = clamp(diag, 1e-6, 1e32), or I)
// B~ is stored full, with its inverse (Cholesky, FP64) as the block-Jacobi
// preconditioner; C~^-1 (adjugate, FP64) is stored packed in T.  A block that
// is not positive definite sets DevState::blockfail: the LM loop rejects the
// iteration (mu grows), single-step entry points report MBA_ERR_NONFINITE.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double damp_term(int damping, double d) {
    if (damping == MBA_DAMP_IDENTITY) return 1.0;
    // clamp(d, 1e-6, 1e32) on the bit patterns (in order for positive numbers; a
    // negative one is below 1e-6 either way): integer work, off the FP64 pipe
    const long long b = max(__double_as_longlong(d), __double_as_longlong(1e-6));
    return __longlong_as_double(min(b, __double_as_longlong(1e32)));
}

__device__ __forceinline__ double current_mu(const DevState *st) {
    return st->mu_override >= 0.0 ? st->mu_override : 1.0 / st->radius;
}

// One warp per camera: B~ (full, stored for the PCG's B~ p) and its inverse.
constexpr int kDampWarps = 4;
__global__ void __launch_bounds__(32 * kDampWarps) damp_cameras_kernel(Prob P, int damping) {
    __shared__ double sA[kDampWarps][81], sY[kDampWarps][81], sil[kDampWarps][9];
    DevState *st = P.st;
    if (st->done) return;
    const double mu = current_mu(st);
    if (blockIdx.x == 0 && threadIdx.x == 0) st->mu = mu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = blockIdx.x * kDampWarps + wid; i < P.nc; i += gridDim.x * kDampWarps) {
        double *A = sA[wid];
        __syncwarp();
        for (int e = lane; e < 81; e += 32) {
            const int a = e / 9, b = e - 9 * (e / 9);
            double v = P.Hpp[45 * (int64_t)i + sym9(a, b)];
            if (a == b) v += mu * damp_term(damping, v);
            A[e] = v;
            P.Bd[81 * (int64_t)i + e] = v;
        }
        __syncwarp();
        if (!warp_spd_inverse9(A, sY[wid], sil[wid], P.Binv + 81 * (int64_t)i) && lane == 0)
            atomicExch(&st->blockfail, 1);
    }
}

// Bound by the FP64 pipe (35 instructions per point; the clamps and the test of
// the determinant are integer work): 85 -> 66 us for 1.0M points.  Runs after
// damp_cameras_kernel, which leaves mu in the state.
template <typename T>
__global__ void damp_points_kernel(Prob P, int damping) {
    DevState *st = P.st;
    if (st->done) return;
    const double mu = st->mu;
    T *Ci = (T *)P.Cinv;
    const bool sorted = P.sorted != 0;  // [6][np_pad] in sorted point order, else [np][6]
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < P.np; s += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = sorted ? __ldg(P.sp_pt + s) : s;
        const int64_t base = sorted ? s : 6 * j, step = sorted ? P.np_pad : 1;
        const double *h = P.Hll + 6 * j;
        const double a00 = h[0] + mu * damp_term(damping, h[0]), a01 = h[1], a02 = h[2];
        const double a11 = h[3] + mu * damp_term(damping, h[3]), a12 = h[4];
        const double a22 = h[5] + mu * damp_term(damping, h[5]);
        const double c00 = a11 * a22 - a12 * a12, c01 = a02 * a12 - a01 * a22, c02 = a01 * a12 - a02 * a11;
        const double det = a00 * c00 + a01 * c01 + a02 * c02;
        const long long db = __double_as_longlong(det);
        if (db <= 0 || db >= 0x7ff0000000000000LL) {  // not positive, infinite or NaN
            atomicExch(&st->blockfail, 1);
            continue;
        }
        const double id = sorted ? fast_rcp(det) : 1.0 / det;
        Ci[base] = (T)(c00 * id);
        Ci[base + step] = (T)(c01 * id);
        Ci[base + 2 * step] = (T)(c02 * id);
        Ci[base + 3 * step] = (T)((a00 * a22 - a02 * a02) * id);
        Ci[base + 4 * step] = (T)((a02 * a01 - a00 * a12) * id);
        Ci[base + 5 * step] = (T)((a00 * a11 - a01 * a01) * id);
    }
}

// ---------------------------------------------------------------------------
// Schur-Jacobi preconditioner (solver variant): S~_ii = B~_i - sum_k
// Jc~_k^T G_k Jc~_k over the observations k of camera i, G_k = Jp~_k C~_j^-1
// Jp~_k^T (2x2).  Camera-major chunks recompute the Jacobian (as the
// linearisation's camera pass does) and write 45 packed chunk sums; each
// camera then subtracts its chunk sums from B~_i in chunk order and, if the
// result is positive definite, replaces the preconditioner block by its
// inverse (Cholesky, FP64).  Otherwise B~_i^-1 stays.
// ---------------------------------------------------------------------------
// One warp per chunk (256 observations): the 45 sums over the lanes by halving
// exchanges, 63 shuffles a chunk where a tree per sum took 225 a warp: with a
// warp per 32 observations the sums cost twice the products.  123 -> about 27 us
// for 0.98M observations of 601 cameras.
template <typename T, bool AD>
__global__ void __launch_bounds__(kBlock) sj_camera_kernel(Prob P) {
    if (P.st->done) return;
    __shared__ T sct[kWarps][kCamTab];
    const T *__restrict__ camtab = (const T *)P.camtab;
    const T *__restrict__ Ci = (const T *)P.Cinv;
    const T delta = (T)P.delta;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T *ctab = sct[wid];
    for (int c = blockIdx.x * kWarps + wid; c < P.n_cchunks; c += gridDim.x * kWarps) {
        const int cam = P.cchunk_cam[c];
        const int b0 = P.cchunk_beg[c], b1 = P.cchunk_beg[c + 1];
        __syncwarp();
        if (lane < kCamTab) ctab[lane] = camtab[(int64_t)cam * kCamTab + lane];
        __syncwarp();
        T acc[64];
#pragma unroll
        for (int q = 0; q < 64; ++q) acc[q] = T(0);
        int ptn = 0, spn = 0;  // the next observation's point, and its place in the sorted order
        if (b0 + lane < b1) {
            ptn = __ldg(P.cm_pt + b0 + lane);
            if (P.sorted) spn = __ldg(P.cm_sp + b0 + lane);
        }
        for (int s = b0 + lane; s < b1; s += 32) {
            constexpr bool FACT = sizeof(T) == 4 && !AD;
            T X0, X1, X2, u0, u1, c6[6];
            const int pt = ptn;
            const int64_t sp = spn;
            if (s + 32 < b1) {
                ptn = __ldg(P.cm_pt + s + 32);
                if (P.sorted) spn = __ldg(P.cm_sp + s + 32);
            }
            if constexpr (FACT) {
                const float4 X = P.sp_X[sp];
                X0 = X.x, X1 = X.y, X2 = X.z;
            } else {
                load_point<T>(P, pt, X0, X1, X2);
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) c6[q] = P.sorted ? Ci[q * P.np_pad + sp] : Ci[6 * (int64_t)pt + q];
            load_uv<T>(P.cm_uv, P.cm_uv32, s, u0, u1);
            T e[2], Jc[18], Jp[6];
            edge_eval<T, AD>(ctab, X0, X1, X2, u0, u1, e, Jc, Jp);
            zero_fixed_columns<T>(P, cam, pt, Jc, Jp);
            T rho, W;
            loss_weight<T>(P.loss, delta, e[0] * e[0] + e[1] * e[1], &rho, &W);
            T q0[3], q1[3];
            // Q = Jp C~^-1 (rows), G = W^2 Q Jp^T
            q0[0] = c6[0] * Jp[0] + c6[1] * Jp[1] + c6[2] * Jp[2];
            q0[1] = c6[1] * Jp[0] + c6[3] * Jp[1] + c6[4] * Jp[2];
            q0[2] = c6[2] * Jp[0] + c6[4] * Jp[1] + c6[5] * Jp[2];
            q1[0] = c6[0] * Jp[3] + c6[1] * Jp[4] + c6[2] * Jp[5];
            q1[1] = c6[1] * Jp[3] + c6[3] * Jp[4] + c6[4] * Jp[5];
            q1[2] = c6[2] * Jp[3] + c6[4] * Jp[4] + c6[5] * Jp[5];
            const T w2 = W * W;
            const T g00 = w2 * (q0[0] * Jp[0] + q0[1] * Jp[1] + q0[2] * Jp[2]);
            const T g01 = w2 * (q0[0] * Jp[3] + q0[1] * Jp[4] + q0[2] * Jp[5]);
            const T g11 = w2 * (q1[0] * Jp[3] + q1[1] * Jp[4] + q1[2] * Jp[5]);
            T F0[9], F1[9];
#pragma unroll
            for (int b = 0; b < 9; ++b) {
                F0[b] = g00 * Jc[b] + g01 * Jc[9 + b];
                F1[b] = g01 * Jc[b] + g11 * Jc[9 + b];
            }
            int idx = 0;
#pragma unroll
            for (int a = 0; a < 9; ++a)
#pragma unroll
                for (int b = a; b < 9; ++b) acc[idx++] += Jc[a] * F0[b] + Jc[9 + a] * F1[b];
        }
        __syncwarp();
        // two exchanges in T, the others in FP64
#pragma unroll
        for (int w = 32; w >= 16; w >>= 1) {
            const bool up = lane & (w >> 1);
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const T send = up ? acc[q] : acc[q + w], keep = up ? acc[q + w] : acc[q];
                acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, w >> 1);
            }
        }
        double sum[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) sum[q] = (double)acc[q];
#pragma unroll
        for (int w = 8; w >= 2; w >>= 1) {
            const bool up = lane & (w >> 1);
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const double send = up ? sum[q] : sum[q + w], keep = up ? sum[q + w] : sum[q];
                sum[q] = keep + __shfl_xor_sync(0xffffffffu, send, w >> 1);
            }
        }
        const int idx = 2 * lane;  // bit 4 of the lane chose 32, ..., bit 0 chose 2
        double *out = P.cpart + 54 * (int64_t)c;
        if (idx < 45) out[idx] = sum[0];
        if (idx + 1 < 45) out[idx + 1] = sum[1];
    }
}

__global__ void __launch_bounds__(32 * kDampWarps) sj_finalize_kernel(Prob P, const int32_t *__restrict__ cfirst) {
    __shared__ double sA[kDampWarps][81], sY[kDampWarps][81], sil[kDampWarps][9];
    if (P.st->done) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = blockIdx.x * kDampWarps + wid; i < P.nc; i += gridDim.x * kDampWarps) {
        double *A = sA[wid];
        __syncwarp();
        for (int e = lane; e < 81; e += 32) {
            const int a = e / 9, b = e - 9 * (e / 9);
            double sum = 0.0;
            for (int c = cfirst[i]; c < cfirst[i + 1]; ++c) sum += P.cpart[54 * (int64_t)c + sym9(a, b)];
            A[e] = P.Bd[81 * (int64_t)i + e] - sum;
        }
        __syncwarp();
        warp_spd_inverse9(A, sY[wid], sil[wid], P.Binv + 81 * (int64_t)i);  // not PD: B~_i^-1 stays
    }
}

// ---------------------------------------------------------------------------
// shared pieces of the point-major passes
// ---------------------------------------------------------------------------

// Streaming variant: evict-first loads, so the once-per-pass Jacobian stream
// does not push the per-observation s vectors and camera data out of L2.
template <typename T>
__device__ __forceinline__ void load_jac_stream(const T *__restrict__ J, int64_t npad, int64_t o, T *Jc, T *Jp) {
#pragma unroll
    for (int q = 0; q < 18; ++q) Jc[q] = __ldcs(J + q * npad + o);
#pragma unroll
    for (int q = 0; q < 6; ++q) Jp[q] = __ldcs(J + (18 + q) * npad + o);
}

template <typename T>
__device__ __forceinline__ void sym3_apply(const T *__restrict__ C, T a0, T a1, T a2, T *b) {
    const T c0 = __ldg(C), c1 = __ldg(C + 1), c2 = __ldg(C + 2), c3 = __ldg(C + 3), c4 = __ldg(C + 4),
            c5 = __ldg(C + 5);
    b[0] = c0 * a0 + c1 * a1 + c2 * a2;
    b[1] = c1 * a0 + c3 * a1 + c4 * a2;
    b[2] = c2 * a0 + c4 * a1 + c5 * a2;
}

// ---------------------------------------------------------------------------
// The implicit Schur product S p = B~ p - E C~^-1 E^T p in two passes per PCG
// iteration, neither of which writes to a shared accumulator:
//  * point pass (point-major, warp chunks of whole points, <= 32
//    observations): b_j = C~_j^-1 sum_k Jp~_k^T Jc~_k p_i(k) by a segmented
//    shuffle scan, then s_k = Jp~_k b_j is stored per observation;
//  * camera pass (camera-major, one warp per camera chunk of <= 1024
//    observations): the chunk's sum of Jc~_k^T s_k; the last warp to finish a
//    camera adds that camera's chunk sums in a fixed order and forms
//    q_i = B~_i p_i - c_i (or the right-hand side g_i = v_i - c_i).
// In FP32-mixed the camera pass recomputes Jc~ from the camera table and the
// point (camera-uniform per warp, cheaper than streaming 72 bytes again); the
// FP64 form streams a camera-major copy written at linearisation.
// ---------------------------------------------------------------------------
template <typename T>
struct V2;
template <>
struct V2<float> {
    using type = float2;
};
template <>
struct V2<double> {
    using type = double2;
};

template <typename T>
__device__ __forceinline__ void gather_p(const T *ps, const T *pT, int cam, T *pa) {
    if (ps) {
#pragma unroll
        for (int a = 0; a < 9; ++a) pa[a] = ps[cam * 9 + a];
    } else {
        const T *pv = pT + (int64_t)cam * kVec;
#pragma unroll
        for (int a = 0; a < 9; ++a) pa[a] = ldcg(pv + a);
    }
}

// E^T p contribution of one observation: u = Jp^T (Jc p)
template <typename T>
__device__ __forceinline__ void et_p(const T *Jc, const T *Jp, const T *pa, T *u) {
    T t0 = T(0), t1 = T(0);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        t0 += Jc[a] * pa[a];
        t1 += Jc[9 + a] * pa[a];
    }
    u[0] = Jp[0] * t0 + Jp[3] * t1;
    u[1] = Jp[1] * t0 + Jp[4] * t1;
    u[2] = Jp[2] * t0 + Jp[5] * t1;
}

template <typename T>
__device__ __forceinline__ void load_sym3(const T *__restrict__ C, T *c) {
#pragma unroll
    for (int q = 0; q < 6; ++q) c[q] = __ldg(C + q);
}
template <typename T>
__device__ __forceinline__ void apply_sym3(const T *c, T a0, T a1, T a2, T *b) {
    b[0] = c[0] * a0 + c[1] * a1 + c[2] * a2;
    b[1] = c[1] * a0 + c[3] * a1 + c[4] * a2;
    b[2] = c[2] * a0 + c[4] * a1 + c[5] * a2;
}

template <typename T>
__device__ __forceinline__ void store_s(typename V2<T>::type *sbuf, int64_t o, const T *Jp, const T *b) {
    typename V2<T>::type v;
    v.x = Jp[0] * b[0] + Jp[1] * b[1] + Jp[2] * b[2];
    v.y = Jp[3] * b[0] + Jp[4] * b[1] + Jp[5] * b[2];
    sbuf[o] = v;
}

// Point pass.  RHS: b_j = C~_j^-1 w_j.  Otherwise b_j = C~_j^-1 sum_k u_k.
template <typename T, bool RHS>
__device__ void point_pass(const Prob &P, const T *ps, const T *pT, typename V2<T>::type *sbuf) {
    const T *__restrict__ J = (const T *)P.J;
    const T *__restrict__ Cinv = (const T *)P.Cinv;
    const int64_t npad = P.npad;
    const int lane = threadIdx.x & 31;
    const int nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    const int gstride = gridDim.x * nwarp;
    int w = blockIdx.x * nwarp + (threadIdx.x >> 5);
    int2 c0 = make_int2(0, 0), c1 = make_int2(0, 0);
    if (w < P.n_wchunks) {
        c0 = P.wchunk[w];
        c1 = P.wchunk[w + 1];
    }
    for (; w < P.n_wchunks; w += gstride) {
        const int wn = w + gstride;
        int2 n0 = c0, n1 = c1;
        if (wn < P.n_wchunks) {
            n0 = P.wchunk[wn];
            n1 = P.wchunk[wn + 1];
        }
        const int o0 = c0.y, m = c1.y - c0.y;
        if (m <= 32) {
            const bool act = lane < m;
            const int64_t o = (int64_t)o0 + (act ? lane : 0);
            // point of each lane from the chunk's point starts (whole points, <= 32 observations)
            const int npts = c1.x - c0.x;
            const int rs = lane < npts ? __ldg(P.pt_ptr + c0.x + lane) - o0 : 32;
            const unsigned starts = __reduce_or_sync(full, rs < 32 ? (1u << rs) : 0u);
            const int pt = act ? c0.x + __popc(starts & (0xffffffffu >> (31 - lane))) - 1 : -1 - lane;
            const int cam = act ? __ldcs(P.pm_cam + o) : 0;
            const int so = act ? __ldcs(P.pm2cm + o) : 0;  // where the camera pass reads s
            T Jc[18], Jp[6], ci[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) Jp[q] = ci[q] = T(0);
#pragma unroll
            for (int q = 0; q < 18; ++q) Jc[q] = T(0);
            if (act) {
#pragma unroll
                for (int q = 0; q < 6; ++q) Jp[q] = __ldcs(J + (18 + q) * npad + o);
                if (!RHS)
#pragma unroll
                    for (int q = 0; q < 18; ++q) Jc[q] = __ldcs(J + q * npad + o);
                load_sym3(Cinv + 6 * (int64_t)pt, ci);
            }
            T b[3] = {T(0), T(0), T(0)};
            if (RHS) {
                if (act)
                    apply_sym3(ci, (T)P.w[3 * (int64_t)pt], (T)P.w[3 * (int64_t)pt + 1], (T)P.w[3 * (int64_t)pt + 2],
                               b);
            } else {
                T u[3] = {T(0), T(0), T(0)};
                if (act) {
                    T pa[9];
                    gather_p(ps, pT, cam, pa);
                    et_p(Jc, Jp, pa, u);
                }
                // inclusive segmented scan keyed by point (segments are contiguous).
                // FP64: only as many levels as the chunk's longest point needs
                // (each level is three warp-wide FP64 adds on the FP64 pipe)
                int span = 32;
                if constexpr (sizeof(T) == 8) {
                    const int nrs = __shfl_down_sync(full, rs, 1);
                    const int len = lane < npts ? (lane + 1 < npts ? nrs : m) - rs : 0;
                    span = __reduce_max_sync(full, len);
                }
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    if (d >= span) break;
                    const int kp = __shfl_up_sync(full, pt, d);
                    const T v0 = __shfl_up_sync(full, u[0], d), v1 = __shfl_up_sync(full, u[1], d),
                            v2 = __shfl_up_sync(full, u[2], d);
                    if (lane >= d && kp == pt) {
                        u[0] += v0;
                        u[1] += v1;
                        u[2] += v2;
                    }
                }
                const int nxt = __shfl_down_sync(full, pt, 1);
                const bool tail = act && (lane == 31 || lane == m - 1 || nxt != pt);
                const unsigned tails = __ballot_sync(full, tail);
                T bt[3];
                apply_sym3(ci, u[0], u[1], u[2], bt);
                const unsigned mine = tails & (0xffffffffu << lane);
                const int src = mine ? __ffs(mine) - 1 : lane;
                b[0] = __shfl_sync(full, bt[0], src);
                b[1] = __shfl_sync(full, bt[1], src);
                b[2] = __shfl_sync(full, bt[2], src);
            }
            if (act) store_s<T>(sbuf, so, Jp, b);
        } else {
            // one point with a long track: two sweeps over 32-observation slices
            const int pt = c0.x;
            T ci[6], b[3];
            load_sym3(Cinv + 6 * (int64_t)pt, ci);
            if (RHS) {
                apply_sym3(ci, (T)P.w[3 * (int64_t)pt], (T)P.w[3 * (int64_t)pt + 1], (T)P.w[3 * (int64_t)pt + 2], b);
            } else {
                T a[3] = {T(0), T(0), T(0)};
                for (int base = 0; base < m; base += 32) {
                    if (base + lane < m) {
                        const int64_t o = (int64_t)o0 + base + lane;
                        T Jc[18], Jp[6], pa[9], u[3];
                        load_jac_stream(J, npad, o, Jc, Jp);
                        gather_p(ps, pT, __ldcs(P.pm_cam + o), pa);
                        et_p(Jc, Jp, pa, u);
                        a[0] += u[0];
                        a[1] += u[1];
                        a[2] += u[2];
                    }
                }
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) {
                    a[0] += __shfl_xor_sync(full, a[0], d);
                    a[1] += __shfl_xor_sync(full, a[1], d);
                    a[2] += __shfl_xor_sync(full, a[2], d);
                }
                apply_sym3(ci, a[0], a[1], a[2], b);
            }
            for (int base = 0; base < m; base += 32) {
                if (base + lane < m) {
                    const int64_t o = (int64_t)o0 + base + lane;
                    T Jp[6];
#pragma unroll
                    for (int q = 0; q < 6; ++q) Jp[q] = __ldcs(J + (18 + q) * npad + o);
                    store_s<T>(sbuf, __ldcs(P.pm2cm + o), Jp, b);
                }
            }
        }
        c0 = n0;
        c1 = n1;
    }
}


// ---------------------------------------------------------------------------
// Factored FP32 form (analytic Jacobian).  With P = R X + t the camera-frame
// point, p = -(P_x, P_y) / P_z, r2 = |p|^2, d = 1 + k1 r2 + k2 r2^2 and
// A = f (d I + (2 k1 + 4 k2 r2) p p^T), the BAL Jacobian of one observation is
//   D = d(pixel)/dP = -(1/P_z) A [I | p],   Jp = D R,   Jc = [-D R [X]x M | D | p (d, f r2, f r2^2)]
// (M: the rotation factor of the camera table).  Because R (a x b) = R a x R b,
// the two products the PCG needs reduce to per-observation data and
// per-camera constants:
//   Jc v = D (n x (P - t) + v_t) + p (v_f + r2 (v_a + r2 v_b)),
//          n = R M v_w,  v_a = k1 v_f + f v_k1,  v_b = k2 v_f + f v_k2;
//   sum_k Jc_k^T s_k = [ (R M)^T sum_k RX_k x y_k ; sum_k y_k ;
//                        (S0 + k1 S1 + k2 S2, f S1, f S2) ],
//          y_k = D_k^T s_k,  S_m = sum_k r2^m p.s,  RX = R X = P - t.
// The two triples of camera transforms are transposes of each other (P.ctr).
//
// Point pass (sliced order, sell.cu): per observation the camera index and
// (px, py, 1/P_z), 16 bytes, and the camera's row from shared memory;
// u = Jp^T t = R^T D^T t, R from its quaternion (two cross products), so that a
// row is 16 floats, four 16-byte shared loads, which bound the pass.  It forms
// (n x (P - t) + v_t) / P_z = n x (-px, -py, 1) + h / P_z with the camera
// constant h = v_t - n x t: one cancellation of order |t| / |RX| per
// observation.
// Camera pass: per observation (RX, 1/P_z), the point index and one 16-byte
// gather of b_j; the camera is uniform in the warp, so s = Jp b and Jc^T s are
// formed in registers.  Gathering (X, b) as one 32-byte record and recomputing
// the projection took 35.1 against 33.4 us on the Venice-shaped problem and 264
// against 225 on the Final-shaped one: the pass is bound by the gathers, which an
// SM issues at about one per two cycles.  The cross products,
// summed over hundreds of observations, use RX itself: forming them from P and t
// instead would cancel after the sum, and that loss broke the PCG near mu ~ 1e-7.
// Against the form that streamed (px, py, 1/P_z) and W Jp point-major, scattered
// s = Jp b into camera-major order and streamed it back with (RX, 1/P_z), 76
// bytes per observation and a segmented shuffle scan per chunk: 1,305 -> 514 us
// per product of 29M observations of 13,000 cameras (used where the camera rows do
// not fit in shared memory; pcg_own.cuh has the figures where they do).
// (In the first-order rotation branch, |w|^2 <= 2.2e-16, both apply
// R = I + [w]x where the Jacobian has I: a relative difference of at most |w|,
// below FP32 rounding.)
//
// Camera row of a vector v: n (3), h (3), v_f, v_a, v_b; in shared memory and in
// the global copy followed by f, k1, k2 and the quaternion (P.camstat).  The
// first nine are linear in v, so row(z) + beta row(p) is the row of z + beta p.
// ---------------------------------------------------------------------------

// A fixed camera's Jacobian columns are zero, so its rows are, whatever the
// vector holds there: zero in a solve, but the upstream gradient's part in an adjoint.
__device__ __forceinline__ bool fixed_camera(const Prob &P, int cam) { return P.has_fixed && P.cam_fixed[cam]; }

// Warp-collective (all 32 lanes call it): lanes 9s..9s+8 hold the nine
// components of camera `cam` (lane s of the three-camera group); returns the
// lane's component of the camera's row.
__device__ __forceinline__ float fact_row_lane(const Prob &P, int cam, double val, int sub, int row) {
    const unsigned full = 0xffffffffu;
    const float v = (float)val;
    const int g0 = row < 3 ? 0 : (row < 6 ? 3 : 6), b = row - g0, at = 9 * sub + g0;
    const float *ct = P.ctr + (int64_t)cam * kCtr + 3 * g0 + b;
    float r = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) r = fmaf(__ldg(ct + 3 * i), __shfl_sync(full, v, (at + i) & 31), r);
    // h = v_t - n x t
    const int b1 = b == 2 ? 0 : b + 1, b2 = b == 0 ? 2 : b - 1;
    const float n1 = __shfl_sync(full, r, (9 * sub + b1) & 31), n2 = __shfl_sync(full, r, (9 * sub + b2) & 31);
    if (g0 == 3) {
        const float *t = P.camstat + (int64_t)cam * kCamStat + 7;
        r -= n1 * __ldg(t + b2) - n2 * __ldg(t + b1);
    }
    return fixed_camera(P, cam) ? 0.f : r;
}

// The whole row of one camera by one thread.
__device__ __forceinline__ void fact_row(const Prob &P, int cam, const float *v, float *r) {
    const float *ct = P.ctr + (int64_t)cam * kCtr, *st = P.camstat + (int64_t)cam * kCamStat;
#pragma unroll
    for (int g = 0; g < 3; ++g)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            float x = 0.f;
#pragma unroll
            for (int i = 0; i < 3; ++i) x = fmaf(__ldg(ct + 9 * g + 3 * i + b), v[3 * g + i], x);
            r[3 * g + b] = x;
        }
    const float t0 = st[7], t1 = st[8], t2 = st[9];
    r[3] -= r[1] * t2 - r[2] * t1;
    r[4] -= r[2] * t0 - r[0] * t2;
    r[5] -= r[0] * t1 - r[1] * t0;
    if (fixed_camera(P, cam))
#pragma unroll
        for (int q = 0; q < 9; ++q) r[q] = 0.f;
#pragma unroll
    for (int q = 0; q < 7; ++q) r[9 + q] = st[q];
}

// A point's b: written inside the PCG launch by other CTAs before a grid
// barrier, so an ordinary load, not the read-only path.
__device__ __forceinline__ float4 load_b(const float4 *at) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(at));
    return v;
}
// 32 bytes by one load; ordinary coherent loads, for rows that other CTAs of
// the same launch wrote before a grid barrier.
__device__ __forceinline__ void load8(const float *at, float4 &x, float4 &y) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w), "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w)
                 : "l"(at));
}

struct CamRow {
    float n0, n1, n2, h0, h1, h2, vf, va, vb, f, k1, k2, q0, q1, q2, q3;
};
// ps: shared memory (stride kRowS); otherwise the global rows (stride kRowG),
// written by other CTAs before the last grid barrier, whose acquire orders
// these loads after the writes.
__device__ __forceinline__ CamRow load_row(const float *ps, const float *rows, int cam) {
    float4 a, b, c, d;
    if (ps) {
        const float4 *src = (const float4 *)(ps + cam * kRowS);
        a = src[0], b = src[1], c = src[2], d = src[3];
    } else {
        load8(rows + (int64_t)cam * kRowG, a, b);
        load8(rows + (int64_t)cam * kRowG + 8, c, d);
    }
    return CamRow{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w};
}

// A and the scaled camera-frame vector w of one observation, then t = Jc v.
struct FactObs {
    float a00, a01, a11, w0, w1, w2, ei;
};
__device__ __forceinline__ FactObs fact_obs(float px, float py, float iz, const CamRow &r) {
    FactObs o;
    const float r2 = px * px + py * py;
    const float d = 1.f + r2 * (r.k1 + r.k2 * r2);
    const float fd = r.f * d, fdd = r.f * (2.f * r.k1 + 4.f * r.k2 * r2);
    const float gx = fdd * px;
    o.a00 = fd + gx * px;
    o.a01 = gx * py;
    o.a11 = fd + fdd * py * py;
    // (n x (P - t) + v_t) / P_z = n x (-px, -py, 1) + h / P_z
    o.w0 = r.n1 + r.n2 * py + iz * r.h0;
    o.w1 = -r.n0 - r.n2 * px + iz * r.h1;
    o.w2 = r.n1 * px - r.n0 * py + iz * r.h2;
    o.ei = r.vf + r2 * (r.va + r2 * r.vb);
    return o;
}
__device__ __forceinline__ void fact_t(const FactObs &o, float px, float py, float &t0, float &t1) {
    const float z0 = o.w0 + px * o.w2, z1 = o.w1 + py * o.w2;
    t0 = px * o.ei - (o.a00 * z0 + o.a01 * z1);
    t1 = py * o.ei - (o.a01 * z0 + o.a11 * z1);
}
// u += W Jp^T t = W R^T D^T t
__device__ __forceinline__ void fact_jpt(const FactObs &o, const CamRow &r, float px, float py, float wiz, float t0,
                                         float t1, float *u) {
    const float y0 = -wiz * (o.a00 * t0 + o.a01 * t1), y1 = -wiz * (o.a01 * t0 + o.a11 * t1), y2 = px * y0 + py * y1;
    const float c0 = r.q2 * y2 - r.q3 * y1, c1 = r.q3 * y0 - r.q1 * y2, c2 = r.q1 * y1 - r.q2 * y0;
    u[0] += y0 - r.q0 * c0 + (r.q2 * c2 - r.q3 * c1);
    u[1] += y1 - r.q0 * c1 + (r.q3 * c0 - r.q1 * c2);
    u[2] += y2 - r.q0 * c2 + (r.q1 * c1 - r.q2 * c0);
}

struct FactStream {
    int cam;
    float px, py, iz, W;
};
__device__ __forceinline__ FactStream load_stream(const Prob &P, int64_t slot) {
    const float4 v = __ldg(P.sl_px + slot);
    return FactStream{__float_as_int(v.x), v.y, v.z, v.w, P.sl_w ? __ldg(P.sl_w + slot) : 1.f};
}

// The sum of W Jp^T Jc v over the lane's observations of one slice.
__device__ __forceinline__ void fact_slice_sum(const Prob &P, const float *ps, const float *rows, int64_t slot, int K,
                                               float *a) {
    a[0] = a[1] = a[2] = 0.f;
#pragma unroll 2
    for (int k = 0; k < K; ++k, slot += 32) {
        const FactStream c = load_stream(P, slot);
        if (c.cam < 0) continue;
        const CamRow r = load_row(ps, rows, c.cam);
        const FactObs o = fact_obs(c.px, c.py, c.iz, r);
        float t0, t1;
        fact_t(o, c.px, c.py, t0, t1);
        fact_jpt(o, r, c.px, c.py, c.W * c.iz, t0, t1, a);
    }
}

// Point pass over this warp's slices: b_j = C~_j^-1 sum_k u_k into the record.
// The stream of the next round (of this slice or the next one, whose
// descriptor is read a slice ahead) is in flight while a round is worked.
__device__ void point_pass_fact(const Prob &P, const float *ps, const float *rows) {
    const float *__restrict__ Ci = (const float *)P.Cinv;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int gstride = gridDim.x * (blockDim.x >> 5);
    int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    if (w >= P.n_slices) return;
    int4 sl = __ldg(P.slice + w);
    FactStream cur = load_stream(P, (int64_t)sl.z + lane);
    for (;;) {
        const int wn = w + gstride;
        const int4 nx = wn < P.n_slices ? __ldg(P.slice + wn) : sl;
        const int K = sl.w & 0xffff, lg = sl.w >> 16, in = lane >> lg;
        const int count = sl.y & 0xff;
        const int s = sl.x + (in < count ? in : 0);
        float a[3] = {0.f, 0.f, 0.f};
        for (int k = 1; k <= K; ++k) {
            const FactStream c = cur;
            cur = load_stream(P, (int64_t)(k < K ? sl.z + 32 * k : nx.z) + lane);
            prefetch_l2(P.sl_px + nx.z + 32 * (k < (nx.w & 0xffff) ? k : 0) + lane);
            if (c.cam >= 0) {
                const CamRow r = load_row(ps, rows, c.cam);
                const FactObs o = fact_obs(c.px, c.py, c.iz, r);
                float t0, t1;
                fact_t(o, c.px, c.py, t0, t1);
                fact_jpt(o, r, c.px, c.py, c.W * c.iz, t0, t1, a);
            }
        }
        float ci[6], b[3];
#pragma unroll
        for (int q = 0; q < 6; ++q) ci[q] = __ldg(Ci + (int64_t)q * P.np_pad + s);
        for (int d = 1; d < (1 << lg); d <<= 1) {
#pragma unroll
            for (int q = 0; q < 3; ++q) a[q] += __shfl_xor_sync(full, a[q], d);
        }
        if (in < count && (lane & ((1 << lg) - 1)) == 0) {
            if (P.has_fixed && P.pt_fixed[P.sp_pt[s]]) a[0] = a[1] = a[2] = 0.f;
            apply_sym3(ci, a[0], a[1], a[2], b);
            P.sp_b[s] = make_float4(b[0], b[1], b[2], 0.f);
        }
        if (wn >= P.n_slices) return;
        w = wn;
        sl = nx;
    }
}

// Right-hand side: b_j = C~_j^-1 w_j.
__device__ void point_pass_fact_rhs(const Prob &P) {
    const float *__restrict__ Ci = (const float *)P.Cinv;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < P.np; s += gridDim.x * blockDim.x) {
        const int64_t pt = __ldg(P.sp_pt + s);
        float ci[6], b[3];
#pragma unroll
        for (int q = 0; q < 6; ++q) ci[q] = __ldg(Ci + (int64_t)q * P.np_pad + s);
        apply_sym3(ci, (float)P.w[3 * pt], (float)P.w[3 * pt + 1], (float)P.w[3 * pt + 2], b);
        if (P.has_fixed && P.pt_fixed[pt]) b[0] = b[1] = b[2] = 0.f;  // its Jacobian columns are zero
        P.sp_b[s] = make_float4(b[0], b[1], b[2], 0.f);
    }
}

template <typename T, bool RHS, bool FACT>
__device__ __forceinline__ void point_pass_any(const Prob &P, const T *ps, const T *pT, typename V2<T>::type *sbuf) {
    if constexpr (FACT && RHS) point_pass_fact_rhs(P);
    else if constexpr (FACT) point_pass_fact(P, (const float *)ps, (const float *)pT);
    else point_pass<T, RHS>(P, ps, pT, sbuf);
}

// Stored form (FP64, and FP32-mixed with dual-number Jacobians): acc += Jc~^T s
// as 18 fused multiply-adds on the stored camera-major Jc~ (sqrt(W) included).
template <typename T>
__device__ __forceinline__ void camera_acc_stored(const Prob &P, int64_t s, T s0, T s1, T *acc) {
    const T *__restrict__ Jc = (const T *)P.JcmT;
#pragma unroll
    for (int a = 0; a < 9; ++a)
        acc[a] = fma(__ldcs(Jc + a * P.npad + s), s0, fma(__ldcs(Jc + (9 + a) * P.npad + s), s1, acc[a]));
}

enum CamMode { CAM_RHS = 0, CAM_ITER = 1, CAM_MATVEC = 2, CAM_SR = 3 };

__device__ __forceinline__ double2 cta_sum2(double x, double y, bool warp_data, double *sb);
__device__ __forceinline__ double3 cta_sum3(double x, double y, double z, bool warp_data, double *sb);


// Sums of 9 values over the warp's lanes by exchanging halves: 14 shuffles
// where nine butterflies take 45.  Lane l with l mod 4 == 0 returns the sum of
// value 4 bit4(l) + 2 bit3(l) + bit2(l); `last` is the sum of v[8] in every lane.
__device__ __forceinline__ float reduce9(float *v, float &last) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    float w = v[8];
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
        const bool up = lane & (h << 2);
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(full, send, h << 2);
        }
        w += __shfl_xor_sync(full, w, h << 2);
    }
    float r = v[0];
    r += __shfl_xor_sync(full, r, 2);
    w += __shfl_xor_sync(full, w, 2);
    r += __shfl_xor_sync(full, r, 1);
    w += __shfl_xor_sync(full, w, 1);
    last = w;
    return r;
}

// gathers of b in flight per lane (Venice-shaped camera pass: 33.4 us with one,
// 34.8 with two, 41.5 with three, which spill)
constexpr int kCamDepth = 1;
// One observation of the factored camera pass: the raw sums RX x y (0..2), y
// (3..5), p.s (1, r2, r2^2) (6..8); X = (R X, 1 / P_z).  R b is formed from the
// same quaternion as the point pass's R^T y: with a rounded matrix here the two
// passes would apply rotations that differ by a fixed rounding per camera, an
// asymmetry of the product that PCG sees in every iteration.
struct CamConst {
    float q0, q1, q2, q3, t0, t1, f, k1, k2;
};
__device__ __forceinline__ void fact_camera_obs(const CamConst &ct, const float4 X, const float4 b, float W, float *acc) {
    const float e0 = ct.q2 * b.z - ct.q3 * b.y, e1 = ct.q3 * b.x - ct.q1 * b.z, e2 = ct.q1 * b.y - ct.q2 * b.x;
    const float b0 = b.x + ct.q0 * e0 + (ct.q2 * e2 - ct.q3 * e1), b1 = b.y + ct.q0 * e1 + (ct.q3 * e0 - ct.q1 * e2),
                b2 = b.z + ct.q0 * e2 + (ct.q1 * e1 - ct.q2 * e0);
    const float iz = X.w;
    const float x = -(X.x + ct.t0) * iz, y = -(X.y + ct.t1) * iz;
    const float r2 = x * x + y * y, f = ct.f, k1 = ct.k1, k2 = ct.k2;
    const float d = 1.f + r2 * (k1 + k2 * r2);
    const float fd = f * d, fdd = f * (2.f * k1 + 4.f * k2 * r2), gx = fdd * x;
    const float a00 = fd + gx * x, a01 = gx * y, a11 = fd + fdd * y * y;
    // s = W Jp b = -(W / P_z) A (Rb_xy + p Rb_z)
    const float c0 = b0 + x * b2, c1 = b1 + y * b2, wz = -W * iz;
    const float s0 = wz * (a00 * c0 + a01 * c1), s1 = wz * (a01 * c0 + a11 * c1);
    const float y0 = -iz * (a00 * s0 + a01 * s1), y1 = -iz * (a01 * s0 + a11 * s1), y2 = x * y0 + y * y1;
    acc[0] += X.y * y2 - X.z * y1;
    acc[1] += X.z * y0 - X.x * y2;
    acc[2] += X.x * y1 - X.y * y0;
    acc[3] += y0;
    acc[4] += y1;
    acc[5] += y2;
    const float ps = x * s0 + y * s1, qs = r2 * ps;
    acc[6] += ps;
    acc[7] += qs;
    acc[8] += r2 * qs;
}

// Camera pass.  Each CTA owns a contiguous run of whole cameras
// [cta_cam[b], cta_cam[b+1]), balanced by observation count at creation; its
// warps reduce parts of the cameras (the stored form: camera chunks) into
// shared-memory slots, then, after a block barrier, each camera's slots are
// added in observation order and the camera is finalised.  No global atomics or fences; results do not depend on
// timing.  CAM_RHS: g = v - c, x = 0, r = g, z = B~^-1 g; returns this CTA's
// (r.r, r.z).  CAM_ITER: p = z + beta p_prev (p = z first), q = B~ p - c;
// returns (p.q, 0).  CAM_MATVEC: q = B~ p - c with p given.  CAM_SR (the
// single-reduction PCG): w = B~ u - c with u in P.z, into P.q; returns (r.r,
// r.u) and w.u in *third.
template <typename T, int MODE, bool JS>
__device__ double2 camera_pass(const Prob &P, const typename V2<T>::type *sbuf, const double *p_prev, double *p_cur,
                               double beta, bool first, double *cslot, double *sb, double *third = nullptr) {
    using T2 = typename V2<T>::type;
    constexpr int U = 4;
    constexpr bool FACT = sizeof(T) == 4 && !JS;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    const int cb = P.cta_cam[blockIdx.x], ce = P.cta_cam[blockIdx.x + 1];
    int k0 = 0, per = 32, o0 = 0;
    if constexpr (FACT) {
        // each warp takes an equal run of the CTA's observations (a multiple of 32)
        // and flushes its sums at every camera boundary; warp w's part of camera i
        // has the slot w + i - cb, which increases along the run, so a camera's
        // parts are consecutive slots in observation order
        o0 = __ldg(P.cam_ptr + cb);
        const int total = __ldg(P.cam_ptr + ce) - o0;
        per = ((total + nwarp - 1) / nwarp + 31) & ~31;
        if (per < 32) per = 32;
        int s0 = o0 + wid * per;
        const int s1 = min(o0 + total, s0 + per);
        int cam = cb;
        if (s0 < s1) {  // the camera of the first observation: last i in [cb, ce) with cam_ptr[i] <= s0
            int hi = ce - 1;
            while (cam < hi) {
                const int mid = (cam + hi + 1) >> 1;
                if (__ldg(P.cam_ptr + mid) <= s0) cam = mid;
                else hi = mid - 1;
            }
        }
        for (; s0 < s1; ++cam) {
            const int e = min(s1, __ldg(P.cam_ptr + cam + 1));
            CamConst ct;
            {
                const float *st = P.camstat + (int64_t)cam * kCamStat;
                ct.f = __ldg(st), ct.k1 = __ldg(st + 1), ct.k2 = __ldg(st + 2);
                ct.q0 = __ldg(st + 3), ct.q1 = __ldg(st + 4), ct.q2 = __ldg(st + 5), ct.q3 = __ldg(st + 6);
                ct.t0 = __ldg(st + 7), ct.t1 = __ldg(st + 8);
            }
            float acc[9];
#pragma unroll
            for (int a = 0; a < 9; ++a) acc[a] = 0.f;
            // kCamDepth observations' (R X, 1/P_z), b and the point index after them
            // are in flight while one is worked; each is copied out of its
            // registers before the next load into them is issued, so that no copy
            // waits for a load in flight
            constexpr int D = kCamDepth;
            float4 X[D], v[D];
            int id[D];
            const int q0 = s0 + lane;
#pragma unroll
            for (int j = 0; j < D; ++j) {
                X[j] = v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (q0 + 32 * j < e) {
                    X[j] = __ldg(P.RXcm + q0 + 32 * j);
                    v[j] = load_b(P.sp_b + __ldg(P.cm_sp + q0 + 32 * j));
                }
                id[j] = q0 + 32 * (j + D) < e ? __ldg(P.cm_sp + q0 + 32 * (j + D)) : 0;
            }
            for (int p = q0; p < e; p += 32 * D) {
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    const int o = p + 32 * j, on = o + 32 * D;
                    const float4 Xc = X[j], vc = v[j];
                    if (on < e) {
                        X[j] = __ldg(P.RXcm + on);
                        v[j] = load_b(P.sp_b + id[j]);
                        if (on + 32 * D < e) id[j] = __ldg(P.cm_sp + on + 32 * D);
                    }
                    if (o < e) fact_camera_obs(ct, Xc, vc, P.cm_w ? __ldg(P.cm_w + o) : 1.f, acc);
                }
            }
            __syncwarp();
            float last;
            const float mine = reduce9(acc, last);
            const int q = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
            double *slot = cslot + 9 * (wid + cam - cb);
            if ((lane & 3) == 0) slot[q] = (double)mine;
            if (lane == 1) slot[8] = (double)last;
            s0 = e;
        }
    } else {
        __shared__ int next_chunk;
        k0 = P.cfirst[cb];
        const int k1 = P.cfirst[ce];
        if (threadIdx.x == 0) next_chunk = k0 + nwarp;
        __syncthreads();
        // warps claim chunks dynamically; each chunk's sum goes to its own slot, so
        // the result does not depend on which warp took it
        for (int k = k0 + wid; k < k1;) {
            const int b0 = P.cchunk_beg[k], b1 = P.cchunk_beg[k + 1];
            T acc[9];
#pragma unroll
            for (int a = 0; a < 9; ++a) acc[a] = T(0);
            for (int s0 = b0; s0 < b1; s0 += 32 * U) {
                // s arrives in camera-major order (the point pass scattered it), so
                // every load of the batch is a coalesced stream
                bool in[U];
                T2 sv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int s = s0 + u * 32 + lane;
                    in[u] = s < b1;
                    if (in[u]) sv[u] = ldcg(sbuf + s);
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (in[u]) camera_acc_stored<T>(P, s0 + u * 32 + lane, (T)sv[u].x, (T)sv[u].y, acc);
            }
            T mine = T(0);
#pragma unroll
            for (int a = 0; a < 9; ++a) {
                T v = acc[a];
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(full, v, d);
                if (lane == a) mine = v;
            }
            if (lane < 9) cslot[(k - k0) * 9 + lane] = (double)mine;  // one conversion per lane
            int nk = 0;
            if (lane == 0) nk = atomicAdd(&next_chunk, 1);
            k = __shfl_sync(full, nk, 0);
        }
    }
    __syncthreads();
    // finalise this CTA's cameras, three per warp (lanes 9s..9s+8 hold rows of
    // camera s): chunk sums added in chunk order
    double d1 = 0.0, d2 = 0.0, d3 = 0.0;
    const int sub = lane / 9, row = lane - 9 * sub;
    for (int c0 = cb + 3 * wid; c0 < ce; c0 += 3 * nwarp) {
        const int cam = c0 + sub;
        const bool act = lane < 27 && cam < ce;
        const int a = act ? row : 0;
        const int cm = act ? cam : c0;
        const int64_t vo = (int64_t)cm * kVec + a;
        // this lane's row of B~^-1 (right-hand side) or B~ (products): in the
        // factored form's standard iterations loaded before the chunk sums, so
        // that its latency overlaps them (109.9 -> 109.3 us per PCG iteration);
        // elsewhere loaded where it is used (the early load raised the
        // single-reduction instance's spills and slowed it, and the FP64 one)
        constexpr bool kEarly = FACT && MODE == CAM_ITER;
        const double *Mrow = (MODE == CAM_RHS ? P.Binv : P.Bd) + 81 * (int64_t)cm + a * 9;
        double brow[9];
#pragma unroll
        for (int b = 0; b < 9; ++b) brow[b] = (kEarly && act) ? __ldg(Mrow + b) : 0.0;
        double cs = 0.0;
        if (act) {
            if constexpr (FACT) {
                const int w0 = (__ldg(P.cam_ptr + cm) - o0) / per, w1 = (__ldg(P.cam_ptr + cm + 1) - 1 - o0) / per;
                for (int k = w0 + cm - cb; k <= w1 + cm - cb; ++k) cs += cslot[k * 9 + a];
            } else {
                for (int k = P.cfirst[cm]; k < P.cfirst[cm + 1]; ++k) cs += cslot[(k - k0) * 9 + a];
            }
        }
        if constexpr (FACT) {  // c = ctr raw, three terms of the lane's group
            const int g0 = a < 3 ? 0 : (a < 6 ? 3 : 6);
            const float *ct = P.ctr + (int64_t)cm * kCtr + 3 * a;
            double c = 0.0;
#pragma unroll
            for (int b = 0; b < 3; ++b)
                c = fma((double)__ldg(ct + b), __shfl_sync(full, cs, (9 * sub + g0 + b) & 31), c);
            cs = c;
        }
        // a fixed camera has no Schur coupling (its Jacobian columns are zero; the
        // factored product forms Jc^T s from the geometry, so it is masked here)
        if (P.has_fixed && act && P.cam_fixed[cm]) cs = 0.0;
        double v1 = 0.0, v2 = 0.0, v3 = 0.0;
        if (MODE == CAM_RHS) {
            const double g = act ? P.v[9 * (int64_t)cm + a] - cs : 0.0;
            double z = 0.0;
#pragma unroll
            for (int b = 0; b < 9; ++b) {
                const double gb = __shfl_sync(full, g, 9 * sub + b);
                if (act) z = fma(kEarly ? brow[b] : __ldg(Mrow + b), gb, z);
            }
            if (act) {
                stcg(P.g + vo, g);
                stcg(P.x + vo, 0.0);
                stcg(P.r + vo, g);
                stcg(P.z + vo, z);
                if (sizeof(T) == 4 && !FACT) stcg((float *)P.zT + vo, (float)z);
                v1 = g * g;
                v2 = g * z;
            }
            if constexpr (FACT) {
                const float rv = fact_row_lane(P, cm, act ? z : 0.0, sub, row);
                if (act) stcg((float *)P.zT + vo, rv);
            }
        } else {
            double p = 0.0;
            if (act) {
                if (MODE == CAM_MATVEC) p = P.p[vo];
                else if (MODE == CAM_SR) p = ldcg(P.z + vo);
                else p = first ? ldcg(P.z + vo) : fma(beta, ldcg(p_prev + vo), ldcg(P.z + vo));
            }
            double bp = 0.0;
#pragma unroll
            for (int b = 0; b < 9; ++b) {
                const double pb = __shfl_sync(full, p, 9 * sub + b);
                if (act) bp = fma(kEarly ? brow[b] : __ldg(Mrow + b), pb, bp);
            }
            const double q = act ? bp - cs : 0.0;
            if (act) {
                stcg(P.q + vo, q);
                if (MODE == CAM_ITER) {
                    stcg(p_cur + vo, p);
                    if (sizeof(T) == 4 && !FACT && P.pcg_use_ps) stcg((T *)(p_cur == P.p ? P.pT : P.pT2) + vo, (T)p);
                }
                if (MODE == CAM_SR) {
                    const double rv = ldcg(P.r + vo);
                    v1 = rv * rv;
                    v2 = rv * p;
                    v3 = q * p;
                } else {
                    v1 = p * q;
                }
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            v1 += __shfl_xor_sync(full, v1, d);
            v2 += __shfl_xor_sync(full, v2, d);
            if (MODE == CAM_SR) v3 += __shfl_xor_sync(full, v3, d);
        }
        d1 += v1;
        d2 += v2;
        d3 += v3;
    }
    if constexpr (MODE == CAM_SR) {
        const double3 t = cta_sum3(lane == 0 ? d1 : 0.0, lane == 0 ? d2 : 0.0, lane == 0 ? d3 : 0.0, false, sb);
        *third = t.z;
        return make_double2(t.x, t.y);
    }
    // CTA partials in a fixed order (warp w's cameras, then a tree over warps);
    // d1, d2 are already warp-uniform, so no per-warp shuffle tree is needed
    return cta_sum2(lane == 0 ? d1 : 0.0, lane == 0 ? d2 : 0.0, false, sb);
}

// Search direction into shared memory (dense nc x 9, in T): p = z + beta p_prev
// (p = z on the first iteration), or the given FP64 p (src_given).  The FP32
// form builds it from float copies of z and p_prev with float4 loads; the FP64
// form from the FP64 vectors, as the camera pass does.
// Factored form: the camera rows instead (stride kRowS): the constants once
// (first), the nine linear entries as row(z) + beta times the row of the
// previous iteration that is still in shared memory, or the rows of the given
// FP64 p.
template <typename T, bool FACT>
__device__ void stage_p(const Prob &P, T *ps, const double *p_prev, const T *pT_prev, double beta, bool first,
                        const double *src_given) {
    if constexpr (FACT) {
        if (!src_given) {
            const float4 *z4 = (const float4 *)P.zT;
            const float fb = (float)beta;
            const int nq = P.nc * 3;  // three float4 per camera: n, h, (v_f, v_a, v_b)
            for (int e = threadIdx.x; e < nq; e += blockDim.x) {
                const int cam = e / 3, part = e - 3 * cam;
                const float4 z = __ldcg(z4 + e);
                float4 *dst = (float4 *)(ps + cam * kRowS) + part;
                float4 v = z;
                if (!first) {
                    const float4 o = *dst;
                    v = make_float4(fmaf(fb, o.x, z.x), fmaf(fb, o.y, z.y), fmaf(fb, o.z, z.z), fmaf(fb, o.w, z.w));
                    if (part == 2) v.y = o.y, v.z = o.z, v.w = o.w;
                } else if (part == 2) {
                    const float *st = P.camstat + (int64_t)cam * kCamStat;
                    v.y = __ldg(st), v.z = __ldg(st + 1), v.w = __ldg(st + 2);
                    dst[1] = make_float4(__ldg(st + 3), __ldg(st + 4), __ldg(st + 5), __ldg(st + 6));
                }
                *dst = v;
            }
        } else {
            for (int cam = threadIdx.x; cam < P.nc; cam += blockDim.x) {
                float v[9], r[kRowG];
#pragma unroll
                for (int j = 0; j < 9; ++j) v[j] = (float)src_given[(int64_t)cam * kVec + j];
                fact_row(P, cam, v, r);
                float4 *dst = (float4 *)(ps + cam * kRowS);
#pragma unroll
                for (int i = 0; i < kRowG / 4; ++i) dst[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
            }
        }
        __syncthreads();
        return;
    }
    const int total = P.nc * 9;
    if (sizeof(T) == 4 && !src_given) {
        const float4 *z4 = (const float4 *)P.zT, *p4 = (const float4 *)pT_prev;
        const float fb = (float)beta;
        const int nq = P.nc * (kVec / 4);  // float4 per camera row: 3 (9 values + padding)
        for (int e = threadIdx.x; e < nq; e += blockDim.x) {
            const int cam = e / 3, part = e - cam * 3;
            const float4 zv = __ldcg(z4 + e);
            float4 v = zv;
            if (!first) {
                const float4 pv = __ldcg(p4 + e);
                v = make_float4(fmaf(fb, pv.x, zv.x), fmaf(fb, pv.y, zv.y), fmaf(fb, pv.z, zv.z), fmaf(fb, pv.w, zv.w));
            }
            float *dst = (float *)ps + cam * 9 + part * 4;
            dst[0] = v.x;
            if (part < 2) {
                dst[1] = v.y;
                dst[2] = v.z;
                dst[3] = v.w;
            }
        }
        __syncthreads();
        return;
    }
    constexpr int U = 4;
    for (int e0 = threadIdx.x; e0 < total; e0 += blockDim.x * U) {
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * blockDim.x;
            v[u] = 0.0;
            if (e < total) {
                const int cam = e / 9, a = e - cam * 9;
                const int64_t vo = (int64_t)cam * kVec + a;
                if (src_given) v[u] = src_given[vo];
                else v[u] = first ? ldcg(P.z + vo) : fma(beta, ldcg(p_prev + vo), ldcg(P.z + vo));
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * blockDim.x;
            if (e < total) ps[e] = (T)v[u];
        }
    }
    __syncthreads();
}

// CTA-wide sums of two doubles in a fixed tree order; every thread gets the
// result.  With warp_data (warp-uniform) the warp first reduces its lanes by a
// shuffle tree; without it lane 0's value is taken as the warp's sum, so warps
// with nothing (or a single value) skip the tree: GB300's FP64 pipe takes 16
// cycles per warp instruction.  Warp 0 then adds the per-warp sums.
__device__ __forceinline__ double2 cta_sum2(double x, double y, bool warp_data, double *sb) {
    __shared__ double2 s_out2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (warp_data) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            y += __shfl_down_sync(0xffffffffu, y, o);
        }
    }
    __syncthreads();
    if (lane == 0) {
        sb[wid] = x;  // lane 0 holds the warp's sum (or its only value)
        sb[32 + wid] = y;
    }
    __syncthreads();
    if (wid == 0) {
        const bool in = lane < (int)(blockDim.x >> 5);
        double sx = in ? sb[lane] : 0.0, sy = in ? sb[32 + lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sx += __shfl_down_sync(0xffffffffu, sx, o);
            sy += __shfl_down_sync(0xffffffffu, sy, o);
        }
        if (lane == 0) s_out2 = make_double2(sx, sy);
    }
    __syncthreads();
    return s_out2;
}


// Two sums of n per-CTA partials in warp 0: each lane adds its partials in
// order (the loads in flight together), then one shuffle tree; valid in thread
// 0, which runs the scalar recurrences that use them.  (All warps adding the
// partials through cta_sum2 costs a second tree and three CTA barriers.)
__device__ __forceinline__ double2 sum_parts2(const double *a, const double *b, int n) {
    double x = 0.0, y = 0.0;
    if (threadIdx.x < 32) {
        for (int i0 = threadIdx.x; i0 < n; i0 += 160) {
            double u[5], v[5];
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const int i = i0 + 32 * j;
                u[j] = i < n ? ldcg(a + i) : 0.0;
                v[j] = (b && i < n) ? ldcg(b + i) : 0.0;
            }
            x += (u[0] + u[1]) + (u[2] + u[3]) + u[4];
            if (b) y += (v[0] + v[1]) + (v[2] + v[3]) + v[4];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            if (b) y += __shfl_down_sync(0xffffffffu, y, o);
        }
    }
    return make_double2(x, y);
}

__device__ __forceinline__ double sum_parts(const double *parts, int n) { return sum_parts2(parts, nullptr, n).x; }

// Three-value forms of cta_sum2 / sum_parts2 (the single-reduction PCG); sb
// holds 96 doubles.
__device__ __forceinline__ double3 cta_sum3(double x, double y, double z, bool warp_data, double *sb) {
    __shared__ double3 s_out3;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (warp_data) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            y += __shfl_down_sync(0xffffffffu, y, o);
            z += __shfl_down_sync(0xffffffffu, z, o);
        }
    }
    __syncthreads();
    if (lane == 0) {
        sb[wid] = x;
        sb[32 + wid] = y;
        sb[64 + wid] = z;
    }
    __syncthreads();
    if (wid == 0) {
        const bool in = lane < (int)(blockDim.x >> 5);
        double sx = in ? sb[lane] : 0.0, sy = in ? sb[32 + lane] : 0.0, sz = in ? sb[64 + lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sx += __shfl_down_sync(0xffffffffu, sx, o);
            sy += __shfl_down_sync(0xffffffffu, sy, o);
            sz += __shfl_down_sync(0xffffffffu, sz, o);
        }
        if (lane == 0) s_out3 = make_double3(sx, sy, sz);
    }
    __syncthreads();
    return s_out3;
}

__device__ __forceinline__ double3 sum_parts3(const double *a, const double *b, const double *c, int n, double *sb) {
    double x = 0.0, y = 0.0, z = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        x += ldcg(a + i);
        y += ldcg(b + i);
        z += ldcg(c + i);
    }
    return cta_sum3(x, y, z, (int)(threadIdx.x & ~31u) < n, sb);
}

// ---------------------------------------------------------------------------
// persistent PCG kernel (cooperative launch, one CTA per SM for the whole solve)
// ---------------------------------------------------------------------------
// JS: the camera pass reads the stored camera-major Jacobian (always in FP64;
// in FP32-mixed when the Jacobian comes from dual numbers).
// SR: the single-reduction recurrence (mba_pcg_variant), also its own instance.
template <typename T, bool JS, bool SR>
__global__ void __launch_bounds__(PcgBlock<T>::value, 1)
    pcg_kernel(Prob P, int mode, int max_iter, double tol, long long spin, int forcing) {
    using T2 = typename V2<T>::type;
    constexpr bool FACT = sizeof(T) == 4 && !JS;  // FP32-mixed, analytic Jacobian: the factored form
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double sb[96];
    DevState *st = P.st;
    if (st->done || st->blockfail) return;  // a failed damping: the LM loop rejects this iteration
    // forcing sequence: the first solve's right-hand side norm as it was before
    // this launch, read before the first grid barrier (block 0 writes it after
    // the last one)
    __shared__ double s_g0;
    if (threadIdx.x == 0) s_g0 = forcing ? st->g0 : 0.0;
    uint32_t epoch = 0;
    const int G = gridDim.x;
    const int nwarp = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T *pT = (T *)P.pT;
    T2 *sbuf = (T2 *)P.sbuf;
    double *part_rho = P.red, *part_rr = P.red + G, *part_pq = P.red + 2 * G;
    const int ncw = (P.nc + 2) / 3;  // warps of camera-row work (3 cameras x 9 rows per warp)
    const int my_sub = lane / 9, row = lane % 9;
    const unsigned full = 0xffffffffu;
    T *ps = P.pcg_use_ps ? (T *)smem_raw : nullptr;
    double *cslot = (double *)(smem_raw + P.pcg_ps_bytes);
    bool ok = true;
    auto barrier = [&]() -> bool { return grid_barrier(st, epoch, spin); };
    // the point pass of one product; rows: the search rows in global memory
    // (read where they are not in shared memory)
    auto point_pass_iter = [&](const T *rows) { point_pass_any<T, false, FACT>(P, ps, rows, sbuf); };
    // owner's copy of a vector's camera row (factored form): the nine linear
    // entries (zT), or the whole row where the point pass reads it from global memory
    auto store_row = [&](int cam, bool act, double val, float *lin, float *whole) {
        const float r = fact_row_lane(P, cam, act ? val : 0.0, my_sub, row);
        if (!act) return;
        if (lin) stcg(lin + (int64_t)cam * kVec + row, r);
        if (whole) {
            stcg(whole + (int64_t)cam * kRowG + row, r);
            if (row < 7) stcg(whole + (int64_t)cam * kRowG + 9 + row, P.camstat[(int64_t)cam * kCamStat + row]);
        }
    };
    // owner phase: p = z + beta p_prev written in FP64 and, for the gathers, as
    // T (or, in the factored form, as the camera's row)
    auto phase_p = [&](const double *p_prev, double *p_cur, double beta, bool first, const double *given) {
        for (int w = blockIdx.x * nwarp + wid; w < ncw; w += G * nwarp) {
            const int cam = w * 3 + my_sub;
            const bool act = lane < 27 && cam < P.nc;
            double pn = 0.0;
            if (act) {
                const int64_t vo = (int64_t)cam * kVec + row;
                pn = given ? given[vo] : (first ? ldcg(P.z + vo) : fma(beta, ldcg(p_prev + vo), ldcg(P.z + vo)));
                if (!given) stcg(p_cur + vo, pn);
                if (!FACT) stcg(pT + vo, (T)pn);
            }
            if constexpr (FACT) store_row(act ? cam : 0, act, pn, nullptr, (float *)pT);
        }
    };

    if (mode == PCG_MATVEC) {
        // p given in P.p (FP64): q = B~ p - E C~^-1 E^T p
        if (ps) {
            stage_p<T, FACT>(P, ps, nullptr, nullptr, 0.0, true, P.p);
        } else {
            phase_p(nullptr, nullptr, 0.0, true, P.p);
            if (!(ok = barrier())) return;
        }
        point_pass_iter(pT);
        if (barrier()) camera_pass<T, CAM_MATVEC, JS>(P, sbuf, nullptr, nullptr, 0.0, true, cslot, sb);
        return;
    }

    // ---- right-hand side g = v - E C~^-1 w (Eq. 3), x = 0, r = g, z = B~^-1 g ----
    point_pass_any<T, true, FACT>(P, nullptr, nullptr, sbuf);
    ok = barrier();
    if (ok) {
        const double2 d = camera_pass<T, CAM_RHS, JS>(P, sbuf, nullptr, nullptr, 0.0, true, cslot, sb);
        if (mode == PCG_RHS_ONLY) return;
        if (threadIdx.x == 0) {
            stcg(part_rr + blockIdx.x, d.x);
            stcg(part_rho + blockIdx.x, d.y);
        }
        ok = barrier();
    }

    if constexpr (SR) {
        // Single-reduction PCG (Chronopoulos-Gear form; the oracle's
        // pcg_single_reduction).  Step n: the point pass forms s~ for u_n,
        // barrier, the camera pass gives w_n = S~ u_n at each camera's owner and
        // the partials of r.r, r.u and w.u, barrier, then every CTA derives
        // alpha and beta from the three sums and the owners update p, s, x, r
        // and u = B~^-1 r and write u's rows, which a third barrier publishes
        // to the next point pass.  Three barriers and one reduction per step
        // (the standard loop: three barriers and two reductions with the rows
        // in shared memory, four barriers otherwise).
        // Not kept: a two-barrier form in which every CTA formed u's rows from
        // the recurrence u_{n+1} = u_n - alpha B~^-1 s_n in FP32.  As |u| falls
        // over the solve, that subtraction cancels and the FP32 rounding of the
        // earlier, larger terms dominates: 1e-3 relative error in the step after
        // 10 PCG steps and 0.03 to 0.15 after 30, against 1.5e-5 for the rows
        // written by the owners.
        __shared__ double s_alpha, s_beta, s_r0, s_rn, s_stop2, s_gprev, s_aprev;
        __shared__ int s_go;
        // where the point pass finds u's rows when they are not in shared memory
        const T *rows_u = FACT ? (const T *)P.pT : (sizeof(T) == 8 ? (const T *)P.z : (const T *)P.zT);
        if (FACT && !ps) {  // u_0's rows, published by a barrier of their own
            phase_p(nullptr, P.p, 0.0, true, nullptr);
            ok = barrier();
        }
        int n = 0;
        while (ok && (n == 0 || n < max_iter)) {
            if (ps) stage_p<T, FACT>(P, ps, nullptr, nullptr, 0.0, true, nullptr);
            point_pass_iter(rows_u);
            if (!(ok = barrier())) break;
            {
                double wu = 0.0;
                const double2 d =
                    camera_pass<T, CAM_SR, JS>(P, sbuf, nullptr, nullptr, 0.0, false, cslot, sb, &wu);
                if (threadIdx.x == 0) {
                    stcg(part_rr + blockIdx.x, d.x);
                    stcg(part_rho + blockIdx.x, d.y);
                    stcg(part_pq + blockIdx.x, wu);
                }
            }
            if (!(ok = barrier())) break;
            const double3 sums = sum_parts3(part_rr, part_rho, part_pq, G, sb);
            if (threadIdx.x == 0) {
                // sums: r.r, gamma = r.u, delta = w.u
                bool go;
                if (n == 0) {
                    const double r0 = sqrt(sums.x);
                    double t = tol;
                    if (forcing) {  // eta = min(0.1, sqrt(|g| / |g_first|)), |g_first| = r0 in the first solve
                        const double g0 = s_g0;
                        t = fmax(t, fmin(0.1, sqrt(r0 / (g0 > 0.0 ? g0 : r0))));
                    }
                    s_r0 = r0;
                    s_stop2 = (t * r0) * (t * r0);
                    go = r0 > 0.0;
                } else {
                    go = !(sums.x <= s_stop2);
                }
                s_rn = sqrt(sums.x);
                go = go && isfinite(sums.y);
                const double beta = n == 0 ? 0.0 : sums.y / s_gprev;
                const double den = n == 0 ? sums.z : sums.z - beta * sums.y / s_aprev;  // p.S p
                go = go && den > 0.0 && isfinite(den);
                const double alpha = go ? sums.y / den : 0.0;
                s_gprev = sums.y;
                s_aprev = alpha;
                s_alpha = alpha;
                s_beta = beta;
                s_go = go ? 1 : 0;
            }
            __syncthreads();
            if (!s_go) break;
            const double alpha = s_alpha, beta = s_beta;
            // p = u + beta p, s = w + beta s (s in the free second direction buffer),
            // x += alpha p, r -= alpha s, u = B~^-1 r over this CTA's own cameras
            const bool last = n + 1 >= max_iter;  // the step cap ends the solve after this update
            {
                double *sv = P.p2;
                double rr = 0.0;  // |r|^2 after the update, taken on the last step only
                const int cb = P.cta_cam[blockIdx.x], ce = P.cta_cam[blockIdx.x + 1];
                for (int c0 = cb + 3 * wid; c0 < ce; c0 += 3 * nwarp) {
                    const int cam = c0 + my_sub;
                    const bool act = lane < 27 && cam < ce;
                    const int64_t vo = (int64_t)(act ? cam : c0) * kVec + row;
                    double rv = 0.0;
                    if (act) {
                        const double u = ldcg(P.z + vo), w = ldcg(P.q + vo);
                        const double pn = n == 0 ? u : fma(beta, ldcg(P.p + vo), u);
                        const double sn = n == 0 ? w : fma(beta, ldcg(sv + vo), w);
                        stcg(P.p + vo, pn);
                        stcg(sv + vo, sn);
                        stcg(P.x + vo, fma(alpha, pn, ldcg(P.x + vo)));
                        rv = fma(-alpha, sn, ldcg(P.r + vo));
                        stcg(P.r + vo, rv);
                        rr = fma(rv, rv, rr);
                    }
                    double z = 0.0;
#pragma unroll
                    for (int c = 0; c < 9; ++c) {
                        const double rc = __shfl_sync(full, rv, my_sub * 9 + c);
                        if (act) z = fma(__ldg(P.Binv + 81 * (int64_t)cam + row * 9 + c), rc, z);
                    }
                    if constexpr (FACT)
                        store_row(act ? cam : c0, act, z, ps ? (float *)P.zT : nullptr, ps ? nullptr : (float *)pT);
                    if (act) {
                        stcg(P.z + vo, z);
                        if (sizeof(T) == 4 && !FACT) stcg((float *)P.zT + vo, (float)z);
                    }
                }
                if (last) {
                    // the residual norm the solve reports, in its own partials (the
                    // step's sums may still be read by other CTAs)
                    const double2 t = cta_sum2(rr, 0.0, true, sb);
                    if (threadIdx.x == 0) stcg(P.red + 3 * G + blockIdx.x, t.x);
                }
            }
            ++n;
            if (last) {
                if (!(ok = barrier())) break;
                const double rrn = sum_parts(P.red + 3 * G, G);
                if (threadIdx.x == 0) s_rn = sqrt(rrn);
                __syncthreads();
                break;
            }
            if (!(ok = barrier())) break;
        }
        if (!ok) atomicCAS(&st->err, 0, (int)MBA_ERR_TIMEOUT);
        if (ok && blockIdx.x == 0 && threadIdx.x == 0) {
            st->pcg_iters = n;
            st->pcg_rel_res = s_r0 > 0.0 ? s_rn / s_r0 : 0.0;
            if (forcing && !(s_g0 > 0.0)) st->g0 = s_r0;
        }
        return;
    }

    // The scalar recurrences (r0, rho, alpha, beta, the stopping test) run in
    // thread 0 alone and are broadcast through shared memory: on this GPU each
    // warp-wide FP64 instruction holds the SM's FP64 pipe for 16 cycles and a
    // division or square root is a chain of about ten of them, so evaluating
    // them redundantly in all 1024 threads would stall every CTA for microseconds.
    // Thread 0's state (r0, rho, |r|, the stopping threshold) also lives in
    // shared memory, so that no register stays reserved for it through the loop.
    __shared__ double s_alpha, s_beta, s_r0, s_rho, s_rn, s_stop;
    __shared__ int s_go;
    int n = 0;
    if (ok) {
        const double2 s0 = sum_parts2(part_rr, part_rho, G);
        if (threadIdx.x == 0) {
            const double r0 = sqrt(s0.x);
            double t = tol;
            if (forcing) {  // eta = min(0.1, sqrt(|g| / |g_first|)), |g_first| = r0 in the first solve
                const double g0 = s_g0;
                t = fmax(t, fmin(0.1, sqrt(r0 / (g0 > 0.0 ? g0 : r0))));
            }
            s_r0 = r0;
            s_rho = s0.y;
            s_rn = r0;
            s_stop = t * r0;
            s_go = (r0 > 0.0 && isfinite(s0.y)) ? 1 : 0;
            s_beta = 0.0;
        }
        __syncthreads();
    }
    if (ok && s_go) {
        for (;;) {
            const double beta = s_beta;
            double *p_cur = (n & 1) ? P.p2 : P.p;
            const double *p_prev = (n & 1) ? P.p : P.p2;
            const T *pT_prev = (n & 1) ? pT : (T *)P.pT2;
            if (ps) {
                stage_p<T, FACT>(P, ps, p_prev, pT_prev, beta, n == 0, nullptr);
            } else {
                phase_p(p_prev, p_cur, beta, n == 0, nullptr);
                if (!(ok = barrier())) break;
            }
            point_pass_iter(pT);
            if (!(ok = barrier())) break;
            {
                const double2 d = camera_pass<T, CAM_ITER, JS>(P, sbuf, p_prev, p_cur, beta, n == 0, cslot, sb);
                if (threadIdx.x == 0) stcg(part_pq + blockIdx.x, d.x);
            }
            if (!(ok = barrier())) break;
            const double pq = sum_parts(part_pq, G);
            if (threadIdx.x == 0) {
                const bool go = (pq > 0.0) && isfinite(pq);
                s_go = go ? 1 : 0;
                s_alpha = go ? s_rho / pq : 0.0;
            }
            __syncthreads();
            if (!s_go) break;
            const double alpha = s_alpha;
            // x += alpha p; r -= alpha q; z = B~^-1 r; partial r.r and r.z, over this
            // CTA's own cameras (three per warp)
            {
                double rr = 0.0, rz = 0.0;
                const int cb = P.cta_cam[blockIdx.x], ce = P.cta_cam[blockIdx.x + 1];
                for (int c0 = cb + 3 * wid; c0 < ce; c0 += 3 * nwarp) {
                    const int cam = c0 + my_sub;
                    const bool act = lane < 27 && cam < ce;
                    const int64_t vo = (int64_t)(act ? cam : c0) * kVec + row;
                    // this lane's row of B~^-1, loaded beside (not after) the r update
                    double bi[9];
#pragma unroll
                    for (int c = 0; c < 9; ++c) bi[c] = act ? __ldg(P.Binv + 81 * (int64_t)cam + row * 9 + c) : 0.0;
                    double rv = 0.0;
                    if (act) {
                        stcg(P.x + vo, fma(alpha, ldcg(p_cur + vo), ldcg(P.x + vo)));
                        rv = fma(-alpha, ldcg(P.q + vo), ldcg(P.r + vo));
                        stcg(P.r + vo, rv);
                    }
                    double z = 0.0;
#pragma unroll
                    for (int c = 0; c < 9; ++c) {
                        const double rc = __shfl_sync(full, rv, my_sub * 9 + c);
                        z = fma(bi[c], rc, z);
                    }
                    if constexpr (FACT) {
                        if (ps) store_row(act ? cam : c0, act, z, (float *)P.zT, nullptr);
                    }
                    if (act) {
                        stcg(P.z + vo, z);
                        if (sizeof(T) == 4 && !FACT) stcg((float *)P.zT + vo, (float)z);
                        rr += rv * rv;
                        rz += rv * z;
                    }
                }
                const bool has = cb + 3 * wid < ce;
                const double2 sr = cta_sum2(rr, rz, has, sb);
                if (threadIdx.x == 0) {
                    stcg(part_rr + blockIdx.x, sr.x);
                    stcg(part_rho + blockIdx.x, sr.y);
                }
            }
            if (!(ok = barrier())) break;
            ++n;
            const double2 sums = sum_parts2(part_rho, part_rr, G);
            if (threadIdx.x == 0) {
                const double rho_prev = s_rho, rho = sums.x, rn = sqrt(sums.y);
                s_rho = rho;
                s_rn = rn;
                const bool go = !(rn <= s_stop || n >= max_iter) && isfinite(rho);
                s_go = go ? 1 : 0;
                s_beta = go ? rho / rho_prev : 0.0;
            }
            __syncthreads();
            if (!s_go) break;
        }
    }
    if (!ok) atomicCAS(&st->err, 0, (int)MBA_ERR_TIMEOUT);
    if (ok && blockIdx.x == 0 && threadIdx.x == 0) {
        st->pcg_iters = n;
        st->pcg_rel_res = s_r0 > 0.0 ? s_rn / s_r0 : 0.0;
        if (forcing && !(s_g0 > 0.0)) st->g0 = s_r0;
    }
}

#include "pcg_own.cuh"

// ---------------------------------------------------------------------------
// back-substitution dp_j = C~_j^-1 (w_j - sum_k Jp~_k^T Jc~_k dc_i(k)) (Eq. 4),
// candidate points, and the model decrease sum_k (-e~_k.d_k - |d_k|^2/2)
// with d_k = Jc~_k dc + Jp~_k dp.
// ---------------------------------------------------------------------------
// Per observation: t = Jc~ dc and Jp~, so that u = jp^T t is this observation's
// term of Jp~^T Jc~ dc.
template <typename T>
__device__ __forceinline__ void backsub_obs(const Prob &P, int64_t o, int cam, T *t, T *jp) {
    T Jc[18];
    load_jac_stream((const T *)P.J, P.npad, o, Jc, jp);
    const double *xc = P.x + (int64_t)cam * kVec;
    t[0] = t[1] = T(0);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const T xa = (T)xc[a];
        t[0] += Jc[a] * xa;
        t[1] += Jc[9 + a] * xa;
    }
}
// Model-decrease term of one observation given its point step: d~ = J~_k (dc, dp),
// -e~.d~ - |d~|^2 / 2.
template <typename T>
__device__ __forceinline__ double backsub_dec(const Prob &P, int64_t o, const T *t, const T *jp, const T *dp) {
    const T d0 = jp[0] * dp[0] + jp[1] * dp[1] + jp[2] * dp[2] + t[0];
    const T d1 = jp[3] * dp[0] + jp[4] * dp[1] + jp[5] * dp[2] + t[1];
    const T *res = (const T *)P.res;
    const double e0 = (double)__ldcs(res + o), e1 = (double)__ldcs(res + P.npad + o);
    const double dd0 = (double)d0, dd1 = (double)d1;
    return -(e0 * dd0 + e1 * dd1) - 0.5 * (dd0 * dd0 + dd1 * dd1);
}
// The point step dp_j = C~_j^-1 (w_j - a), its FP64 copy and the candidate point.
template <typename T>
__device__ __forceinline__ void backsub_point(const Prob &P, int pt, const T *a, T *dp) {
    const T t0 = (T)P.w[3 * (int64_t)pt] - a[0], t1 = (T)P.w[3 * (int64_t)pt + 1] - a[1],
            t2 = (T)P.w[3 * (int64_t)pt + 2] - a[2];
    sym3_apply((const T *)P.Cinv + 6 * (int64_t)pt, t0, t1, t2, dp);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        P.dp[3 * (int64_t)pt + k] = (double)dp[k];
        P.pts_new[3 * (int64_t)pt + k] = P.pts[3 * (int64_t)pt + k] + (double)dp[k];
    }
}

// ---------------------------------------------------------------------------
// back-substitution dp_j = C~_j^-1 (w_j - sum_k Jp~_k^T Jc~_k dc_i(k)) (Eq. 4),
// candidate points, and the model decrease sum_k (-e~_k.d_k - |d_k|^2/2)
// with d_k = Jc~_k dc + Jp~_k dp, in one sweep over point-major warp chunks:
// a segmented scan gives each point's sum, its last lane forms dp and the
// point's lanes take it by a shuffle.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kBlock) backsub_kernel(Prob P, double *partial) {
    __shared__ double sb[kWarps];
    if (P.st->done) return;
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    double ldec = 0.0;
    for (int w = blockIdx.x * nwarp + (threadIdx.x >> 5); w < P.n_wchunks; w += gridDim.x * nwarp) {
        const int2 c0 = P.wchunk[w], c1 = P.wchunk[w + 1];
        const int o0 = c0.y, m = c1.y - c0.y;
        if (m <= 32) {
            const bool act = lane < m;
            const int64_t o = (int64_t)o0 + (act ? lane : 0);
            const int npts = c1.x - c0.x;
            const int rs = lane < npts ? __ldg(P.pt_ptr + c0.x + lane) - o0 : 32;
            const unsigned starts = __reduce_or_sync(full, rs < 32 ? (1u << rs) : 0u);
            const int pt = act ? c0.x + __popc(starts & (0xffffffffu >> (31 - lane))) - 1 : -1 - lane;
            T t[2] = {T(0), T(0)}, jp[6], u[3];
#pragma unroll
            for (int k = 0; k < 6; ++k) jp[k] = T(0);
            if (act) backsub_obs<T>(P, o, __ldg(P.pm_cam + o), t, jp);
            u[0] = jp[0] * t[0] + jp[3] * t[1];
            u[1] = jp[1] * t[0] + jp[4] * t[1];
            u[2] = jp[2] * t[0] + jp[5] * t[1];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int kp = __shfl_up_sync(full, pt, d);
                const T v0 = __shfl_up_sync(full, u[0], d), v1 = __shfl_up_sync(full, u[1], d),
                        v2 = __shfl_up_sync(full, u[2], d);
                if (lane >= d && kp == pt) {
                    u[0] += v0;
                    u[1] += v1;
                    u[2] += v2;
                }
            }
            const int nxt = __shfl_down_sync(full, pt, 1);
            const bool tail = act && (lane == m - 1 || nxt != pt);
            T dp[3] = {T(0), T(0), T(0)};
            if (tail) backsub_point<T>(P, pt, u, dp);
            const unsigned tails = __ballot_sync(full, tail);
            const unsigned mine = tails & (0xffffffffu << lane);
            const int src = mine ? __ffs(mine) - 1 : lane;
            T dq[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) dq[k] = __shfl_sync(full, dp[k], src);
            if (act) ldec += backsub_dec<T>(P, o, t, jp, dq);
        } else {
            // one point with a long track: the sum over 32-observation slices, then
            // a second sweep for the model decrease
            const int pt = c0.x;
            T a[3] = {T(0), T(0), T(0)};
            for (int base = 0; base < m; base += 32) {
                if (base + lane < m) {
                    const int64_t o = (int64_t)o0 + base + lane;
                    T t[2], jp[6];
                    backsub_obs<T>(P, o, __ldg(P.pm_cam + o), t, jp);
#pragma unroll
                    for (int k = 0; k < 3; ++k) a[k] += jp[k] * t[0] + jp[3 + k] * t[1];
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) a[k] += __shfl_xor_sync(full, a[k], d);
            T dp[3] = {T(0), T(0), T(0)};
            if (lane == 0) backsub_point<T>(P, pt, a, dp);
#pragma unroll
            for (int k = 0; k < 3; ++k) dp[k] = __shfl_sync(full, dp[k], 0);
            for (int base = 0; base < m; base += 32) {
                if (base + lane < m) {
                    const int64_t o = (int64_t)o0 + base + lane;
                    T t[2], jp[6];
                    backsub_obs<T>(P, o, __ldg(P.pm_cam + o), t, jp);
                    ldec += backsub_dec<T>(P, o, t, jp, dp);
                }
            }
        }
    }
    const double s = block_sum(ldec, sb);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// The same over the slices of the factored form: t and u as in the PCG point
// pass from the rows of dc; the second sweep over the lane's observations
// recomputes t, adds Jp dp = D R dp (R from the quaternion) and the residual
// e = f d p - u, and sums the model decrease -W (e.d + |d|^2 / 2), one FP64
// addition per observation.  SMEM: the CTA forms the rows of dc in shared memory.
template <bool SMEM>
__global__ void __launch_bounds__(1024, 1) backsub_slices_kernel(Prob P, double *partial) {
    __shared__ double sb[32];
    if (P.st->done) return;
    extern __shared__ __align__(16) float s_rows[];
    if (SMEM) {
        for (int cam = threadIdx.x; cam < P.nc; cam += blockDim.x) {
            float v[9], r[kRowG];
#pragma unroll
            for (int j = 0; j < 9; ++j) v[j] = (float)P.x[(int64_t)cam * kVec + j];
            fact_row(P, cam, v, r);
            float4 *dst = (float4 *)(s_rows + cam * kRowS);
#pragma unroll
            for (int i = 0; i < kRowG / 4; ++i) dst[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
        }
        __syncthreads();
    }
    const float *ps = SMEM ? s_rows : nullptr, *rows = (const float *)P.pT;
    const float *__restrict__ Ci = (const float *)P.Cinv;
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    double ldec = 0.0;
    for (int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < P.n_slices; w += gridDim.x * nwarp) {
        const int4 sl = __ldg(P.slice + w);
        const int K = sl.w & 0xffff, lg = sl.w >> 16, in = lane >> lg;
        const bool act = in < (sl.y & 0xff);
        const int s = sl.x + (act ? in : 0);
        float a[3];
        fact_slice_sum(P, ps, rows, (int64_t)sl.z + lane, K, a);
        for (int d = 1; d < (1 << lg); d <<= 1) {
#pragma unroll
            for (int q = 0; q < 3; ++q) a[q] += __shfl_xor_sync(full, a[q], d);
        }
        const int64_t pt = __ldg(P.sp_pt + s);
        if (P.has_fixed && P.pt_fixed[pt]) a[0] = a[1] = a[2] = 0.f;
        float ci[6], dp[3];
#pragma unroll
        for (int q = 0; q < 6; ++q) ci[q] = __ldg(Ci + (int64_t)q * P.np_pad + s);
        apply_sym3(ci, (float)P.w[3 * pt] - a[0], (float)P.w[3 * pt + 1] - a[1], (float)P.w[3 * pt + 2] - a[2], dp);
        if (act && (lane & ((1 << lg) - 1)) == 0) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                P.dp[3 * pt + k] = (double)dp[k];
                P.pts_new[3 * pt + k] = P.pts[3 * pt + k] + (double)dp[k];
            }
        }
        const bool fixed = P.has_fixed && P.pt_fixed[pt];
        const float f0 = fixed ? 0.f : dp[0], f1 = fixed ? 0.f : dp[1], f2 = fixed ? 0.f : dp[2];
        for (int k = 0; k < K; ++k) {
            const int64_t slot = (int64_t)sl.z + 32 * k + lane;
            const FactStream st = load_stream(P, slot);
            if (st.cam < 0) continue;
            const float px = st.px, py = st.py, iz = st.iz, W = st.W;
            const float2 uv = __ldg(P.sl_uv32 + slot);
            const CamRow r = load_row(ps, rows, st.cam);
            FactObs o = fact_obs(px, py, iz, r);
            const float c0 = r.q2 * f2 - r.q3 * f1, c1 = r.q3 * f0 - r.q1 * f2, c2 = r.q1 * f1 - r.q2 * f0;
            o.w0 += iz * (f0 + r.q0 * c0 + (r.q2 * c2 - r.q3 * c1));
            o.w1 += iz * (f1 + r.q0 * c1 + (r.q3 * c0 - r.q1 * c2));
            o.w2 += iz * (f2 + r.q0 * c2 + (r.q1 * c1 - r.q2 * c0));
            float d0, d1;
            fact_t(o, px, py, d0, d1);
            const float r2 = px * px + py * py, fd = r.f * (1.f + r2 * (r.k1 + r.k2 * r2));
            const float e0 = fd * px - uv.x, e1 = fd * py - uv.y;
            ldec -= (double)(W * (d0 * (e0 + 0.5f * d0) + d1 * (e1 + 0.5f * d1)));
        }
    }
    const double s = block_sum(ldec, sb);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// FP64 form over slices (block-owned layout): u = H alpha + g sigma as in the
// PCG; with delta = alpha + dp the model term of an observation is
// |d|^2 = delta^T H delta + 2 sigma g.delta + sigma^2 W r2, and
// -sum e~.d = v.dc + w.dp, the gradient against the step.
__global__ void __launch_bounds__(512, 1) backsub_slices64_kernel(Prob P, double *partial) {
    __shared__ double sb[32];
    if (P.st->done) return;
    extern __shared__ __align__(16) double s_rows64[];
    for (int e = threadIdx.x; e < 10 * P.nc; e += blockDim.x) {
        const int cam = e / 10, q = e - 10 * cam, g0 = q < 3 ? 0 : (q < 6 ? 3 : 6);
        double r;
        if (q == 9) {
            r = __ldg((const double *)P.camtab + (int64_t)cam * kCamTab + 24);
        } else {
            const double *ct = P.ctr64 + (int64_t)cam * kCtr + 3 * g0 + (q - g0), *v = P.x + (int64_t)cam * kVec + g0;
            r = fixed_camera(P, cam) ? 0.0 : fma(ct[0], v[0], fma(ct[3], v[1], ct[6] * v[2]));
        }
        s_rows64[cam * kRowD + q] = r;
    }
    __syncthreads();
    const double *__restrict__ Ci = (const double *)P.Cinv;
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    double ldec = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 9 * (int64_t)P.nc; t += (int64_t)gridDim.x * blockDim.x)
        ldec = fma(P.v[t], P.x[t / 9 * kVec + t % 9], ldec);
    for (int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < P.n_slices; w += gridDim.x * nwarp) {
        const int4 sl = __ldg(P.slice + w);
        const int K = sl.w & 0xffff, lg = sl.w >> 16, in = lane >> lg;
        const bool act = in < (sl.y & 0xff);
        const int s = sl.x + (act ? in : 0);
        const double X[3] = {__ldg(P.sp_X64 + 4 * (int64_t)s), __ldg(P.sp_X64 + 4 * (int64_t)s + 1),
                             __ldg(P.sp_X64 + 4 * (int64_t)s + 2)};
        double a[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < K; ++k) {
            const HgObs o = load_hg(P, (int64_t)sl.z + 32 * k + lane);
            if (o.cam >= 0) hg_u(P, o, s_rows64 + o.cam * kRowD, X, a);
        }
        for (int d = 1; d < (1 << lg); d <<= 1) {
#pragma unroll
            for (int q = 0; q < 3; ++q) a[q] += __shfl_xor_sync(full, a[q], d);
        }
        const int64_t pt = __ldg(P.sp_pt + s);
        if (P.has_fixed && P.pt_fixed[pt]) a[0] = a[1] = a[2] = 0.0;
        double ci[6], dp[3];
#pragma unroll
        for (int q = 0; q < 6; ++q) ci[q] = __ldg(Ci + (int64_t)q * P.np_pad + s);
        const double w0 = P.w[3 * pt], w1 = P.w[3 * pt + 1], w2 = P.w[3 * pt + 2];
        apply_sym3(ci, w0 - a[0], w1 - a[1], w2 - a[2], dp);
        if (act && (lane & ((1 << lg) - 1)) == 0) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                P.dp[3 * pt + k] = dp[k];
                P.pts_new[3 * pt + k] = P.pts[3 * pt + k] + dp[k];
            }
            ldec += w0 * dp[0] + w1 * dp[1] + w2 * dp[2];
        }
        if (P.has_fixed && P.pt_fixed[pt]) dp[0] = dp[1] = dp[2] = 0.0;  // moves no pixel
        for (int k = 0; k < K; ++k) {
            const int64_t slot = (int64_t)sl.z + 32 * k + lane;
            const HgObs o = load_hg(P, slot);
            if (o.cam < 0) continue;
            const double *r = s_rows64 + o.cam * kRowD;
            double al[3];
            hg_alpha(P, r, o.cam, X, al);
            const double sg = fma(o.v[9], fma(o.v[9], r[8], r[7]), r[6]);
            const double d0 = al[0] + dp[0], d1 = al[1] + dp[1], d2 = al[2] + dp[2];
            const double h0 = fma(o.v[0], d0, fma(o.v[1], d1, fma(o.v[2], d2, 2.0 * sg * o.v[6])));
            const double h1 = fma(o.v[1], d0, fma(o.v[3], d1, fma(o.v[4], d2, 2.0 * sg * o.v[7])));
            const double h2 = fma(o.v[2], d0, fma(o.v[4], d1, fma(o.v[5], d2, 2.0 * sg * o.v[8])));
            const double wr = P.sl_w64 ? __ldg(P.sl_w64 + slot) * o.v[9] : o.v[9];
            ldec -= 0.5 * fma(d0, h0, fma(d1, h1, fma(d2, h2, sg * sg * wr)));
        }
    }
    const double s = block_sum(ldec, sb);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// Camera rows (with the constants) of the PCG solution dc, for the factored
// back-substitution of problems whose rows do not fit in shared memory.
__global__ void fact_rows_kernel(Prob P, const double *__restrict__ x, float *__restrict__ rows) {
    if (P.st->done) return;
    for (int cam = blockIdx.x * blockDim.x + threadIdx.x; cam < P.nc; cam += gridDim.x * blockDim.x) {
        float v[9], r[kRowG];
#pragma unroll
        for (int j = 0; j < 9; ++j) v[j] = (float)x[(int64_t)cam * kVec + j];
        fact_row(P, cam, v, r);
        float4 *dst = (float4 *)(rows + (int64_t)cam * kRowG);
#pragma unroll
        for (int i = 0; i < kRowG / 4; ++i) dst[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
    }
}

__global__ void cams_new_kernel(Prob P) {
    if (P.st->done) return;
    const int64_t total = (int64_t)P.nc * 9;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / 9, a = t % 9;
        P.cams_new[t] = P.cams[t] + P.x[i * kVec + a];
    }
}

__global__ void ldec_final_kernel(const double *partial, int nb, DevState *st) {
    __shared__ double sb[kWarps];
    if (st->done) return;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += partial[i];
    const double s = block_sum(acc, sb);
    if (threadIdx.x == 0) st->model_dec = s;
}


}  // namespace

cudaError_t launch_damp(const Prob &P, int damping, int precond, const int32_t *cfirst, cudaStream_t s) {
    damp_cameras_kernel<<<(P.nc + kDampWarps - 1) / kDampWarps, 32 * kDampWarps, 0, s>>>(P, damping);
    const int64_t nb = (P.np + kBlock - 1) / kBlock;
    const unsigned g = (unsigned)(nb > 152 * 16 ? 152 * 16 : nb);
    if (P.fp32) damp_points_kernel<float><<<g, kBlock, 0, s>>>(P, damping);
    else damp_points_kernel<double><<<g, kBlock, 0, s>>>(P, damping);
    if (precond == MBA_PRECOND_SCHUR_JACOBI) {
        const int cw = (P.n_cchunks + kWarps - 1) / kWarps;
        const unsigned gc = (unsigned)(cw < 152 * 16 ? (cw > 0 ? cw : 1) : 152 * 16);
        if (P.fp32) {
            if (P.autodiff) sj_camera_kernel<float, true><<<gc, kBlock, 0, s>>>(P);
            else sj_camera_kernel<float, false><<<gc, kBlock, 0, s>>>(P);
        } else {
            if (P.autodiff) sj_camera_kernel<double, true><<<gc, kBlock, 0, s>>>(P);
            else sj_camera_kernel<double, false><<<gc, kBlock, 0, s>>>(P);
        }
        sj_finalize_kernel<<<(P.nc + kDampWarps - 1) / kDampWarps, 32 * kDampWarps, 0, s>>>(P, cfirst);
    }
    return cudaGetLastError();
}

// Shared-memory plan: the camera-pass chunk slots of the busiest CTA, plus the
// search direction (nc x 9) when it also fits; otherwise the point pass
// gathers p from global memory and an extra barrier is needed.
void plan_pcg_smem(Prob &P) {
    if (P.own) return;  // planned with the blocks (sell.cu)
    const int w = P.fp32 ? 4 : 8;
    const int per_cam = P.fact ? kRowS : 9;  // the factored form stages a row per camera
    const int64_t budget = 227 * 1024 - 12 * 1024;
    const int64_t slots = (int64_t)(P.fact ? P.pcg_max_cta_cams + 32 : P.pcg_max_cta_chunks) * 9 * 8;
    const int64_t psb = (((int64_t)P.nc * per_cam * w) + 127) & ~(int64_t)127;
    P.pcg_use_ps = (psb + slots <= budget) ? 1 : 0;
    P.pcg_ps_bytes = P.pcg_use_ps ? (int)psb : 0;
    P.pcg_smem = (int)(P.pcg_ps_bytes + slots);
}

int pcg_block(const Prob &P) { return P.fp32 ? PcgBlock<float>::value : PcgBlock<double>::value; }

template <bool SR>
static const void *pcg_fn_v(const Prob &P) {
    if (P.own && !P.fp32) return (const void *)pcg_own_kernel<double, SR, false>;
    if (P.own) return P.long_runs ? (const void *)pcg_own_kernel<float, SR, true> : (const void *)pcg_own_kernel<float, SR, false>;
    if (!P.fp32) return (const void *)pcg_kernel<double, true, SR>;
    return P.autodiff ? (const void *)pcg_kernel<float, true, SR> : (const void *)pcg_kernel<float, false, SR>;
}
static const void *pcg_fn(const Prob &P, int variant = MBA_PCG_STANDARD) {
    return variant == MBA_PCG_SINGLE_REDUCTION ? pcg_fn_v<true>(P) : pcg_fn_v<false>(P);
}

static int resident(const void *fn, int block, size_t smem) {
    int blocks = 0;
    if (allow_smem(fn) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, block, smem) != cudaSuccess) return 0;
    return blocks;
}

// One CTA per SM (the camera partition is built for exactly that many);
// returns 0 if either PCG instance (standard, single-reduction) cannot be
// resident with its shared memory.
int pcg_grid_size(const Prob &P) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = (size_t)P.pcg_smem;
    const bool ok = resident(pcg_fn(P), pcg_block(P), smem) >= 1 &&
                    resident(pcg_fn(P, MBA_PCG_SINGLE_REDUCTION), pcg_block(P), smem) >= 1;
    return ok ? sms : 0;
}

cudaError_t launch_pcg(const Prob &P, int mode, int max_iter, double tol, long long spin_limit, int grid,
                       cudaStream_t s, int forcing, int variant) {
    // the right-hand-side and product-only modes are the standard kernel's
    if (mode != PCG_SOLVE) variant = MBA_PCG_STANDARD;
    const size_t smem = (size_t)P.pcg_smem;
    // the barrier targets count arrivals from zero in every launch
    cudaError_t e = cudaMemsetAsync(&P.st->barrier, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    e = allow_smem(pcg_fn(P, variant));
    if (e != cudaSuccess) return e;
    Prob Pc = P;
    void *args[] = {(void *)&Pc, (void *)&mode, (void *)&max_iter, (void *)&tol, (void *)&spin_limit, (void *)&forcing};
    return cudaLaunchCooperativeKernel(pcg_fn(P, variant), dim3(grid), dim3(pcg_block(P)), args, smem, s);
}

cudaError_t launch_backsub(const Prob &P, double *partial, int nb, cudaStream_t s) {
    if (P.fact) {
        const int smem = P.nc * kRowS * 4;
        const SliceGrid g = slice_grid(P);
        nb = g.ctas;
        if (smem <= 220 * 1024) {
            if (cudaError_t e = allow_smem((const void *)backsub_slices_kernel<true>)) return e;
            backsub_slices_kernel<true><<<g.ctas, g.threads, smem, s>>>(P, partial);
        } else {
            fact_rows_kernel<<<(P.nc + 127) / 128, 128, 0, s>>>(P, P.x, (float *)P.pT);
            backsub_slices_kernel<false><<<g.ctas, g.threads, 0, s>>>(P, partial);
        }
    } else if (P.own) {
        const int smem = P.nc * kRowD * 8;  // fits: the block-owned product holds the same rows
        const SliceGrid g = slice_grid(P, 512);
        nb = g.ctas;
        if (cudaError_t e = allow_smem((const void *)backsub_slices64_kernel)) return e;
        backsub_slices64_kernel<<<g.ctas, g.threads, smem, s>>>(P, partial);
    } else if (P.fp32) {
        backsub_kernel<float><<<nb, kBlock, 0, s>>>(P, partial);
    } else {
        backsub_kernel<double><<<nb, kBlock, 0, s>>>(P, partial);
    }
    ldec_final_kernel<<<1, kBlock, 0, s>>>(partial, nb, P.st);
    cams_new_kernel<<<(P.nc * 9 + kBlock - 1) / kBlock, kBlock, 0, s>>>(P);
    return cudaGetLastError();
}

}  // namespace mba
