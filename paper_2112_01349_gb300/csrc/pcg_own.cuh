// pcg_own.cuh -- the PCG with block-owned products (layout: own.cu), included
// by pcg.cu.  Analytic Jacobian, FP32-mixed and FP64, where the camera rows fit
// in shared memory.
//
// Point side (per lane one point, or 1/G of it): u = W Jp^T Jc p.
//   FP32: from (px, py, 1/P_z) and the camera's row (see the factored form).
//   FP64: from H = W Jp^T Jp, g = W Jp^T p and r2, ten values per observation:
//     with m = M v_w and a' = R^T v_t per camera, Jc v = Jp alpha + p sigma,
//     alpha = a' + m x X, sigma = v_f + r2 (v_a + r2 v_b), so u = H alpha + g sigma:
//     20 FP64 instructions where the stored Jacobian takes 24, and 80 bytes
//     instead of 192.
// Camera side (per lane a run, or 1/G of it): the raw sums of a run,
//   FP32: RX x y, y, (1, r2, r2^2) p.s with y = D^T W Jp b from (RX, 1/P_z);
//   FP64: X x y, y, (1, r2, r2^2) q with y = H b, q = g.b: 24 instructions, and
//     none for reductions (the stored form's nine warp trees per chunk were a
//     fifth of its FP64 instructions, on the pipe that bounds it).
// The owner of a camera adds the partial sums of all blocks in block order and
// applies the camera's transform once (P.ctr, P.ctr64).
// In the first-order rotation branch (|w|^2 <= DBL_EPSILON) the Jacobian has
// -D [X]x where this form has -Jp [X]x: the FP64 rows carry a flag, and such
// cameras take the term w x (m x X) (and w x y) that makes up the difference.

template <typename T>
struct OwnShape;
template <>
struct OwnShape<float> {
    static constexpr int row = kRowS, part = kPartF;
};
template <>
struct OwnShape<double> {
    static constexpr int row = kRowD, part = kPartD;
};

// Warp-collective: the lane's component of a camera's row (FP64: m, a', v_f, v_a, v_b).
__device__ __forceinline__ float own_row_lane(const Prob &P, int cam, float v, int sub, int row) {
    return fact_row_lane(P, cam, (double)v, sub, row);
}
__device__ __forceinline__ double own_row_lane(const Prob &P, int cam, double v, int sub, int row) {
    const int g0 = row < 3 ? 0 : (row < 6 ? 3 : 6), at = 9 * sub + g0;
    const double *ct = P.ctr64 + (int64_t)cam * kCtr + 3 * g0 + (row - g0);
    double r = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) r = fma(__ldg(ct + 3 * i), __shfl_sync(0xffffffffu, v, (at + i) & 31), r);
    return fixed_camera(P, cam) ? 0.0 : r;
}

// Camera rows in shared memory: row(z) + beta row(previous p) (first: row(z) and
// the constants), or the rows of the given FP64 vector.
__device__ void own_stage(const Prob &P, float *rows, double beta, bool first, const double *given) {
    if (first || given) {
        for (int cam = threadIdx.x; cam < P.nc; cam += blockDim.x) {
            const float *t = P.camstat + (int64_t)cam * kCamStat + 7;
            rows[cam * kRowS + 16] = __ldg(t);
            rows[cam * kRowS + 17] = __ldg(t + 1);
        }
    }
    stage_p<float, true>(P, rows, nullptr, nullptr, beta, first, given);
}
__device__ void own_stage(const Prob &P, double *rows, double beta, bool first, const double *given) {
    if (given) {
        for (int cam = threadIdx.x; cam < P.nc; cam += blockDim.x) {
            const double *ct = P.ctr64 + (int64_t)cam * kCtr, *v = given + (int64_t)cam * kVec;
            const bool fixed = fixed_camera(P, cam);
            for (int g = 0; g < 3; ++g)
                for (int b = 0; b < 3; ++b) {
                    double x = 0.0;
                    for (int i = 0; i < 3; ++i) x = fma(__ldg(ct + 9 * g + 3 * i + b), v[3 * g + i], x);
                    rows[cam * kRowD + 3 * g + b] = fixed ? 0.0 : x;
                }
            rows[cam * kRowD + 9] = __ldg((const double *)P.camtab + (int64_t)cam * kCamTab + 24);
        }
    } else {
        const double *z = (const double *)P.zT;
        const int total = 9 * P.nc;
        for (int e = threadIdx.x; e < total; e += blockDim.x) {
            const int cam = e / 9, q = e - 9 * cam;
            const double zv = ldcg(z + (int64_t)cam * kVec + q);
            double *r = rows + cam * kRowD + q;
            *r = first ? zv : fma(beta, *r, zv);
            if (first && q == 0) r[9] = __ldg((const double *)P.camtab + (int64_t)cam * kCamTab + 24);
        }
    }
    __syncthreads();
}

// b of the slice's points: a summed over the point's lanes, b = C~^-1 a (zero for
// fixed points, also where the right-hand side of an adjoint has an entry
// there), written by the first lane of each point.
template <typename T>
__device__ __forceinline__ void own_store_b(const Prob &P, int s, int loc, const T *b, float *bs) {
    if constexpr (sizeof(T) == 4) {
        bs[loc] = b[0];
        bs[P.own_pb + loc] = b[1];
        bs[2 * P.own_pb + loc] = b[2];
    } else {
        double2 *o = (double2 *)(P.sp_b64 + 4 * (int64_t)s);
        o[0] = make_double2(b[0], b[1]);
        o[1] = make_double2(b[2], 0.0);
    }
}

struct HgObs {
    int cam;
    double v[10];  // H00 H01 H02 H11 H12 H22 g0 g1 g2 r2
};
__device__ __forceinline__ void load_hg(const double2 *hg, int64_t stride, double *v) {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double2 d = __ldg(hg + q * stride);
        v[2 * q] = d.x;
        v[2 * q + 1] = d.y;
    }
}
__device__ __forceinline__ HgObs load_hg(const Prob &P, int64_t slot) {
    HgObs o;
    o.cam = __ldg(P.sl_cam + slot);
    load_hg(P.sl_hg + slot, P.slot_cap, o.v);
    return o;
}
// The first-order branch's terms, out of line: inlined they become predicated
// instructions that occupy the FP64 pipe for every observation.
__device__ __noinline__ void small_alpha(const Prob &P, int cam, const double *X, double m0, double m1, double m2,
                                         double *al) {
    const double *w = (const double *)P.camtab + (int64_t)cam * kCamTab + 25;
    const double c0 = m1 * X[2] - m2 * X[1], c1 = m2 * X[0] - m0 * X[2], c2 = m0 * X[1] - m1 * X[0];
    al[0] -= w[1] * c2 - w[2] * c1;
    al[1] -= w[2] * c0 - w[0] * c2;
    al[2] -= w[0] * c1 - w[1] * c0;
}
__device__ __noinline__ double3 small_y(const Prob &P, int cam, double y0, double y1, double y2) {
    const double *w = (const double *)P.camtab + (int64_t)cam * kCamTab + 25;
    return make_double3(y0 + (w[1] * y2 - w[2] * y1), y1 + (w[2] * y0 - w[0] * y2), y2 + (w[0] * y1 - w[1] * y0));
}
__device__ __forceinline__ bool row_small(double flag) { return __double2hiint(flag) != 0; }
__device__ __forceinline__ void hg_alpha(const Prob &P, const double *r, int cam, const double *X, double *al) {
    const double m0 = r[0], m1 = r[1], m2 = r[2];
    al[0] = fma(m1, X[2], fma(-m2, X[1], r[3]));
    al[1] = fma(m2, X[0], fma(-m0, X[2], r[4]));
    al[2] = fma(m0, X[1], fma(-m1, X[0], r[5]));
    if (row_small(r[9])) small_alpha(P, cam, X, m0, m1, m2, al);
}
__device__ __forceinline__ void hg_u(const Prob &P, const HgObs &o, const double *r, const double *X, double *a) {
    double al[3];
    hg_alpha(P, r, o.cam, X, al);
    const double sg = fma(o.v[9], fma(o.v[9], r[8], r[7]), r[6]);
    a[0] = fma(o.v[0], al[0], fma(o.v[1], al[1], fma(o.v[2], al[2], fma(o.v[6], sg, a[0]))));
    a[1] = fma(o.v[1], al[0], fma(o.v[3], al[1], fma(o.v[4], al[2], fma(o.v[7], sg, a[1]))));
    a[2] = fma(o.v[2], al[0], fma(o.v[4], al[1], fma(o.v[5], al[2], fma(o.v[8], sg, a[2]))));
}

// The next slice of a warp: slices are sorted by decreasing length, so claiming
// them in order balances the warps (a fixed assignment left a third of the FP32
// warps' time at the barrier after the pass).  Who works a slice does not change
// its result.
__device__ __forceinline__ int claim(int *next) {
    int v = 0;
    if ((threadIdx.x & 31) == 0) v = atomicAdd(next, 1);
    return __shfl_sync(0xffffffffu, v, 0);
}

// Point pass of one block (RHS: b = C~^-1 w).
template <typename T, bool RHS>
__device__ void own_points(const Prob &P, const T *rows, float *bs, int blk, int *next) {
    const T *__restrict__ Ci = (const T *)P.Cinv;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    int w = blk + P.nblk * (threadIdx.x >> 5);
    if (w >= P.n_slices) return;
    int4 sl = __ldg(P.slice + w);
    FactStream cur;
    HgObs cur64;
    if (!RHS) {
        if constexpr (sizeof(T) == 4) cur = load_stream(P, (int64_t)sl.z + lane);
        else cur64 = load_hg(P, (int64_t)sl.z + lane);
    }
    for (;;) {
        const int wn = blk + P.nblk * claim(next);
        const int4 nx = wn < P.n_slices ? __ldg(P.slice + wn) : sl;
        const int K = sl.w & 0xffff, lg = sl.w >> 16, count = sl.y & 0xff;
        const int in = RHS ? lane : lane >> lg;
        const int s = sl.x + (in < count ? in : 0);
        T ci[6], a[3] = {T(0), T(0), T(0)}, b[3];
        if constexpr (RHS) {
            const int64_t pt = __ldg(P.sp_pt + s);
#pragma unroll
            for (int q = 0; q < 3; ++q) a[q] = (T)P.w[3 * pt + q];
        } else if constexpr (sizeof(T) == 4) {
            for (int k = 1; k <= K; ++k) {
                const FactStream c = cur;
                cur = load_stream(P, (int64_t)(k < K ? sl.z + 32 * k : nx.z) + lane);
                prefetch_l2(P.sl_px + nx.z + 32 * (k < (nx.w & 0xffff) ? k : 0) + lane);
                if (c.cam >= 0) {
                    const CamRow r = load_row((const float *)rows, nullptr, c.cam);
                    const FactObs o = fact_obs(c.px, c.py, c.iz, r);
                    float t0, t1;
                    fact_t(o, c.px, c.py, t0, t1);
                    fact_jpt(o, r, c.px, c.py, c.W * c.iz, t0, t1, (float *)a);
                }
            }
        } else {
            const double2 x01 = __ldg((const double2 *)(P.sp_X64 + 4 * (int64_t)s));
            const double X[3] = {x01.x, x01.y, __ldg(P.sp_X64 + 4 * (int64_t)s + 2)};
            for (int k = 1; k <= K; ++k) {
                const HgObs c = cur64;
                cur64 = load_hg(P, (int64_t)(k < K ? sl.z + 32 * k : nx.z) + lane);
                if (c.cam >= 0) {
                    const double2 *src = (const double2 *)((const double *)rows + c.cam * kRowD);
                    double r[10];
#pragma unroll
                    for (int q = 0; q < 5; ++q) {
                        const double2 v = src[q];
                        r[2 * q] = v.x;
                        r[2 * q + 1] = v.y;
                    }
                    hg_u(P, c, r, X, (double *)a);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) ci[q] = __ldg(Ci + (int64_t)q * P.np_pad + s);
        if (!RHS) {
            for (int d = 1; d < (1 << lg); d <<= 1) {
#pragma unroll
                for (int q = 0; q < 3; ++q) a[q] += __shfl_xor_sync(full, a[q], d);
            }
        }
        if (in < count && (RHS || (lane & ((1 << lg) - 1)) == 0)) {
            if (P.has_fixed && P.pt_fixed[P.sp_pt[s]]) a[0] = a[1] = a[2] = T(0);
            apply_sym3(ci, a[0], a[1], a[2], b);
            own_store_b<T>(P, s, (sl.y >> 8) + in, b, bs);
        }
        if (wn >= P.n_slices) return;
        w = wn;
        sl = nx;
    }
}

// The layout words of a warp's first run slice: loaded before the barrier that
// publishes b, so that their latency overlaps it.
struct RunBegin {
    int j, j0, j1;  // the warp's slice; the block's first (FP32: after the long runs) and end
    int2 rs, ln;
};
template <typename T>
__device__ __forceinline__ RunBegin own_cameras_begin(const Prob &P, int blk) {
    RunBegin rb;
    const int4 b = __ldg(P.blk_run + blk);
    rb.j0 = sizeof(T) == 4 ? b.y : b.x, rb.j1 = b.z;
    rb.j = rb.j0 + (threadIdx.x >> 5);
    rb.rs = rb.ln = make_int2(0, 0);
    if (rb.j < rb.j1) {
        rb.rs = __ldg(P.rslice + rb.j);
        rb.ln = __ldg(P.rlane + 32 * (int64_t)rb.j + (threadIdx.x & 31));
    }
    return rb;
}

// The sums over a run's G lanes into the block's row of the partials, or onto what
// the run's earlier rounds left there.
__device__ __forceinline__ void own_store_sums(const Prob &P, int2 ln, int G, bool add, float *acc) {
    for (int d = 1; d < G; d <<= 1) {
#pragma unroll
        for (int a = 0; a < 9; ++a) acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], d);
    }
    if (ln.x < 0 || (threadIdx.x & (G - 1))) return;
    float4 *o = (float4 *)((float *)P.c_part + ((int64_t)ln.y * P.nc + ln.x) * kPartF);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float4 v = make_float4(acc[4 * a], acc[4 * a + 1], acc[4 * a + 2], acc[4 * a + 3]);
        if (add) {
            const float4 u = __ldcg(o + a);
            v = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
        }
        __stcg(o + a, v);
    }
}
__device__ __forceinline__ CamConst own_cam_const(const float *rows, int cam) {
    const float *row = rows + (cam < 0 ? 0 : cam) * kRowS;
    const float4 c = ((const float4 *)row)[2], q = ((const float4 *)row)[3];
    const float2 t = ((const float2 *)row)[8];
    CamConst ct;
    ct.f = c.y, ct.k1 = c.z, ct.k2 = c.w, ct.t0 = t.x, ct.t1 = t.y;
    ct.q0 = q.x, ct.q1 = q.y, ct.q2 = q.z, ct.q3 = q.w;
    return ct;
}

// Runs of more than kRunRounds rounds (a warp each): that many rounds at a time,
// added up in the block's row, so that no FP32 sum grows longer.  In kernel
// instances of its own (LONG): its registers cost the others 2 % of an iteration.
__device__ __forceinline__ void own_long_runs(const Prob &P, const float *rows, const float *bs, int blk) {
    const int lane = threadIdx.x & 31, pb = P.own_pb;
    const int4 b = __ldg(P.blk_run + blk);
    for (int j = b.x + (threadIdx.x >> 5); j < b.y; j += blockDim.x >> 5) {
        const int2 rs = __ldg(P.rslice + j), ln = __ldg(P.rlane + 32 * (int64_t)j + lane);
        const int K = rs.y & kRunMask;
#pragma unroll 1
        for (int k0 = 0; k0 < K; k0 += kRunRounds) {
            const CamConst ct = own_cam_const(rows, ln.x);
            float acc[12];
#pragma unroll
            for (int a = 0; a < 12; ++a) acc[a] = 0.f;
            const int k1 = min(K, k0 + kRunRounds);
#pragma unroll 1
            for (int k = k0; k < k1; ++k) {
                const int64_t slot = (int64_t)rs.x + 32 * k + lane;
                const int p = __ldg(P.r_pt16 + slot);
                if (p != 0xffff)
                    fact_camera_obs(ct, __ldg(P.r_rx + slot), make_float4(bs[p], bs[pb + p], bs[2 * pb + p], 0.f),
                                    P.r_w ? __ldg(P.r_w + slot) : 1.f, acc);
            }
            own_store_sums(P, ln, 32, k0 > 0, acc);
        }
    }
}

// Camera pass of one block: every run's nine raw sums into the block's partials.
// LONG: some blocks have runs of more than kRunRounds rounds.  600 cameras, 500k
// observations, one camera with 5 % of them, against as many lanes for every run:
// FP64 338 -> 102 us per PCG iteration, FP32 35 -> 28; with 25 %, 745 -> 93 and
// 57 -> 26.
template <bool LONG>
__device__ void own_cameras(const Prob &P, const float *rows, const float *bs, int *next, const RunBegin &rb, int blk) {
    const int lane = threadIdx.x & 31;
    if constexpr (LONG) own_long_runs(P, rows, bs, blk);
    const int j1 = rb.j1, pb = P.own_pb;
    int jn = 0;
    int2 rs = rb.rs, ln = rb.ln;
    for (int j = rb.j; j < j1; j = jn) {
        jn = rb.j0 + claim(next);
        if (j != rb.j) rs = __ldg(P.rslice + j), ln = __ldg(P.rlane + 32 * (int64_t)j + lane);
        // the warp's next slice goes to L2 while this one is worked
        const int2 nx = __ldg(P.rslice + (jn < j1 ? jn : j));
        const int64_t pf = nx.x;
        const int pk = nx.y & kRunMask, K = rs.y & kRunMask;
        int64_t slot = (int64_t)rs.x + lane;
        float4 Xn = __ldg(P.r_rx + slot);
        int pn = __ldg(P.r_pt16 + slot);
        const CamConst ct = own_cam_const(rows, ln.x);
        float acc[12];
#pragma unroll
        for (int a = 0; a < 12; ++a) acc[a] = 0.f;
        for (int k = 0; k < K; ++k, slot += 32) {
            const float4 X = Xn;
            const int p = pn;
            prefetch_l2(P.r_rx + pf + 32 * (k < pk ? k : 0) + lane);
            if (k + 1 < K) {
                Xn = __ldg(P.r_rx + slot + 32);
                pn = __ldg(P.r_pt16 + slot + 32);
            }
            if (p != 0xffff)
                fact_camera_obs(ct, X, make_float4(bs[p], bs[pb + p], bs[2 * pb + p], 0.f),
                                P.r_w ? __ldg(P.r_w + slot) : 1.f, acc);
        }
        own_store_sums(P, ln, 1 << (rs.y >> kRunLg), false, acc);
    }
}
// One observation of an FP64 run: H, g, r2 and its point's X and b (b written by
// this CTA before the last barrier).
struct RunObs {
    int p;
    double h[10], X0, X1, X2, b0, b1, b2;
    __device__ __forceinline__ void load(const Prob &P, int pt, int64_t slot) {
        p = pt;
        if (p < 0) return;
        const double2 *xb = (const double2 *)(P.sp_X64 + 4 * (int64_t)p), *bb = (const double2 *)(P.sp_b64 + 4 * (int64_t)p);
        const double2 xa = __ldg(xb), ba = __ldcg(bb);
        X2 = __ldg(P.sp_X64 + 4 * (int64_t)p + 2);
        b2 = __ldcg(P.sp_b64 + 4 * (int64_t)p + 2);
        X0 = xa.x, X1 = xa.y, b0 = ba.x, b1 = ba.y;
        load_hg(P.r_hg + slot, P.rslot_cap, h);
    }
};
template <bool LONG>
__device__ void own_cameras(const Prob &P, const double *rows, const float *, int *next, const RunBegin &rb, int) {
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int j1 = rb.j1;
    int jn = 0;
    int2 rs = rb.rs, ln = rb.ln;
    for (int j = rb.j; j < j1; j = jn) {
        jn = rb.j0 + claim(next);
        if (j != rb.j) rs = __ldg(P.rslice + j), ln = __ldg(P.rlane + 32 * (int64_t)j + lane);
        const int cam = ln.x < 0 ? 0 : ln.x;
        const bool small = row_small(rows[cam * kRowD + 9]);
        double acc[10];
#pragma unroll
        for (int a = 0; a < 10; ++a) acc[a] = 0.0;
        // the next round's values are in flight while one is worked, the point
        // index another round ahead
        const int K = rs.y & kRunMask;
        int64_t slot = (int64_t)rs.x + lane;
        RunObs nxt;
        nxt.load(P, __ldg(P.r_pt + slot), slot);
        int p2 = K > 1 ? __ldg(P.r_pt + slot + 32) : -1;
        for (int k = 0; k < K; ++k, slot += 32) {
            const RunObs c = nxt;
            if (k + 1 < K) {
                nxt.load(P, p2, slot + 32);
                p2 = k + 2 < K ? __ldg(P.r_pt + slot + 64) : -1;
            }
            if (c.p < 0) continue;
            const double *h = c.h;
            const double y0 = fma(h[0], c.b0, fma(h[1], c.b1, h[2] * c.b2));
            const double y1 = fma(h[1], c.b0, fma(h[3], c.b1, h[4] * c.b2));
            const double y2 = fma(h[2], c.b0, fma(h[4], c.b1, h[5] * c.b2));
            const double q = fma(h[6], c.b0, fma(h[7], c.b1, h[8] * c.b2)), rq = h[9] * q;
            acc[3] += y0;
            acc[4] += y1;
            acc[5] += y2;
            acc[6] += q;
            acc[7] += rq;
            acc[8] = fma(h[9], rq, acc[8]);
            double v0 = y0, v1 = y1, v2 = y2;
            if (small) {  // X x (y + w x y)
                const double3 v = small_y(P, cam, y0, y1, y2);
                v0 = v.x, v1 = v.y, v2 = v.z;
            }
            acc[0] = fma(c.X1, v2, fma(-c.X2, v1, acc[0]));
            acc[1] = fma(c.X2, v0, fma(-c.X0, v2, acc[1]));
            acc[2] = fma(c.X0, v1, fma(-c.X1, v0, acc[2]));
        }
        const int G = 1 << (rs.y >> kRunLg);
        for (int d = 1; d < G; d <<= 1) {
#pragma unroll
            for (int a = 0; a < 9; ++a) acc[a] += __shfl_xor_sync(full, acc[a], d);
        }
        if (ln.x >= 0 && (lane & (G - 1)) == 0) {
            double2 *o = (double2 *)((double *)P.c_part + ((int64_t)ln.y * P.nc + ln.x) * kPartD);
#pragma unroll
            for (int a = 0; a < 5; ++a) __stcg(o + a, make_double2(acc[2 * a], acc[2 * a + 1]));
        }
    }
}

// Sum over the lanes 0..8, 9..17 and 18..26 of the same component, in every lane.
__device__ __forceinline__ double sum_thirds(double v, int a) {
    const unsigned full = 0xffffffffu;
    const double x = __shfl_sync(full, v, a), y = __shfl_sync(full, v, a + 9), z = __shfl_sync(full, v, a + 18);
    return (x + y) + z;
}

// Sums of the CTA's per-camera dot products (n values each in dots, dots +
// stride, ...), by warp 0; valid in thread 0.
__device__ __forceinline__ double own_dot_sum(const double *dots, int n) {
    double x = 0.0;
    for (int i = threadIdx.x & 31; i < n; i += 32) x += dots[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return x;
}

// The owner's vectors, nine values per camera of the CTA, in shared memory for
// the whole launch: only z's rows and the partial sums travel.
struct OwnVec {
    double *x, *r, *z, *p, *q, *s;
};

// Owner's part of a product: the cameras [cb, cb + m) of this CTA.  Groups of
// kGroup blocks' partials are added in T, the groups in FP64, in block order;
// then one warp per camera, 27 lanes: lane 9 t + a holds component a and a third
// t of every 9-term row product (the row is loaded before the partials, so that
// its latency overlaps theirs).  Modes as camera_pass; leaves the dot products in
// dots (three arrays of 9 m).
constexpr int kGroup = 16;
template <typename T, int MODE>
__device__ void own_finalize(const Prob &P, int cb, int m, const OwnVec &V, double *gsum, double *dots, double beta,
                             bool first) {
    constexpr int PS = OwnShape<T>::part;
    const T *part = (const T *)P.c_part;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    const int ng = (P.n_vblk + kGroup - 1) / kGroup, m9 = 9 * m;
    const int th = lane < 27 ? lane / 9 : 0, a = lane < 27 ? lane - 9 * th : 0;
    const double *Mat = MODE == CAM_RHS ? P.Binv : P.Bd;
    const int64_t mo = a * 9 + 3 * th;
    double r0 = 0.0, r1 = 0.0, r2 = 0.0;
    if (wid < m) {
        const double *M = Mat + 81 * (int64_t)(cb + wid) + mo;
        r0 = __ldg(M), r1 = __ldg(M + 1), r2 = __ldg(M + 2);
    }
    for (int t = threadIdx.x; t < m9 * ng; t += blockDim.x) {
        const int g = t / m9, r = t - g * m9, c = r / 9, q = r - 9 * c;
        T v[kGroup];
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
            const int blk = g * kGroup + j;
            v[j] = blk < P.n_vblk ? __ldcg(part + ((int64_t)blk * P.nc + cb + c) * PS + q) : T(0);
        }
#pragma unroll
        for (int h = kGroup / 2; h >= 1; h >>= 1)
#pragma unroll
            for (int j = 0; j < h; ++j) v[j] += v[j + h];
        gsum[t] = (double)v[0];
    }
    __syncthreads();
    for (int c = wid; c < m; c += nwarp) {
        const int cam = cb + c, vo = 9 * c + a;
        if (c != wid) {
            const double *M = Mat + 81 * (int64_t)cam + mo;
            r0 = __ldg(M), r1 = __ldg(M + 1), r2 = __ldg(M + 2);
        }
        double pv = 0.0;
        if (MODE == CAM_RHS) pv = P.v[9 * (int64_t)cam + a];
        else if (MODE == CAM_MATVEC) pv = P.p[(int64_t)cam * kVec + a];
        else if (MODE == CAM_SR) pv = V.z[vo];
        else pv = first ? V.z[vo] : fma(beta, V.p[vo], V.z[vo]);
        double s = 0.0;
        for (int g = th; g < ng; g += 3) s += gsum[g * m9 + vo];
        s = sum_thirds(s, a);
        const int g0 = a < 3 ? 0 : (a < 6 ? 3 : 6);
        double cs = 0.0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double raw = __shfl_sync(full, s, g0 + b);
            if constexpr (sizeof(T) == 4) cs = fma((double)__ldg(P.ctr + (int64_t)cam * kCtr + 3 * a + b), raw, cs);
            else cs = fma(__ldg(P.ctr64 + (int64_t)cam * kCtr + 3 * a + b), raw, cs);
        }
        if (fixed_camera(P, cam)) cs = 0.0;
        // the vector of the row product: g = v - c (right-hand side) or p
        const double x = MODE == CAM_RHS ? pv - cs : pv;
        double y = r0 * __shfl_sync(full, x, 3 * th);
        y = fma(r1, __shfl_sync(full, x, 3 * th + 1), y);
        y = fma(r2, __shfl_sync(full, x, 3 * th + 2), y);
        y = sum_thirds(y, a);
        if (MODE == CAM_RHS) {
            const T row = own_row_lane(P, cam, (T)y, 0, a);
            if (lane < 9) {
                stcg(P.g + (int64_t)cam * kVec + a, x);
                stcg((T *)P.zT + (int64_t)cam * kVec + a, row);
                V.x[vo] = 0.0;
                V.r[vo] = x;
                V.z[vo] = y;
                dots[vo] = x * x;
                dots[m9 + vo] = x * y;
            }
        } else {
            const double q = y - cs;
            if (lane < 9) {
                if (MODE == CAM_MATVEC) {
                    stcg(P.q + (int64_t)cam * kVec + a, q);
                } else if (MODE == CAM_SR) {
                    const double rv = V.r[vo];
                    V.q[vo] = q;
                    dots[vo] = rv * rv;
                    dots[m9 + vo] = rv * pv;
                    dots[2 * m9 + vo] = q * pv;
                } else {
                    V.q[vo] = q;
                    V.p[vo] = pv;
                    dots[vo] = pv * q;
                }
            }
        }
    }
    __syncthreads();
}

// z = B~^-1 r of one camera by its warp (27 lanes), r in every lane's component.
__device__ __forceinline__ double own_precond(const double *b, double rv, int th, int a) {
    const unsigned full = 0xffffffffu;
    double z = b[0] * __shfl_sync(full, rv, 3 * th);
    z = fma(b[1], __shfl_sync(full, rv, 3 * th + 1), z);
    z = fma(b[2], __shfl_sync(full, rv, 3 * th + 2), z);
    return sum_thirds(z, a);
}

// The whole solve in one cooperative launch, one CTA per SM.  Per iteration, against
// the kernel with segmented scans and a scattered s (FP32) or a stored Jacobian
// (FP64) that it replaced: FP32, 1,700 cameras and 5.0M observations 106 -> 75.5 us
// (point side 28.5, camera side 24.5: latency and issue; the streams alone take 30
// at the measured 6.8 TB/s), 200 cameras and 250k observations 21.4 -> 19.1
// (barriers and dependent sums).  FP64, 5.0M observations 747 -> 445 us (point side
// 179, camera side 224: the FP64 pipe), 780k 156 -> 105, 250k 63 -> 53, 10k
// 37 -> 18.6.
template <typename T, bool SR, bool LONG>
__global__ void __launch_bounds__(PcgBlock<T>::value, 1)
    pcg_own_kernel(Prob P, int mode, int max_iter, double tol, long long spin, int forcing) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    DevState *st = P.st;
    if (st->done || st->blockfail) return;  // a failed damping: the LM loop rejects this iteration
    __shared__ double s_g0;
    __shared__ int s_next[2];  // claim counters of the point and camera passes
    const int G = gridDim.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    if (threadIdx.x == 0) {
        s_g0 = forcing ? st->g0 : 0.0;
        s_next[0] = s_next[1] = nwarp;
    }
    uint32_t epoch = 0;
    const int cb = (int)((int64_t)blockIdx.x * P.nc / G), m = (int)((int64_t)(blockIdx.x + 1) * P.nc / G) - cb;
    const int m9 = 9 * m;
    T *rows = (T *)smem_raw;
    float *bs = (float *)(smem_raw + P.own_off_b);      // b of the block's points (FP32)
    double *gsum = (double *)(smem_raw + P.own_off_b);  // the owner's group sums, after the products of all blocks
    double *dots = (double *)(smem_raw + P.own_off_dots);
    double *part_rho = P.red, *part_rr = P.red + G, *part_pq = P.red + 2 * G;
    bool ok = true;
    auto barrier = [&]() -> bool { return grid_barrier(st, epoch, spin); };
    auto product = [&](auto rhs) {
        for (int blk = blockIdx.x; blk < P.nblk; blk += G) {
            own_points<T, decltype(rhs)::value>(P, rows, bs, blk, s_next);
            const RunBegin rb = own_cameras_begin<T>(P, blk);
            __syncthreads();
            if (threadIdx.x == 0) s_next[0] = nwarp;
            own_cameras<LONG>(P, rows, bs, s_next + 1, rb, blk);
            __syncthreads();
            if (threadIdx.x == 0) s_next[1] = nwarp;
        }
    };
    // per-CTA sums of n dot arrays into the partials
    auto publish = [&](int n, double *p0, double *p1, double *p2) {
        if (wid < n) {
            const double s = own_dot_sum(dots + wid * m9, m9);
            double *to = wid == 0 ? p0 : (wid == 1 ? p1 : p2);
            if (lane == 0) stcg(to + blockIdx.x, s);
        }
    };
    const int th = lane < 27 ? lane / 9 : 0, a = lane < 27 ? lane - 9 * th : 0;
    double *vec = dots + 3 * m9;
    const OwnVec V = {vec, vec + m9, vec + 2 * m9, vec + 3 * m9, vec + 4 * m9, vec + 5 * m9};
    // this lane's third of its row of B~^-1 for the warp's first camera (or c)
    auto load_binv = [&](int c, double *b) {
        const double *B = P.Binv + 81 * (int64_t)(cb + c) + a * 9 + 3 * th;
        b[0] = __ldg(B), b[1] = __ldg(B + 1), b[2] = __ldg(B + 2);
    };
    double binv[3] = {0.0, 0.0, 0.0};

    if (mode == PCG_MATVEC) {
        // p given in P.p (FP64): q = B~ p - E C~^-1 E^T p
        own_stage(P, rows, 0.0, true, P.p);
        product(std::false_type{});
        if (barrier()) own_finalize<T, CAM_MATVEC>(P, cb, m, V, gsum, dots, 0.0, true);
        return;
    }

    // ---- right-hand side g = v - E C~^-1 w (Eq. 3), x = 0, r = g, z = B~^-1 g ----
    // (the runs read the rows' constants, so they are staged from the zero vector first)
    own_stage(P, rows, 0.0, true, nullptr);
    product(std::true_type{});
    ok = barrier();
    if (ok) {
        own_finalize<T, CAM_RHS>(P, cb, m, V, gsum, dots, 0.0, true);
        if (mode == PCG_RHS_ONLY) return;
        publish(2, part_rr, part_rho, nullptr);
        ok = barrier();
    }
    __shared__ double s_alpha, s_beta, s_r0, s_rho, s_rn, s_stop, s_gprev, s_aprev;
    __shared__ int s_go;
    int n = 0;

    if constexpr (SR) {
        // Single-reduction recurrence; see pcg_kernel.
        while (ok && (n == 0 || n < max_iter)) {
            own_stage(P, rows, 0.0, true, nullptr);
            product(std::false_type{});
            if (!(ok = barrier())) break;
            if (wid < m) load_binv(wid, binv);
            own_finalize<T, CAM_SR>(P, cb, m, V, gsum, dots, 0.0, false);
            publish(3, part_rr, part_rho, part_pq);
            if (!(ok = barrier())) break;
            const double2 rz = sum_parts2(part_rr, part_rho, G);
            const double wu = sum_parts(part_pq, G);
            if (threadIdx.x == 0) {
                bool go;
                if (n == 0) {
                    const double r0 = sqrt(rz.x);
                    double t = tol;
                    if (forcing) {  // eta = min(0.1, sqrt(|g| / |g_first|)), |g_first| = r0 in the first solve
                        const double g0 = s_g0;
                        t = fmax(t, fmin(0.1, sqrt(r0 / (g0 > 0.0 ? g0 : r0))));
                    }
                    s_r0 = r0;
                    s_stop = (t * r0) * (t * r0);
                    go = r0 > 0.0;
                } else {
                    go = !(rz.x <= s_stop);
                }
                s_rn = sqrt(rz.x);
                go = go && isfinite(rz.y);
                const double beta = n == 0 ? 0.0 : rz.y / s_gprev;
                const double den = n == 0 ? wu : wu - beta * rz.y / s_aprev;  // p.S p
                go = go && den > 0.0 && isfinite(den);
                const double alpha = go ? rz.y / den : 0.0;
                s_gprev = rz.y;
                s_aprev = alpha;
                s_alpha = alpha;
                s_beta = beta;
                s_go = go ? 1 : 0;
            }
            __syncthreads();
            if (!s_go) break;
            const double alpha = s_alpha, beta = s_beta;
            const bool last = n + 1 >= max_iter;  // the step cap ends the solve after this update
            for (int c = wid; c < m; c += nwarp) {
                const int vo = 9 * c + a;
                if (c != wid) load_binv(c, binv);
                const double u = V.z[vo], w = V.q[vo];
                const double pn = n == 0 ? u : fma(beta, V.p[vo], u);
                const double sn = n == 0 ? w : fma(beta, V.s[vo], w);
                const double rv = fma(-alpha, sn, V.r[vo]), xv = fma(alpha, pn, V.x[vo]);
                const double z = own_precond(binv, rv, th, a);
                const T row = own_row_lane(P, cb + c, (T)z, 0, a);
                __syncwarp();
                if (lane < 9) {
                    V.p[vo] = pn;
                    V.s[vo] = sn;
                    V.x[vo] = xv;
                    V.r[vo] = rv;
                    V.z[vo] = z;
                    stcg((T *)P.zT + (int64_t)(cb + c) * kVec + a, row);
                    dots[vo] = rv * rv;
                }
            }
            ++n;
            if (last) {
                __syncthreads();
                publish(1, P.red + 3 * G, nullptr, nullptr);
                if (!(ok = barrier())) break;
                const double rrn = sum_parts(P.red + 3 * G, G);
                if (threadIdx.x == 0) s_rn = sqrt(rrn);
                __syncthreads();
                break;
            }
            if (!(ok = barrier())) break;
        }
    } else {
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
                s_rn = s0.x;
                s_stop = (t * r0) * (t * r0);
                s_go = (r0 > 0.0 && isfinite(s0.y)) ? 1 : 0;
                s_beta = 0.0;
            }
            __syncthreads();
        }
        if (ok && s_go) {
            for (;;) {
                const double beta = s_beta;
                own_stage(P, rows, beta, n == 0, nullptr);
                product(std::false_type{});
                if (!(ok = barrier())) break;
                own_finalize<T, CAM_ITER>(P, cb, m, V, gsum, dots, beta, n == 0);
                publish(1, part_pq, nullptr, nullptr);
                if (wid < m) load_binv(wid, binv);
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
                // x += alpha p; r -= alpha q; z = B~^-1 r, one warp per camera
                for (int c = wid; c < m; c += nwarp) {
                    const int vo = 9 * c + a;
                    if (c != wid) load_binv(c, binv);
                    const double xv = fma(alpha, V.p[vo], V.x[vo]), rv = fma(-alpha, V.q[vo], V.r[vo]);
                    const double z = own_precond(binv, rv, th, a);
                    const T row = own_row_lane(P, cb + c, (T)z, 0, a);
                    __syncwarp();
                    if (lane < 9) {
                        V.x[vo] = xv;
                        V.r[vo] = rv;
                        V.z[vo] = z;
                        stcg((T *)P.zT + (int64_t)(cb + c) * kVec + a, row);
                        dots[vo] = rv * rv;
                        dots[m9 + vo] = rv * z;
                    }
                }
                __syncthreads();
                publish(2, part_rr, part_rho, nullptr);
                if (!(ok = barrier())) break;
                ++n;
                const double2 sums = sum_parts2(part_rho, part_rr, G);
                if (threadIdx.x == 0) {
                    // |r| <= t |r0| as squares: a root less on every iteration's scalar chain
                    const double rho_prev = s_rho, rho = sums.x;
                    s_rho = rho;
                    s_rn = sums.y;
                    const bool go = !(sums.y <= s_stop || n >= max_iter) && isfinite(rho);
                    s_go = go ? 1 : 0;
                    s_beta = go ? rho / rho_prev : 0.0;
                }
                __syncthreads();
                if (!s_go) break;
            }
        }
    }
    if (!ok) atomicCAS(&st->err, 0, (int)MBA_ERR_TIMEOUT);
    __syncthreads();
    if (ok)
        for (int t = threadIdx.x; t < m9; t += blockDim.x) P.x[(int64_t)(cb + t / 9) * kVec + t % 9] = V.x[t];
    if (ok && blockIdx.x == 0 && threadIdx.x == 0) {
        st->pcg_iters = n;
        const double rn = SR ? s_rn : sqrt(s_rn);  // the standard loop keeps the square
        st->pcg_rel_res = s_r0 > 0.0 ? rn / s_r0 : 0.0;
        if (forcing && !(s_g0 > 0.0)) st->g0 = s_r0;
    }
}
