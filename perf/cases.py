"""The bundle-adjustment calls whose time matters, as measurable cases.

Each case is a call (or the few calls) that a program makes again and again on
a problem it holds: LM solves from a tiny calibration scene to a
Final-13682-shaped reconstruction, batches of sliding windows, the
differentiable layer forward and backward, one damped step and one Schur
product for programs that run their own outer loop.  Scenes follow the recipe
of ``scenes/generate.py`` (cameras on a circle of radius 8, points in a unit
cube, uniform visibility, pixel noise, perturbed initial estimate), drawn on
the GPU from the seed.

``exact`` restates the solver in 64-bit torch operations: BAL projection,
IRLS, Schur complement, block-Jacobi or Schur-Jacobi PCG, Levenberg-Marquardt
with Nielsen's radius rule, and the implicit-function adjoint.

The FP32-mixed form computes steps in 32 bits, so its results are taken as
float32 arrays, as a network or a renderer that consumes them would.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_01349_gb300 import mba
from paper_2112_01349_gb300.layer import ba_layer

LOGNORMAL_CAP = 300
# mu with E[min(cap, 2 + floor(exp(N(mu, 1))))] = 6.5, the workloads' mean track
LOGNORMAL_MU = 1.10991


def listed():
    return [
        # a calibration rig or an AR anchor: the smallest solves, where launches and barriers count
        dict(name="tiny-solve-fp64", kind="solve", nc=16, npts=2000, track="fixed5", precision="fp64",
             lm=5, pcg=30),
        # a few sliding windows of one robot, solved with gradients for a learned front end
        dict(name="windows8-fp64-adjoint", kind="batch", windows=8, precision="fp64", lm=4, pcg=30, adjoint=True),
        # the sliding windows of a fleet or of a dataset, re-solved every frame
        dict(name="windows512-fp32", kind="batch", windows=512, precision="fp32", lm=3, pcg=30, adjoint=False),
        # a local map of a SLAM back end
        dict(name="local-map-fp32", kind="solve", nc=200, npts=50_000, track="geom", precision="fp32", lm=4, pcg=30),
        # the differentiable layer inside a training step: problem set-up, solve, adjoint
        dict(name="layer-fp64", kind="layer", nc=200, npts=50_000, track="geom", precision="fp64", lm=4, pcg=30),
        # a photo collection with outliers and long tracks: robust loss, the faster preconditioner, inexact steps
        dict(name="collection-fp32-huber", kind="solve", nc=601, npts=150_001, track="lognormal", precision="fp32",
             lm=5, pcg=100, huber=True, precond="schur_jacobi", forcing=True),
        # dual-number Jacobians, the path of user-defined edges
        dict(name="autodiff-fp32", kind="solve", nc=340, npts=200_000, track="geom", precision="fp32", lm=3, pcg=30,
             jacobian="autodiff"),
        # one damped step of a program that runs its own trust region
        dict(name="step-fp64", kind="step", nc=503, npts=120_001, track="lognormal", precision="fp64", pcg=30),
        # one reduced-system product of a program that runs its own Krylov method
        dict(name="matvec-fp32", kind="matvec", nc=1201, npts=700_003, track="geom", precision="fp32"),
        # the paper's Venice-1778 shape in both precisions
        dict(name="venice-fp32", kind="solve", nc=1700, npts=1_000_000, track="geom", precision="fp32", lm=4, pcg=50),
        dict(name="venice-fp64", kind="solve", nc=1700, npts=1_000_000, track="geom", precision="fp64", lm=3, pcg=30),
        # the paper's Final-13682 shape: the largest
        dict(name="final-fp32-huber", kind="solve", nc=13_000, npts=4_500_000, track="lognormal", precision="fp32",
             lm=2, pcg=24, huber=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "layer", "step", "matvec"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "batch":
        return dict(kind=kind, windows=log_int(4, 512), precision=precision, lm=rng.randint(2, 4), pcg=30,
                    adjoint=rng.random() < 0.5)
    top = 60_000 if kind == "layer" else 300_000 if precision == "fp64" else 1_000_000
    npts = log_int(1_500, top)
    nc = max(8, min(npts // 60, log_int(10, 3_000)))
    case = dict(kind=kind, nc=nc, npts=npts, track=rng.choice(["geom", "geom", "lognormal", "fixed5"]),
                precision=precision)
    if kind == "matvec":
        return case
    case["pcg"] = rng.randint(20, 40)
    if kind == "step":
        return case
    case["lm"] = rng.randint(2, 4)
    if kind == "solve":
        case["huber"] = rng.random() < 0.3
        if rng.random() < 0.25:
            case["precond"] = "schur_jacobi"
        case["forcing"] = rng.random() < 0.25
        if rng.random() < 0.2:
            case["jacobian"] = "autodiff"
    return case


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _skew(w):
    o = torch.zeros_like(w[:, 0])
    return torch.stack([torch.stack([o, -w[:, 2], w[:, 1]], 1), torch.stack([w[:, 2], o, -w[:, 0]], 1),
                        torch.stack([-w[:, 1], w[:, 0], o], 1)], 1)


def _rotation(w):
    """Rotation matrices of angle-axis vectors (Rodrigues; first order at zero)."""
    th2 = (w * w).sum(1)
    small = th2 <= torch.finfo(torch.float64).eps
    th = torch.sqrt(torch.where(small, torch.ones_like(th2), th2))
    K = _skew(w)
    eye = torch.eye(3, dtype=w.dtype, device=w.device)
    a, b = torch.sin(th) / th, (1 - torch.cos(th)) / (th * th)
    R = eye + a[:, None, None] * K + b[:, None, None] * (K @ K)
    return torch.where(small[:, None, None], eye + K, R), small, torch.where(small, torch.ones_like(th2), th2)


def _circle_cameras(index, count):
    """Angle-axis and translation of camera ``index`` of ``count`` on the circle, looking at the origin."""
    phi = 2 * math.pi * index.double() / count.double()
    s, c, o = torch.sin(phi), torch.cos(phi), torch.zeros_like(phi)
    one = torch.ones_like(phi)
    R = torch.stack([torch.stack([-s, c, o], 1), torch.stack([o, o, one], 1), torch.stack([c, s, o], 1)], 1)
    # quaternion of a rotation matrix as the leading eigenvector of its 4x4 form
    Q = torch.zeros(len(phi), 4, 4, dtype=torch.float64, device=phi.device)
    Q[:, 0, 0] = R[:, 0, 0] - R[:, 1, 1] - R[:, 2, 2]
    Q[:, 1, 1] = R[:, 1, 1] - R[:, 0, 0] - R[:, 2, 2]
    Q[:, 2, 2] = R[:, 2, 2] - R[:, 0, 0] - R[:, 1, 1]
    Q[:, 3, 3] = R[:, 0, 0] + R[:, 1, 1] + R[:, 2, 2]
    for i, j, v in ((0, 1, R[:, 0, 1] + R[:, 1, 0]), (0, 2, R[:, 0, 2] + R[:, 2, 0]), (1, 2, R[:, 1, 2] + R[:, 2, 1]),
                    (0, 3, R[:, 2, 1] - R[:, 1, 2]), (1, 3, R[:, 0, 2] - R[:, 2, 0]), (2, 3, R[:, 1, 0] - R[:, 0, 1])):
        Q[:, i, j] = v
        Q[:, j, i] = v
    q = torch.linalg.eigh(Q.cpu() / 3)[1][:, :, 3].to(phi.device)
    q = q * torch.where(q[:, 3:] < 0, -1.0, 1.0)
    n = q[:, :3].norm(dim=1)
    w = q[:, :3] * (2 * torch.atan2(n, q[:, 3]) / n.clamp_min(1e-300))[:, None]
    t = -(R @ torch.stack([8 * c, 8 * s, o], 1)[:, :, None])[:, :, 0]
    return w, t


def _pixels(cams, pts, ci, pi):
    R = _rotation(cams[:, :3])[0]
    P = (R[ci] @ pts[pi][:, :, None])[:, :, 0] + cams[ci, 3:6]
    p = -P[:, :2] / P[:, 2:]
    r2 = (p * p).sum(1)
    return (cams[ci, 6] * (1 + cams[ci, 7] * r2 + cams[ci, 8] * r2 * r2))[:, None] * p


def _lengths(track, u, z, cap):
    if track == "fixed5":
        L = torch.full_like(u, 5.0)
    elif track == "lognormal":
        L = 2 + torch.floor(torch.exp(LOGNORMAL_MU + z))
    else:  # 1 + geometric, mean 5 (geom) or 4 (window)
        L = 1 + torch.ceil(torch.log1p(-u) / math.log1p(-(0.25 if track == "geom" else 1.0 / 3.0))).clamp_min(1)
    return torch.minimum(L.clamp_max(LOGNORMAL_CAP), cap.double()).long()


def _scene(case, seed):
    """Inputs on the device: cams, pts, uv, camera and point index, window of each camera and point."""
    dev = _dev()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))

    shape = torch.Generator(device=dev)  # window sizes and track lengths belong to the case, not to the seed
    shape.manual_seed(20)

    def rand(*s, by=g):
        return torch.rand(*s, generator=by, device=dev, dtype=torch.float64)

    def randn(*s, by=g):
        return torch.randn(*s, generator=by, device=dev, dtype=torch.float64)

    if case["kind"] == "batch":
        nw = case["windows"]
        ncw, npw = 5 + (rand(nw, by=shape) * 26).long(), 200 + (rand(nw, by=shape) * 2801).long()
        track = "window"
    else:
        ncw, npw = (torch.tensor([case[k]], device=dev) for k in ("nc", "npts"))
        track = case["track"]
    cw = torch.repeat_interleave(torch.arange(len(ncw), device=dev), ncw)
    pw = torch.repeat_interleave(torch.arange(len(npw), device=dev), npw)
    coff, poff = torch.cumsum(ncw, 0) - ncw, torch.cumsum(npw, 0) - npw
    local = torch.arange(len(cw), device=dev) - coff[cw]
    w, t = _circle_cameras(local, ncw[cw])
    intr = torch.cat([500 + 1000 * rand(len(cw), 1), 0.01 * randn(len(cw), 2)], 1)
    true = torch.cat([w, t, intr], 1)
    X = rand(len(pw), 3) - 0.5
    L = _lengths(track, rand(len(pw), by=shape), randn(len(pw), by=shape), ncw[pw])
    first = torch.arange(len(pw), device=dev) - poff[pw]
    most = int(ncw.max())
    if most <= 64:  # distinct cameras by ranking random keys; the first points cover every camera
        keys = rand(len(pw), most)
        keys[torch.arange(most, device=dev)[None, :] >= ncw[pw][:, None]] = 2.0
        cover = first < ncw[pw]
        keys[cover.nonzero()[:, 0], first[cover]] = -1.0
        order = torch.argsort(keys, 1)
        mask = torch.arange(most, device=dev)[None, :] < L[:, None]
        ci, pi = order[mask], mask.nonzero()[:, 0]
    else:  # draws, those that repeat a (camera, point) pair drawn again; the first points cover every camera
        nc = int(ncw[0])
        pi = torch.repeat_interleave(torch.arange(len(pw), device=dev), L)
        ci = (rand(len(pi)) * nc).long()
        cover = first < nc
        ci[(torch.cumsum(L, 0) - L)[cover]] = first[cover]
        while True:
            key, order = torch.sort(pi * nc + ci, stable=True)
            again = order[1:][key[1:] == key[:-1]]
            if len(again) == 0:
                break
            ci[again] = (rand(len(again)) * nc).long()
    perm = torch.argsort(rand(len(ci)))
    if case["kind"] == "batch":  # windows stay contiguous, shuffled inside
        perm = perm[torch.argsort(pw[pi[perm]], stable=True)]
    ci, pi = ci[perm], pi[perm]
    gi = ci + coff[pw[pi]]
    uv = _pixels(true, X, gi, pi) + randn(len(ci), 2)
    if case.get("huber"):
        out = rand(len(ci)) < 0.01
        ang = 2 * math.pi * rand(len(ci))
        uv = uv + 50.0 * out[:, None] * torch.stack([torch.cos(ang), torch.sin(ang)], 1)
    cams = true.clone()
    cams[:, :3] += 0.01 * randn(len(cw), 3)
    cams[:, 3:6] *= 1 + 0.02 * randn(len(cw), 3)
    pts = X + 0.02 * randn(len(pw), 3)
    extra = (randn(len(cw), 9), randn(len(pw), 3))
    return dict(cams=cams, pts=pts, uv=uv, ci=gi, ci_local=ci, pi=pi, cw=cw, pw=pw, extra=extra,
                offsets=(ncw, npw, torch.bincount(pw[pi], minlength=len(ncw))))


def _host(t, dtype=np.float64):
    return np.ascontiguousarray(t.cpu().numpy(), dtype=dtype)


def _radius(case):
    """Initial trust region: the default in 64 bits, a tighter one (as for a map that is
    already close, or a network's estimate) where the steps are computed in 32."""
    return 1e4 if case["precision"] == "fp64" else 10.0


def _solver(case):
    o = dict(max_iter=case.get("lm", 1), pcg_max_iter=case["pcg"], pcg_rel_tol=1e-10,
             initial_radius=_radius(case))
    if case.get("precond"):
        o["preconditioner"] = case["precond"]
    if case.get("forcing"):
        o["forcing"] = True
    return o


def _step_mu(case):
    """The damping that a trust region passes to a single step or product."""
    return 1e-3 if case["precision"] == "fp64" else 0.1


def _adjoint_mu(case):
    """Proximal weight of the adjoint."""
    return 1e-2 if case["precision"] == "fp64" else 0.3


def prepare(case, seed):
    sc = _scene(case, seed)
    kind = case["kind"]
    if kind == "layer":  # a network's outputs: tensors on the GPU that ask for gradients
        leaf = {k: sc[k].clone().requires_grad_(True) for k in ("uv", "cams", "pts")}
        return dict(case=case, leaf=leaf, ci=sc["ci"].int(), pi=sc["pi"].int(), seeds=sc["extra"])
    cams, pts, uv = _host(sc["cams"]), _host(sc["pts"]), _host(sc["uv"])
    ci, pi = _host(sc["ci_local"], np.int32), _host(sc["pi"], np.int32)
    if kind == "batch":
        nc, npt, n = (np.concatenate([[0], np.cumsum(_host(o, np.int64))]) for o in sc["offsets"])
        windows = [(cams[nc[k]:nc[k + 1]], pts[npt[k]:npt[k + 1]], uv[n[k]:n[k + 1]], ci[n[k]:n[k + 1]],
                    pi[n[k]:n[k + 1]] - np.int32(npt[k])) for k in range(case["windows"])]
        state = dict(case=case, batch=mba.Batch(windows, precision=case["precision"]))
        if case["adjoint"]:
            state["grads"] = tuple(_host(e) for e in sc["extra"])
        return state
    pr = mba.Problem(cams, pts, uv, ci, pi, precision=case["precision"],
                     loss="huber" if case.get("huber") else "none", huber_delta=2.0 if case.get("huber") else 0.0,
                     jacobian=case.get("jacobian", "analytic"))
    return dict(case=case, problem=pr, x=_host(sc["extra"][0]))


def run(state):
    case = state["case"]
    kind = case["kind"]
    result = np.float32 if case["precision"] == "fp32" else np.float64
    if kind == "layer":
        leaf = state["leaf"]
        cams, pts = ba_layer(leaf["uv"], leaf["cams"], leaf["pts"], state["ci"], state["pi"],
                             precision=case["precision"], adjoint_mu=_adjoint_mu(case), adjoint_pcg_max_iter=case["pcg"],
                             **_solver(case))
        grads = torch.autograd.grad((cams, pts), (leaf["uv"], leaf["cams"], leaf["pts"]), state["seeds"])
        out = (cams.detach(), pts.detach(), *grads)
        return list(out) if result is np.float64 else [o.float() for o in out]
    if kind == "batch":
        b = state["batch"]
        b.reset()
        if case["adjoint"]:
            b.solve(*state["grads"], adjoint_pcg_max_iter=case["pcg"], adjoint_mu=_adjoint_mu(case), **_solver(case))
            g = b.gradients()
            out = [*b.parameters(), g["grad_obs"], g["grad_init_cam"], g["grad_init_pt"]]
        else:
            b.solve(**_solver(case))
            out = [*b.parameters()]
        return [o.astype(result, copy=False) for o in out]
    pr = state["problem"]
    if kind == "solve":
        pr.reset()
        s = pr.solve(**_solver(case))
        cams, pts = pr.parameters()
        return [cams.astype(result, copy=False), pts.astype(result, copy=False), result(s["final_cost"])]
    if kind == "step":
        r = pr.step(_step_mu(case), **_solver(case))
        return [r["dc"].astype(result, copy=False), r["dp"].astype(result, copy=False), result(r["model_dec"])]
    return [pr.schur_matvec(_step_mu(case), state["x"]).astype(result, copy=False)]


def _sizes(case):
    """Cameras, points and observations (expected where the scene draws them)."""
    if case["kind"] == "batch":
        return 17.5 * case["windows"], 1600.0 * case["windows"], 6200.0 * case["windows"]
    mean = {"fixed5": 5.0, "geom": 5.0, "lognormal": 6.5}[case["track"]]
    return float(case["nc"]), float(case["npts"]), case["npts"] * min(mean, 0.6 * case["nc"])


def work(case):
    """Each input read once and each result written once; operations of the
    method: per observation about 450 for the linearisation and 96 per Schur
    product (Jc p, Jp^T t, Jp b, Jc^T s), per camera 162 twice per product."""
    nc, npt, n = _sizes(case)
    kind = case["kind"]
    w = 4 if case["precision"] == "fp32" else 8
    nbytes = n * (16 + 8) + 8 * (9 * nc + 3 * npt)
    lm = case.get("lm", 1)
    products = {"matvec": 1, "step": case.get("pcg", 0)}.get(kind, lm * case.get("pcg", 0))
    if case.get("forcing"):
        products = lm * 8
    out = w * (9 * nc + (0 if kind == "matvec" else 3 * npt))
    if kind == "layer" or case.get("adjoint"):
        out += w * (2 * n + 9 * nc + 3 * npt)
        products += case["pcg"]
    return {"bytes": nbytes + out, "flops": lm * n * 450.0 + products * (96.0 * n + 18.0 * npt + 324.0 * nc)}


# ---------------------------------------------------------------------------
# the same computation in 64-bit torch operations
# ---------------------------------------------------------------------------
def _sum_by(index, values, count):
    out = torch.zeros((count, *values.shape[1:]), dtype=values.dtype, device=values.device)
    return out.index_add_(0, index, values)


def _loss(s, huber):
    if not huber:
        return s, torch.ones_like(s)
    far, r = s > 4.0, torch.sqrt(s.clamp_min(4.0))
    return torch.where(far, 4.0 * r - 4.0, s), torch.where(far, 2.0 / r, torch.ones_like(s))


class _Exact:
    """Every window of a scene at once (a single problem is one window)."""

    def __init__(self, sc, huber):
        self.sc, self.huber = sc, huber
        order = torch.argsort(sc["ci"], stable=True)  # camera-major: the camera sums become prefix differences
        self.order, self.ci, self.pi, self.uv = order, sc["ci"][order], sc["pi"][order], sc["uv"][order]
        self.cw, self.pw = sc["cw"], sc["pw"]
        self.nc, self.npt, self.nw = len(self.cw), len(self.pw), len(sc["offsets"][0])
        # camera sums in two levels (runs of 64 observations, then cameras): few additions meet at one address
        count = torch.bincount(self.ci, minlength=self.nc)
        runs = (count + 63) // 64
        place = torch.arange(len(self.ci), device=self.ci.device) - (torch.cumsum(count, 0) - count)[self.ci]
        self.run_of = (torch.cumsum(runs, 0) - runs)[self.ci] + place // 64
        self.run_cam = torch.repeat_interleave(torch.arange(self.nc, device=self.ci.device), runs)

    def window_sum(self, index, v):
        return _sum_by(index, v, self.nw)

    def camera_sum(self, v):
        return _sum_by(self.run_cam, _sum_by(self.run_of, v, len(self.run_cam)), self.nc)

    def cost(self, cams, pts):
        e = _pixels(cams, pts, self.ci, self.pi) - self.uv
        return 0.5 * self.window_sum(self.cw, self.camera_sum(_loss((e * e).sum(1), self.huber)[0]))

    def linearise(self, cams, pts):
        ci = self.ci
        R, small, th2 = _rotation(cams[:, :3])
        w, eye = cams[:, :3], torch.eye(3, dtype=cams.dtype, device=cams.device)
        K = _skew(w)
        dR = []
        for k in range(3):  # derivative of the exponential map (Gallego and Yezzi, 2015)
            col = torch.linalg.cross(w, (eye - R)[:, :, k], dim=1)
            d = ((w[:, k, None, None] * K + _skew(col)) @ R) / th2[:, None, None]
            dR.append(torch.where(small[:, None, None], _skew(eye[k].expand_as(w)), d))
        X = pts[self.pi]
        P = (R[ci] @ X[:, :, None])[:, :, 0] + cams[ci, 3:6]
        iz = 1 / P[:, 2]
        p = -P[:, :2] * iz[:, None]
        r2 = (p * p).sum(1)
        f, k1, k2 = cams[ci, 6], cams[ci, 7], cams[ci, 8]
        d = 1 + k1 * r2 + k2 * r2 * r2
        e = (f * d)[:, None] * p - self.uv
        A = (f * (2 * k1 + 4 * k2 * r2))[:, None, None] * p[:, :, None] * p[:, None, :]
        A = A + (f * d)[:, None, None] * torch.eye(2, dtype=p.dtype, device=p.device)
        proj = torch.cat([torch.eye(2, dtype=p.dtype, device=p.device).expand(len(p), 2, 2), p[:, :, None]], 2)
        D = -(A @ proj) * iz[:, None, None]
        dPdw = torch.stack([(m[ci] @ X[:, :, None])[:, :, 0] for m in dR], 2)
        intr = torch.stack([d[:, None] * p, (f * r2)[:, None] * p, (f * r2 * r2)[:, None] * p], 2)
        Jc, Jp = torch.cat([D @ dPdw, D, intr], 2), D @ R[ci]
        self.sw = torch.sqrt(_loss((e * e).sum(1), self.huber)[1])
        self.Jc, self.Jp, self.e = Jc * self.sw[:, None, None], Jp * self.sw[:, None, None], e * self.sw[:, None]
        self.B = self.camera_sum(self.Jc.transpose(1, 2) @ self.Jc)
        self.C = _sum_by(self.pi, self.Jp.transpose(1, 2) @ self.Jp, self.npt)
        self.v = -self.camera_sum((self.Jc * self.e[:, :, None]).sum(1))
        self.w = -_sum_by(self.pi, (self.Jp * self.e[:, :, None]).sum(1), self.npt)

    def damp(self, mu, precond):
        self.Dc = self.B.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32)
        self.Dp = self.C.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32)
        self.Bd = self.B + torch.diag_embed(mu[self.cw][:, None] * self.Dc)
        self.Ci = torch.linalg.inv(self.C + torch.diag_embed(mu[self.pw][:, None] * self.Dp))
        M = self.Bd
        if precond == "schur_jacobi":
            F = self.Jc.transpose(1, 2) @ (self.Jp @ self.Ci[self.pi] @ self.Jp.transpose(1, 2)) @ self.Jc
            M = self.Bd - self.camera_sum(F)
        self.M = torch.linalg.inv(M)

    def couple_t(self, p):  # E^T p
        t = (self.Jc * p[self.ci][:, None, :]).sum(2)
        return _sum_by(self.pi, (self.Jp * t[:, :, None]).sum(1), self.npt)

    def couple(self, b):  # E b
        s = (self.Jp * b[self.pi][:, None, :]).sum(2)
        return self.camera_sum((self.Jc * s[:, :, None]).sum(1))

    def apply(self, M, x):
        return (M @ x[:, :, None])[:, :, 0]

    def product(self, p):
        return self.apply(self.Bd, p) - self.couple(self.apply(self.Ci, self.couple_t(p)))

    def dot(self, a, b):
        return self.window_sum(self.cw, (a * b).sum(1))

    def pcg(self, most, tol, first_norm=None):
        r = self.v - self.couple(self.apply(self.Ci, self.w))
        x, z = torch.zeros_like(r), self.apply(self.M, r)
        p, rho, r0 = z, self.dot(r, z), torch.sqrt(self.dot(r, r))
        self.g_norm = r0
        if first_norm is not None:
            g1 = torch.where(first_norm > 0, first_norm, r0)
            tol = torch.clamp(torch.sqrt(r0 / g1), max=0.1).clamp_min(tol)
        go = r0 > 0
        for _ in range(most):
            if not bool(go.any()):
                break
            q = self.product(p)
            pq = self.dot(p, q)
            go = go & (pq > 0)
            a = torch.where(go, rho / pq, torch.zeros_like(pq))[self.cw][:, None]
            x, r = x + a * p, r - a * q
            z = self.apply(self.M, r)
            rn, new = torch.sqrt(self.dot(r, r)), self.dot(r, z)
            go = go & (rn > tol * r0)
            p = z + torch.where(go, new / rho, torch.zeros_like(rho))[self.cw][:, None] * p
            rho = torch.where(go, new, rho)
        return x, self.apply(self.Ci, self.w - self.couple_t(x))

    def model_decrease(self, dc, dp):
        d = (self.Jc @ dc[self.ci][:, :, None])[:, :, 0] + (self.Jp @ dp[self.pi][:, :, None])[:, :, 0]
        return self.window_sum(self.cw, self.camera_sum(-(self.e * d).sum(1) - 0.5 * (d * d).sum(1)))

    def solve(self, case):
        cams, pts = self.sc["cams"].clone(), self.sc["pts"].clone()
        one = torch.ones(self.nw, dtype=torch.float64, device=cams.device)
        radius, factor, F, g1 = _radius(case) * one, 2 * one, self.cost(cams, pts), 0 * one
        for _ in range(case["lm"]):
            self.linearise(cams, pts)
            self.damp(1 / radius, case.get("precond"))
            dc, dp = self.pcg(case["pcg"], 1e-10, g1 if case.get("forcing") else None)
            g1 = torch.where(g1 > 0, g1, self.g_norm)
            L, Fn = self.model_decrease(dc, dp), self.cost(cams + dc, pts + dp)
            gain = (F - Fn) / L
            ok = (L > 0) & torch.isfinite(Fn) & (gain > 1e-3)
            grown = radius / torch.clamp(1 - (2 * gain - 1) ** 3, min=1 / 3)
            radius = torch.where(ok, grown, radius / factor).clamp(1e-32, 1e16)
            factor = torch.where(ok, 2 * one, 2 * factor)
            cams = torch.where(ok[self.cw][:, None], cams + dc, cams)
            pts = torch.where(ok[self.pw][:, None], pts + dp, pts)
            F = torch.where(ok, Fn, F)
        return cams, pts, F

    def adjoint(self, cams, pts, gc, gp, case):
        weight = _adjoint_mu(case)
        mu = torch.full((self.nw,), weight, dtype=torch.float64, device=cams.device)
        self.linearise(cams, pts)
        self.damp(mu, None)
        self.v, self.w = gc, gp
        vc, vp = self.pcg(case["pcg"], 1e-12)
        d = (self.Jc @ vc[self.ci][:, :, None])[:, :, 0] + (self.Jp @ vp[self.pi][:, :, None])[:, :, 0]
        go = torch.empty_like(d)
        go[self.order] = self.sw[:, None] * d
        return go, weight * self.Dc * vc, weight * self.Dp * vp


def exact(case, seed):
    sc = _scene(case, seed)
    ex = _Exact(sc, bool(case.get("huber")))
    kind = case["kind"]
    if kind in ("step", "matvec"):
        ex.linearise(sc["cams"], sc["pts"])
        ex.damp(torch.full((1,), _step_mu(case), dtype=torch.float64, device=sc["cams"].device), None)
        if kind == "matvec":
            return [ex.product(sc["extra"][0])]
        dc, dp = ex.pcg(case["pcg"], 1e-10)
        return [dc, dp, ex.model_decrease(dc, dp)[0]]
    cams, pts, F = ex.solve(case)
    if kind == "solve":
        return [cams, pts, F[0]]
    if kind == "batch" and not case["adjoint"]:
        return [cams, pts]
    return [cams, pts, *ex.adjoint(cams, pts, *sc["extra"], case)]
