"""The Schur products' layouts at the sizes where they change: lanes per point
and rounds of the sliced point order, the block-owned product and its runs
(few cameras: split runs), the gathered FP32 product and the stored FP64 one
where the camera rows do not fit in shared memory, the first-order rotation
branch, and the batched windows' clusters, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_close
from scenes import make_scene, make_windows

pytestmark = pytest.mark.gpu

# (cameras, points, track): one point; one and two lanes per point; tracks around
# one and two warps; few cameras with long runs (split into parts); cameras
# around the 128 that stop the splitting; rows beyond shared memory
SHAPES = {
    "one-point": (2, 1, ("fixed", 2)),
    "few-points": (3, 33, ("fixed", 3)),
    "tracks-32-33": (40, 70, ("fixed", 33)),
    "tracks-17": (40, 300, ("fixed", 17)),
    "mixed-long": (70, 400, ("lognormal", 20.0, 70)),
    "split-runs": (5, 9000, ("geom", 0.4)),
    "cams-127": (127, 5000, ("geom", 0.25)),
    "cams-129": (129, 40_000, ("geom", 0.25)),
    "rows-in-L2": (2500, 30_000, ("geom", 0.25)),
}


@pytest.fixture(scope="module")
def mba():
    from paper_2112_01349_gb300 import _build, mba as m

    _build.build()
    m.load()
    return m


def _scene(shape, seed=7):
    nc, npts, track = SHAPES[shape]
    return make_scene(nc, npts, track=track, sigma=0.5, seed=seed, outlier_frac=0.02 if npts > 1 else 0.0)


def _args(sc):
    return sc.cameras, sc.points, sc.observations, sc.cam_idx, sc.pt_idx


@pytest.mark.parametrize("loss", ["none", "huber"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-4)])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_product_and_step(mba, shape, precision, tol, loss):
    """One Schur product and one damped step.  Tolerances: the ones these entry
    points have elsewhere (products 1e-9 / 1e-4; steps of a few PCG iterations 1e-6 / 2e-3)."""
    sc = _scene(shape)
    x = np.random.default_rng(5).normal(size=(sc.nc, 9))
    mu = 0.1
    with mba.Problem(*_args(sc), precision=precision, loss=loss, huber_delta=2.0 if loss == "huber" else 0.0) as pr:
        y = pr.schur_matvec(mu, x)
        ls = pr.linear_system(mu)
        st = pr.step(mu, pcg_max_iter=6, pcg_rel_tol=0.0)
        so = pr.solve(max_iter=2, pcg_max_iter=6, initial_radius=10.0)
    ref = oracle.schur(*_args(sc), mu, x=x.reshape(-1), loss=loss, delta=2.0)
    rel_close(y, ref["y"].reshape(-1, 9), tol, "S x")
    rel_close(ls["rhs"], ref["rhs"].reshape(-1, 9), 10 * tol, "rhs")
    rs = oracle.step(*_args(sc), mu, pcg_max=6, pcg_tol=0.0, loss=loss, delta=2.0)
    stol = 1e-6 if precision == "fp64" else 2e-3
    for a in range(9):  # per parameter: the blocks differ in scale by orders
        rel_close(st["dc"][:, a], rs["dc"].reshape(-1, 9)[:, a], stol, f"dc[{a}]")
    rel_close(st["dp"], rs["dp"].reshape(-1, 3), stol, "dp")
    if 2 * sc.n < 9 * sc.nc + 3 * sc.np_:
        return  # underdetermined: the cost goes to zero, below what FP32 residuals resolve
    rl = oracle.lm_solve(*_args(sc), max_iter=2, pcg_max=6, initial_radius=10.0, loss=loss, delta=2.0)
    rel_close(so["final_cost"], rl["final_cost"], 1e-6 if precision == "fp64" else 1e-4, "final cost")


@pytest.mark.parametrize("jacobian", ["analytic", "autodiff"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-6), ("fp32", 2e-3)])
@pytest.mark.parametrize("per_camera", [31, 32, 33, 255, 256, 257, 513])
def test_schur_jacobi_chunk_edges(mba, per_camera, precision, tol, jacobian):
    """The Schur-Jacobi blocks of cameras with observations around a warp and
    around a chunk of 256.  Tolerances: those of a step of a few PCG iterations."""
    sc = make_scene(2, per_camera, track=("fixed", 2), sigma=0.5, seed=11)
    with mba.Problem(*_args(sc), precision=precision, jacobian=jacobian) as pr:
        st = pr.step(0.1, pcg_max_iter=4, pcg_rel_tol=0.0, preconditioner="schur_jacobi")
    rs = oracle.step(*_args(sc), 0.1, pcg_max=4, pcg_tol=0.0, precond="schur_jacobi")
    for a in range(9):
        rel_close(st["dc"][:, a], rs["dc"].reshape(-1, 9)[:, a], tol, f"dc[{a}]")
    rel_close(st["dp"], rs["dp"].reshape(-1, 3), tol, "dp")


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-4)])
@pytest.mark.parametrize("shape", ["cams-127", "rows-in-L2"])
def test_first_order_rotations_and_fixed_nodes(mba, shape, precision, tol):
    """Cameras on the first-order rotation branch (|w|^2 <= DBL_EPSILON, w not
    zero) beside ordinary ones, and fixed nodes in the product."""
    sc = _scene(shape)
    cams = sc.cameras.copy()
    cams[::5, :3] = np.random.default_rng(1).normal(size=cams[::5, :3].shape) * 4e-9
    cams[::5, 3:6] = [0.0, 0.0, -8.0]
    args = (cams, *_args(sc)[1:])
    rng = np.random.default_rng(2)
    x = rng.normal(size=(sc.nc, 9))
    mu = 0.1
    with mba.Problem(*args, precision=precision) as pr:
        y = pr.schur_matvec(mu, x)
        cf, pf = rng.random(sc.nc) < 0.2, rng.random(sc.np_) < 0.2
        pr.set_fixed(cf, pf)
        st = pr.step(mu, pcg_max_iter=6, pcg_rel_tol=0.0)
    rel_close(y, oracle.schur(*args, mu, x=x.reshape(-1))["y"].reshape(-1, 9), tol, "S x")
    rs = oracle.step(*args, mu, pcg_max=6, pcg_tol=0.0, cam_fixed=cf, pt_fixed=pf)
    rel_close(st["dc"], rs["dc"].reshape(-1, 9), 1e-6 if precision == "fp64" else 2e-3, "dc")
    assert np.all(st["dc"][cf] == 0.0) and np.all(st["dp"][pf] == 0.0)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-3)])
@pytest.mark.parametrize("count,cams", [(1, (2, 64)), (3, (5, 30)), (9, (5, 30)), (38, (3, 12)), (80, (3, 9))])
def test_clusters_agree_with_one_cta_per_window(mba, count, cams, precision, tol):
    """The automatic schedule (a cluster of CTAs per window; 16 down to 2 ranks
    with the number of windows) against one CTA per window, forward and adjoint."""
    ws = make_windows(count, seed=count, cams=cams, pts=(20, 400))
    tup = [_args(w) for w in ws]
    rng = np.random.default_rng(3)
    out = []
    for auto in (True, False):
        with mba.Batch(tup, precision=precision) as b:
            if not auto:
                b.set_schedule(256, 1, "explicit")
            gc, gp = rng.normal(size=(b.info["nc"], 9)), rng.normal(size=(b.info["np"], 3))
            rng = np.random.default_rng(3)
            r = b.solve(gc if auto else g0[0], gp if auto else g0[1], adjoint_mu=0.3, adjoint_pcg_max_iter=20,
                        max_iter=3, pcg_max_iter=15, initial_radius=10.0)
            g0 = (gc, gp) if auto else g0
            g = b.gradients()
            again = None
            if auto:
                b.reset()
                b.solve(gc, gp, adjoint_mu=0.3, adjoint_pcg_max_iter=20, max_iter=3, pcg_max_iter=15, initial_radius=10.0)
                again = b.parameters()
            out.append((r["summaries"], b.parameters(), g))
            if again is not None:
                np.testing.assert_array_equal(again[0], out[0][1][0])
    (s1, p1, g1), (s2, p2, g2) = out
    assert [s["accepted"] for s in s1] == [s["accepted"] for s in s2]
    rel_close([s["final_cost"] for s in s1], [s["final_cost"] for s in s2], tol, "final costs")
    rel_close(p1[0], p2[0], tol, "cameras")
    rel_close(p1[1], p2[1], tol, "points")
    for k in ("grad_obs", "grad_init_cam", "grad_init_pt"):
        rel_close(g1[k], g2[k], 100 * tol if precision == "fp64" else 3e-2, k)


@pytest.mark.parametrize("loss", ["none", "huber"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-4)])
@pytest.mark.parametrize("nc,npts", [(40, 9000), (300, 60_000), (300, 200_000)])
def test_a_camera_that_sees_every_point(mba, nc, npts, precision, tol, loss):
    """One camera with far longer runs than the others: a warp per run, and (FP32)
    runs of more than 32 rounds.  The layout does not grow with the longest run: a
    block pads one slice of 32 slots to at most 32 rounds (84 bytes per slot in
    FP64, 152 blocks).  Tolerances as above."""
    plain = make_scene(nc, npts, track=("fixed", 2), sigma=0.5, seed=9)
    # the first observation of every point not yet seen by camera 0 moves there
    cam = plain.cam_idx.copy()
    _, first = np.unique(plain.pt_idx, return_index=True)
    seen = np.zeros(npts, bool)
    seen[plain.pt_idx[cam == 0]] = True
    move = first[~seen]
    cam[move] = 0
    assert np.bincount(cam, minlength=nc).min() > 0
    true = oracle.evaluate(plain.cameras_true, plain.points_true, np.zeros((plain.n, 2)), cam, plain.pt_idx,
                           jacobians=False)[1]
    uv = true + np.random.default_rng(4).normal(size=true.shape)
    args = (plain.cameras, plain.points, uv, cam, plain.pt_idx)
    x = np.random.default_rng(5).normal(size=(nc, 9))
    opts = dict(precision=precision, loss=loss, huber_delta=2.0 if loss == "huber" else 0.0)
    with mba.Problem(*_args(plain), **opts) as pr:
        size = pr.info["device_bytes"]
    with mba.Problem(*args, **opts) as pr:
        assert pr.info["device_bytes"] < 1.1 * size + 152 * 32 * 32 * 84
        y = pr.schur_matvec(0.1, x)
        steps = {v: pr.step(0.1, pcg_max_iter=6, pcg_rel_tol=0.0, pcg_variant=v) for v in ("standard", "single_reduction")}
    rel_close(y, oracle.schur(*args, 0.1, x=x.reshape(-1), loss=loss, delta=2.0)["y"].reshape(-1, 9), tol, "S x")
    stol = 1e-6 if precision == "fp64" else 2e-3
    for variant, st in steps.items():
        rs = oracle.step(*args, 0.1, pcg_max=6, pcg_tol=0.0, loss=loss, delta=2.0, pcg_variant=variant)
        for a in range(9):
            rel_close(st["dc"][:, a], rs["dc"].reshape(-1, 9)[:, a], stol, f"{variant} dc[{a}]")
        rel_close(st["dp"], rs["dp"].reshape(-1, 3), stol, f"{variant} dp")


# b of a CTA's points beside the camera rows in shared memory: two, three and four
# blocks per CTA, two with split runs, and more points than four can hold (gathered)
@pytest.mark.parametrize("nc,npts,track,loss", [(2000, 900_000, 2, "none"), (2000, 1_600_000, 2, "huber"),
                                                (1824, 3_000_000, 1, "none"), (100, 3_000_000, 1, "huber"),
                                                (2290, 480_000, 3, "huber")])
def test_blocks_per_cta(mba, nc, npts, track, loss):
    """Tolerances as above."""
    sc = make_scene(nc, npts, track=("fixed", track), sigma=0.5, seed=12)
    x = np.random.default_rng(5).normal(size=(nc, 9))
    with mba.Problem(*_args(sc), precision="fp32", loss=loss, huber_delta=2.0 if loss == "huber" else 0.0) as pr:
        y = pr.schur_matvec(0.1, x)
        st = pr.step(0.1, pcg_max_iter=4, pcg_rel_tol=0.0)
        f = pr.solve(max_iter=1, pcg_max_iter=4, initial_radius=10.0)["final_cost"]
    rel_close(y, oracle.schur(*_args(sc), 0.1, x=x.reshape(-1), loss=loss, delta=2.0)["y"].reshape(-1, 9), 1e-4, "S x")
    rs = oracle.step(*_args(sc), 0.1, pcg_max=4, pcg_tol=0.0, loss=loss, delta=2.0)
    for a in range(9):
        rel_close(st["dc"][:, a], rs["dc"].reshape(-1, 9)[:, a], 2e-3, f"dc[{a}]")
    rel_close(st["dp"], rs["dp"].reshape(-1, 3), 2e-3, "dp")
    ref = oracle.lm_solve(*_args(sc), max_iter=1, pcg_max=4, initial_radius=10.0, loss=loss, delta=2.0)
    rel_close(f, ref["final_cost"], 1e-4, "final cost")


@pytest.mark.parametrize("loss", ["none", "huber"])
@pytest.mark.parametrize("nc,npts,first_order", [(16, 2000, False), (127, 5000, False), (127, 5000, True)])
def test_camera_blocks_fp64(mba, nc, npts, first_order, loss):
    """B of the block-owned FP64 form, entry by entry against the geometric mean of
    its diagonal entries: a dozen roundings per observation, sums of at most 8 in a
    lane, five levels of lanes and a few chunks, and two 3 x 3 transforms, here and
    in the oracle: 100 units of 2^-53 at most."""
    sc = make_scene(nc, npts, track=("fixed", 5), sigma=0.5, seed=13)
    cams = sc.cameras.copy()
    if first_order:
        cams[::2, :3] = np.random.default_rng(1).normal(size=cams[::2, :3].shape) * 4e-9
        cams[1::4, :3] = 0.0
        cams[:, 3:6] = [0.0, 0.0, -8.0]
    args = (cams, *_args(sc)[1:])
    with mba.Problem(*args, precision="fp64", loss=loss, huber_delta=2.0 if loss == "huber" else 0.0) as pr:
        got = pr.linear_system(0.1)["Hpp"]
    ref = oracle.blocks(*args, loss=loss, delta=2.0)[0]
    d = np.sqrt(np.einsum("iaa->ia", ref))
    assert np.max(np.abs(got - ref) / (d[:, :, None] * d[:, None, :])) < 100 * 2.0**-53


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-4)])
@pytest.mark.parametrize("nc,npts", [(2, 30), (127, 5000), (2500, 30_000)])
def test_cameras_without_rotation(mba, nc, npts, precision, tol):
    """All cameras at w = 0 exactly, where the first-order and the general branch of
    the rotation agree: no first-order terms.  Tolerances as above."""
    sc = make_scene(nc, npts, track=("fixed", min(nc, 5)), sigma=0.5, seed=14)
    cams = sc.cameras.copy()
    cams[:, :3] = 0.0
    cams[:, 3:6] = [0.0, 0.0, -8.0]
    args = (cams, *_args(sc)[1:])
    x = np.random.default_rng(5).normal(size=(nc, 9))
    with mba.Problem(*args, precision=precision) as pr:
        _, e, jc, jp = pr.evaluate()
        y = pr.schur_matvec(0.1, x)
        st = pr.step(0.1, pcg_max_iter=6, pcg_rel_tol=0.0)
    _, eo, jco, jpo, _ = oracle.evaluate(*args)
    for got, ref in ((e, eo), (jc, jco), (jp, jpo)):
        rel_close(got, ref, tol, "evaluate")
    rel_close(y, oracle.schur(*args, 0.1, x=x.reshape(-1))["y"].reshape(-1, 9), tol, "S x")
    rs = oracle.step(*args, 0.1, pcg_max=6, pcg_tol=0.0)
    rel_close(st["dc"], rs["dc"].reshape(-1, 9), 1e-6 if precision == "fp64" else 2e-3, "dc")
