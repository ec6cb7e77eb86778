"""The fused step and evaluation give a QP m lanes when the batch leaves the
GPU idle otherwise, one lane when it is large or a tile is asked for.  Both
forms do the same arithmetic in the same order: poses, moments, energies,
forces, residuals and status are bitwise equal."""
import numpy as np
import pytest

from gpu_helpers import I, cuda, torch

import paper_2412_16490_gb300 as bx

pytestmark = pytest.mark.gpu

COLLISION = dict(w_pen=100.0, w_self=100.0, w_lim=10.0, eta_pen=0.005, eta_lim=0.05)


def _scene(name, B, s, grid):
    hand = I.hand_template(name)
    obj = I.grid_object(3, n=32) if grid else I.sphere_object()
    T = I.wrench_set(12)
    T = T[:s] if s <= 12 else np.concatenate([T, np.roll(0.5 * T, 1, axis=1)[:s - 12]])
    x = I.initial_poses(hand, obj, min(B, 40), seed=5)
    return bx.Hand(hand), bx.Object(obj), cuda(np.tile(x, (-(-B // 40), 1))[:B]), cuda(T)


def _step(H, Ob, x, T, sp, steps):
    st = bx.State(H, x.shape[0], T.shape[0])
    st.set_pose(x)
    E, status = torch.empty(x.shape[0], device="cuda"), torch.empty(x.shape[0], dtype=torch.int32, device="cuda")
    for n in steps:  # the second launch starts from the first one's iterates
        bx.bodex_step(H, Ob, st, T, n, sp, E_last=E, status=status)
    return [st.pose(), *st.adam()[:2], st.residual(), E, status]


@pytest.mark.parametrize("name,s,B", [("hand5", 12, 1), ("hand5", 12, 700), ("hand5", 7, 33), ("hand5", 16, 5), ("hand4", 6, 64), ("hand4x4", 12, 801),
                                      ("hand4x4", 1, 130), ("hand3", 12, 799), ("hand3", 1, 200), ("hand3", 12, 1301), ("hand5", 1, 2600)])
@pytest.mark.parametrize("cone", [0, 1])
@pytest.mark.parametrize("collide", [False, True])
def test_step_is_bitwise_the_one_lane_form(name, s, B, cone, collide):
    H, Ob, x, T = _scene(name, B, s, grid=s != 6)
    P = I.default_params(**(COLLISION if collide else {}))
    for qp in (bx.qp_params(max_iter=20, cone=cone), bx.qp_params(max_iter=60, eps_abs=1e-3, check_every=7, cone=cone)):
        wide = _step(H, Ob, x, T, bx.step_params(P, qp=qp), (3, 2))
        one = _step(H, Ob, x, T, bx.step_params(P, qp=qp, grasps_per_cta=8), (3, 2))
        for k, (a, b) in enumerate(zip(wide, one)):
            assert torch.equal(a, b), k


@pytest.mark.parametrize("name,s,B", [("hand5", 12, 50), ("hand4", 6, 90), ("hand3", 5, 77)])
@pytest.mark.parametrize("eps", [0.0, 1e-4, 1e-6])
def test_evaluation_is_bitwise_the_one_lane_form(name, s, B, eps):
    H, Ob, x, T = _scene(name, B, s, grid=True)
    qp = bx.qp_params(max_iter=400 if eps else 25, eps_abs=eps)
    outs = []
    for tile in (0, 4):
        warm = bx.State(H, B, s)
        sp = bx.step_params(I.default_params(), qp=qp, grasps_per_cta=tile)
        outs.append([bx.bodex_energy_grad(H, Ob, x, T, sp), bx.bodex_energy_grad(H, Ob, x, T, sp, warm=warm),
                     bx.bodex_energy_grad(H, Ob, x, T, sp, warm=warm)])
    for wide, one in zip(*outs):
        for k in wide:
            assert torch.equal(wide[k], one[k]), k


def test_nonfinite_pose_is_flagged_alone():
    H, Ob, x, T = _scene("hand5", 30, 12, grid=True)
    clean = _step(H, Ob, x, T, bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=20)), (2,))
    x[11, 9] = float("nan")
    out = _step(H, Ob, x, T, bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=20)), (2,))
    assert int(out[5][11]) & bx.ST_NONFINITE
    keep = [k for k in range(30) if k != 11]
    for a, b in zip(out, clean):
        assert torch.equal(a[keep], b[keep])


@pytest.mark.parametrize("name", ["hand3", "hand5"])
@pytest.mark.parametrize("tile", [0, 8])
@pytest.mark.parametrize("solver", [bx.QP_ADMM, bx.QP_EXACT])
def test_fewer_wrenches_than_contacts(name, tile, solver):
    """A QP does not depend on the other wrenches of its grasp; with fewer
    lanes than contacts every contact is still placed."""
    H, Ob, x, T = _scene(name, 37, 12, grid=True)
    sp = bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=64, solver=solver), grasps_per_cta=tile)
    full = bx.bodex_energy_grad(H, Ob, x, T, sp)
    few = bx.bodex_energy_grad(H, Ob, x, T[:2].contiguous(), sp)
    for k in ("Q", "y"):
        assert torch.equal(few[k], full[k][:, :2]), k


@pytest.mark.parametrize("cone", [0, 1])
@pytest.mark.parametrize("s", [1, 6, 12])
def test_several_jobs_in_one_wide_launch(cone, s):
    """Jobs of every contact count in one launch (few QPs: the wide form),
    bitwise as with a tile asked for (the one-lane form)."""
    scenes = [_scene(n, B, s, grid=g) for n, B, g in (("hand5", 33, True), ("hand3", 7, False), ("hand4x4", 50, True), ("hand3", 1, True))]
    outs = []
    for tile in (0, 8):
        sp = bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=20, cone=cone), grasps_per_cta=tile)
        jobs = []
        for k, (H, Ob, x, T) in enumerate(scenes):
            st = bx.State(H, x.shape[0], s)
            st.set_pose(x)
            jobs.append(dict(hand=H, obj=Ob, state=st, T=T, n_steps=3 + k, E_last=torch.empty(x.shape[0], device="cuda"),
                             status=torch.empty(x.shape[0], dtype=torch.int32, device="cuda")))
        bx.bodex_step_multi(jobs, sp)
        outs.append([t for j in jobs for t in (j["state"].pose(), *j["state"].adam()[:2], j["state"].residual(), j["E_last"], j["status"])])
    for a, b in zip(*outs):
        assert torch.equal(a, b)
