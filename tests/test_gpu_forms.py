"""Which kernel a fused step takes.  The wide form (m lanes per QP) and the
one-lane form give the same bits; the default takes the one whose estimated
time is shorter, and a requested tile the one-lane form.  The kernels that a
call launches are read from a captured graph."""
import dataclasses
import re
import warnings

import numpy as np
import pytest

from gpu_helpers import I, O, cuda, host, torch

import paper_2412_16490_gb300 as bx

pytestmark = pytest.mark.gpu

COLLISION = dict(w_pen=100.0, w_self=100.0, w_lim=10.0, eta_pen=0.005, eta_lim=0.05)


def _launched(call, tmp_path, names=r"(fused_wide_kernel|fused_kernel|multi_wide_kernel|multi_kernel)"):
    """Names of the step kernels that `call` launches."""
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g):
        call()
    path = tmp_path / "graph.dot"
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")  # the dump announces itself
        g.debug_dump(str(path))
    return re.findall(names, path.read_text())


def _scene(name, B, s):
    hand = I.hand_template(name) if isinstance(name, str) else name
    obj = I.grid_object(3, n=32)
    T = I.wrench_set(12)
    T = T[:s] if s <= 12 else np.concatenate([T, np.roll(0.5 * T, 1, axis=1)[:s - 12]])
    x = I.initial_poses(hand, obj, min(B, 40), seed=5)
    H = bx.Hand(hand)
    st = bx.State(H, B, s)
    st.set_pose(cuda(np.tile(x, (-(-B // 40), 1))[:B]))
    return dict(hand=H, obj=bx.Object(obj), state=st, T=cuda(T))


def _step(j, sp, n=1):
    bx.bodex_step(j["hand"], j["obj"], j["state"], j["T"], n, sp)


@pytest.mark.parametrize("name,s,B", [("hand5", 12, 1), ("hand5", 12, 700), ("hand5", 7, 33), ("hand5", 16, 5), ("hand4", 6, 64),
                                      ("hand4x4", 12, 801), ("hand3", 12, 799), ("hand3", 12, 1301)])
@pytest.mark.parametrize("cone", [0, 1])
@pytest.mark.parametrize("collide", [False, True])
def test_small_batches_take_the_wide_form(name, s, B, cone, collide, tmp_path):
    """The cases whose two forms test_gpu_wide compares do run in two forms."""
    P = I.default_params(**(COLLISION if collide else {}))
    j = _scene(name, B, s)
    for qp in (bx.qp_params(max_iter=20, cone=cone), bx.qp_params(max_iter=60, eps_abs=1e-3, check_every=7, cone=cone)):
        assert _launched(lambda: _step(j, bx.step_params(P, qp=qp)), tmp_path) == ["fused_wide_kernel"]
        assert _launched(lambda: _step(j, bx.step_params(P, qp=qp, grasps_per_cta=8)), tmp_path) == ["fused_kernel"]


@pytest.mark.parametrize("s", [1, 6, 12])
def test_several_small_jobs_take_the_wide_form(s, tmp_path):
    jobs = [dict(_scene(n, B, s), n_steps=1) for n, B in (("hand5", 33), ("hand3", 7), ("hand4x4", 50), ("hand3", 1))]
    for tile, kernel in ((0, "multi_wide_kernel"), (8, "multi_kernel")):
        sp = bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=20), grasps_per_cta=tile)
        assert _launched(lambda: bx.bodex_step_multi(jobs, sp), tmp_path) == [kernel]


def _outputs(j, sp, steps, multi=False):
    B = j["state"].B
    j = dict(j, E_last=torch.empty(B, device="cuda"), status=torch.empty(B, dtype=torch.int32, device="cuda"))
    x = j["state"].pose()
    for n, p in zip(steps, sp if isinstance(sp, (list, tuple)) else [sp] * len(steps)):
        if multi:
            bx.bodex_step_multi([dict(j, n_steps=n)], p)
        else:
            bx.bodex_step(j["hand"], j["obj"], j["state"], j["T"], n, p, E_last=j["E_last"], status=j["status"])
    out = [j["state"].pose(), *j["state"].adam()[:2], j["state"].residual(), j["E_last"], j["status"]]
    j["state"].set_pose(x)
    return out


@pytest.mark.parametrize("name,s,B", [("hand5", 1, 40), ("hand5", 1, 2603), ("hand5", 2, 1901), ("hand5", 4, 77), ("hand4x4", 1, 1301),
                                      ("hand4x4", 3, 1003), ("hand3", 1, 1303), ("hand3", 2, 1501)])
@pytest.mark.parametrize("cone", [0, 1])
@pytest.mark.parametrize("collide", [False, True])
def test_fewer_wrenches_than_contacts_equal_the_one_lane_form(name, s, B, cone, collide, tmp_path):
    """With s < m a step always takes the wide form, in large batches with
    several grasps a block and as few as three lanes a grasp; the several-job
    launch with a tile runs the same QPs a lane each."""
    P = I.default_params(**(COLLISION if collide else {}))
    j = _scene(name, B, s)
    for kw in (dict(max_iter=20), dict(max_iter=60, eps_abs=1e-3, check_every=7)):
        qp = bx.qp_params(cone=cone, **kw)
        wide, lane = bx.step_params(P, qp=qp), bx.step_params(P, qp=qp, grasps_per_cta=8)
        assert _launched(lambda: _step(j, wide), tmp_path) == ["fused_wide_kernel"]
        assert _launched(lambda: bx.bodex_step_multi([dict(j, n_steps=1)], lane), tmp_path) == ["multi_kernel"]
        j = _scene(name, B, s)
        for a, b in zip(_outputs(j, wide, (3, 2)), _outputs(j, lane, (3, 2), multi=True)):
            assert torch.equal(a, b)


@pytest.mark.parametrize("name,s", [("hand3", 1), ("hand3", 2), ("hand4", 3), ("hand5", 1), ("hand5", 4)])
@pytest.mark.parametrize("B", [33, 1777])
def test_evaluation_with_fewer_wrenches_matches_the_oracle(name, s, B):
    """E and dE/dx on a sphere object, every QP solved tightly (bounds as in
    the parity tests: E relative 1e-4, gradient relative 1e-3)."""
    hand, obj = I.hand_template(name), I.sphere_object()
    P = I.default_params(eps_reg=1e-3)
    x0 = I.initial_poses(hand, obj, 33, seed=7)
    T = I.wrench_set(12)[:s]
    sp = bx.step_params(P, qp=bx.qp_params(eps_abs=1e-6, eps_reg=1e-3, max_iter=20000, check_every=10))
    out = bx.bodex_energy_grad(bx.Hand(hand), bx.Object(obj), cuda(np.tile(x0, (-(-B // 33), 1))[:B]), cuda(T), sp)
    ev = O.evaluate(O.Hand(hand), O.Object(obj), x0.astype(np.float64), T, P)
    rows = np.arange(B) % 33
    ok = (host(out["status"]) & bx.ST_NOT_CONVERGED) == 0
    assert ok.mean() >= 0.9
    np.testing.assert_allclose(host(out["E"])[ok], ev["E"][rows][ok], rtol=1e-4, atol=1e-6)
    g, ref = host(out["dEdx"]), ev["grad"][rows]
    rel = np.linalg.norm(g - ref, axis=1) / np.maximum(np.linalg.norm(ref, axis=1), 1e-3)
    assert (rel[ok] <= 1e-3).all(), rel[ok].max()


@pytest.mark.parametrize("spheres", [41, 44, 48])
@pytest.mark.parametrize("B", [5, 300])
def test_collision_spheres_beyond_the_split_scratch(spheres, B, tmp_path):
    """A lane per sphere needs 6 K + 9 (n + 1) words of scratch; a hand with
    more spheres walks them by slot in the wide form too (48 spheres of the
    22-joint hand need 495 of 490)."""
    hand = I.hand_template("hand5")
    more = spheres - len(hand.sphere_link)
    pick = np.arange(more) * 5
    hand = dataclasses.replace(hand, sphere_link=np.concatenate([hand.sphere_link, hand.sphere_link[pick]]),
                               sphere_local=np.concatenate([hand.sphere_local, hand.sphere_local[pick] + np.float32(4e-3)]),
                               sphere_radius=np.concatenate([hand.sphere_radius, hand.sphere_radius[pick]]))
    P = I.default_params(**COLLISION)
    j = _scene(hand, B, 12)
    sp = [bx.step_params(P, qp=bx.qp_params(max_iter=20), grasps_per_cta=tile) for tile in (0, 8)]
    assert _launched(lambda: _step(j, sp[0]), tmp_path) == ["fused_wide_kernel"]
    j = _scene(hand, B, 12)
    for a, b in zip(*(_outputs(j, p, (3, 2)) for p in sp)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("name,s,B", [("hand5", 12, 100), ("hand3", 7, 64)])
def test_a_state_moves_between_the_forms(name, s, B):
    """The warm start of either form continues in the other."""
    j = _scene(name, B, s)
    wide, lane = (bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=20), grasps_per_cta=t) for t in (0, 8))
    outs = [_outputs(j, forms, (2, 3, 2)) for forms in ((lane, lane, lane), (wide, lane, wide), (lane, wide, lane))]
    for other in outs[1:]:
        for a, b in zip(outs[0], other):
            assert torch.equal(a, b)


def _times(calls, reps=9):
    """Shortest time of each call in ms, the calls taken in turn."""
    best = [float("inf")] * len(calls)
    for r in range(reps):
        for k, (reset, call) in enumerate(calls):
            reset()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            if r:
                best[k] = min(best[k], a.elapsed_time(b))
    return best


# sizes around the second wave of either form, at few wrenches and many, few iterations and many;
# the shorter of the two estimates is at most some 10% from the faster form
@pytest.mark.parametrize("name,s,B,cone,iters,collide", [
    ("hand5", 16, 893, 0, 20, False), ("hand5", 16, 893, 0, 50, False), ("hand5", 5, 2857, 0, 20, False),
    ("hand5", 16, 1653, 1, 3, False), ("hand5", 8, 3306, 1, 3, False), ("hand4x4", 8, 4218, 1, 3, False),
    ("hand5", 16, 893, 1, 3, True), ("hand3", 12, 1216, 0, 300, True), ("hand4x4", 12, 1500, 0, 50, True),
    ("hand3", 16, 720, 0, 150, False), ("hand5", 12, 1000, 0, 50, False), ("hand3", 12, 400, 0, 50, False),
])
def test_default_form_is_not_the_slower_one(name, s, B, cone, iters, collide):
    sp = [bx.step_params(I.default_params(**(COLLISION if collide else {})), qp=bx.qp_params(max_iter=iters, cone=cone),
                         grasps_per_cta=tile) for tile in (0, 96 // s)]
    j = _scene(name, B, s)
    x = j["state"].pose()
    auto, lane = _times([(lambda: j["state"].set_pose(x), lambda p=p: _step(j, p, 8)) for p in sp])
    assert auto <= 1.15 * lane, (auto, lane)


@pytest.mark.parametrize("mix,s,collide", [((("hand5", 900),), 16, False), ((("hand3", 1400),), 12, True),
                                           ((("hand5", 400), ("hand3", 400), ("hand4x4", 400)) * 2, 6, True),
                                           ((("hand5", 140), ("hand3", 140), ("hand4x4", 140)) * 2, 16, False)])
def test_default_form_of_several_jobs_is_not_the_slower_one(mix, s, collide):
    P = I.default_params(**(COLLISION if collide else {}))
    jobs = [dict(_scene(n, B, s), n_steps=8) for n, B in mix]
    xs = [j["state"].pose() for j in jobs]

    def reset():
        for j, x in zip(jobs, xs):
            j["state"].set_pose(x)

    sp = [bx.step_params(P, qp=bx.qp_params(max_iter=20), grasps_per_cta=tile) for tile in (0, 96 // s)]
    auto, lane = _times([(reset, lambda p=p: bx.bodex_step_multi(jobs, p)) for p in sp])
    assert auto <= 1.15 * lane, (auto, lane)


MIX = ("hand5", "hand5", "hand4x4", "hand4x4", "hand3")


@pytest.mark.parametrize("names", [MIX, ("hand5", "hand3"), ("hand3", "hand4x4", "hand5") * 2])
@pytest.mark.parametrize("total", [1000, 3000, 4864, 5700, 6500, 9000])
def test_several_jobs_with_exact_qps_take_no_longer_than_their_widest_hand(names, total):
    """Several contact counts with exact QPs in one launch: the SMs run one
    count's code each (1.0 to 1.3 times one hand's job of as many grasps when
    this was written; up to 2.7 times with three counts' code on every SM)."""
    sp = bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=64, solver=bx.QP_EXACT))
    calls = []
    for group in (names, ("hand5",)):
        jobs = [dict(_scene(n, total // len(group), 12), n_steps=5) for n in group]
        xs = [j["state"].pose() for j in jobs]

        def reset(jobs=jobs, xs=xs):
            for j, x in zip(jobs, xs):
                j["state"].set_pose(x)

        calls.append((reset, lambda jobs=jobs: bx.bodex_step_multi(jobs, sp)))
    mixed, one = _times(calls, reps=5)
    assert mixed <= 1.6 * one, (mixed, one)


@pytest.mark.parametrize("sizes", [(40, 30, 20), (900, 700, 803), (1500, 1300, 1207), (2100, 1800, 1701), (2600, 2500, 2401)])
@pytest.mark.parametrize("order", [("hand3", "hand5", "hand4x4"), ("hand4x4", "hand3", "hand5")])
def test_exact_items_in_any_order_equal_the_jobs_alone(sizes, order):
    """Up to, at and beyond the sizes whose items are laid out by SM, last
    tiles partial: each job as in its own launch."""
    sp = bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=64, solver=bx.QP_EXACT))
    jobs = [_scene(n, B, 12) for n, B in zip(order, sizes)]
    alone = [_outputs(j, sp, (2,)) for j in jobs]
    for j in jobs:
        B = j["state"].B
        j.update(n_steps=2, E_last=torch.empty(B, device="cuda"), status=torch.empty(B, dtype=torch.int32, device="cuda"))
    bx.bodex_step_multi(jobs, sp)
    for j, want in zip(jobs, alone):
        for a, b in zip([j["state"].pose(), *j["state"].adam()[:2], j["state"].residual(), j["E_last"], j["status"]], want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("cone", [0, 1])
@pytest.mark.parametrize("few", [("hand5", 1), ("hand5", 2), ("hand3", 1), ("hand4x4", 1), ("hand4x4", 2)])
@pytest.mark.parametrize("tile", [0, 1, 3])
def test_adaptive_jobs_with_threads_beyond_their_grasps(few, tile, cone):
    """Several jobs with adaptive rho in blocks of 96 threads: where shared
    memory or a requested tile leaves a job fewer grasps a block than its
    wrenches would, the threads beyond them have no record to read (that read
    was out of bounds).  Each job as with full blocks, or alone."""
    qp = bx.qp_params(max_iter=60, eps_abs=1e-3, check_every=7, adaptive_rho=1, cone=cone)
    sizes = (("hand5", 5, 40), ("hand3", 12, 33), (*few, 165))
    outs = []
    for t, group in ((tile, sizes), (0, sizes[:2])):
        sp = bx.step_params(I.default_params(), qp=qp, grasps_per_cta=t)
        jobs = [dict(_scene(n, B, s), n_steps=3, E_last=torch.empty(B, device="cuda"),
                     status=torch.empty(B, dtype=torch.int32, device="cuda")) for n, s, B in group]
        bx.bodex_step_multi(jobs, sp)
        outs.append([[j["state"].pose(), *j["state"].adam()[:2], j["state"].residual(), j["E_last"], j["status"]] for j in jobs])
    alone = _outputs(_scene(few[0], 165, few[1]), bx.step_params(I.default_params(), qp=qp), (3,))
    for got, want in zip(outs[0], [*outs[1], alone]):
        for a, b in zip(got, want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("cone", [0, 1])
@pytest.mark.parametrize("few", [("hand5", 4), ("hand3", 2), ("hand4x4", 1)])
@pytest.mark.parametrize("adapt", [0, 1])
def test_jobs_alone_and_beside_one_of_few_wrenches(few, cone, adapt, tmp_path):
    """Several jobs run in a kernel without the loop over contacts, unless one
    has fewer wrenches than contacts; the same bits."""
    sp = bx.step_params(I.default_params(), grasps_per_cta=8,
                        qp=bx.qp_params(max_iter=60, eps_abs=1e-3, check_every=7, adaptive_rho=adapt, cone=cone))
    names = (("hand5", 5, 201), ("hand3", 3, 33), ("hand4x4", 12, 803), ("hand5", 12, 8))
    kernels, outs = [], []
    for extra in ((), ((*few, 65),)):
        jobs = []
        for n, s, B in names + extra:
            jobs.append(dict(_scene(n, B, s), n_steps=3, E_last=torch.empty(B, device="cuda"),
                             status=torch.empty(B, dtype=torch.int32, device="cuda")))
        bx.bodex_step_multi(jobs, sp)
        outs.append([a for j in jobs[:4] for a in (j["state"].pose(), *j["state"].adam()[:2], j["state"].residual(),
                                                   j["E_last"], j["status"])])
        (kernel,) = _launched(lambda: bx.bodex_step_multi(jobs, sp), tmp_path, r"multi_kernel[\w<>, ]*")
        kernels.append(kernel)
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    assert kernels[0] != kernels[1]


@pytest.mark.parametrize("names,s,total,cone,iters,steps", [
    (("hand5", "hand5", "hand5", "hand3"), 8, 4050, 1, 40, (4,)), (("hand5", "hand5", "hand5", "hand3"), 8, 4400, 1, 40, (4,)),
    (("hand5", "hand5", "hand5", "hand3"), 12, 4700, 0, 30, (2, 8, 5)), (("hand5", "hand5", "hand5", "hand3"), 8, 3150, 0, 30, (2, 8, 5))])
def test_unequal_jobs_do_not_take_the_slower_form(names, s, total, cone, iters, steps):
    """The one-lane form's last wave is the cheap job's alone; the wide form's
    waves drift apart where the jobs' steps differ."""
    jobs = [dict(_scene(n, total // len(names), s), n_steps=steps[i % len(steps)]) for i, n in enumerate(names)]
    xs = [j["state"].pose() for j in jobs]

    def reset():
        for j, x in zip(jobs, xs):
            j["state"].set_pose(x)

    sp = [bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=iters, cone=cone), grasps_per_cta=tile) for tile in (0, 96 // s)]
    auto, lane = _times([(reset, lambda p=p: bx.bodex_step_multi(jobs, p)) for p in sp])
    assert auto <= 1.15 * lane, (auto, lane)
