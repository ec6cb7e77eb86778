"""The refinement and the contact metrics run with a warp or with eight lanes
per grasp, by the samples, the batch and the object.  Both forms find the
sample with the smallest phi, lowest index on ties, at any sample count."""
import dataclasses
import re
import warnings

import numpy as np
import pytest

from gpu_helpers import I, O, cuda, host, torch

import paper_2412_16490_gb300 as bx

pytestmark = pytest.mark.gpu

BIG = 16401  # eight lanes for few samples, 16 grasps a block, the last one partial


def _case(name, kind, S, B=41):
    hand = I.hand_template(name)
    obj = I.grid_object(2, n=32) if kind == "grid" else I.sphere_object()
    tips = np.concatenate([hand.tip_samples] * 4, axis=1)
    rng = np.random.default_rng(S)
    tips = np.ascontiguousarray((tips + rng.normal(scale=1e-3, size=tips.shape))[:, :S].astype(np.float32))
    x = I.initial_poses(hand, obj, B, seed=12, gap=(-0.01, 0.005), flex=0.8)
    return dataclasses.replace(hand, tip_samples=tips), obj, x


def _refine(H, Ob, x, pc, steps):
    B = x.shape[0]
    st = bx.State(H, B, 1)
    st.set_pose(x)
    E, k = torch.empty(B, device="cuda"), torch.empty((B, H.m), dtype=torch.int32, device="cuda")
    status = torch.empty(B, dtype=torch.int32, device="cuda")
    bx.bodex_refine(H, Ob, st, pc, steps, 0.01, 300.0, bx.step_params(I.default_params()), E_last=E, kstar=k, status=status)
    return [st.pose(), *st.adam()[:2], E, k, status]


@pytest.mark.parametrize("name", ["hand3", "hand4x4", "hand5"])
@pytest.mark.parametrize("kind", ["grid", "sphere"])
@pytest.mark.parametrize("S", [1, 7, 12, 31, 33, 64])
def test_samples_of_any_count_match_the_oracle_and_the_other_form(name, kind, S):
    hand, obj, x0 = _case(name, kind, S)
    H, Ob = bx.Hand(hand), bx.Object(obj)
    x = cuda(x0)
    pc = bx.bodex_fk_contacts(H, Ob, x)["p"]
    small = _refine(H, Ob, x, pc, 1)
    ref = O.refine_eval(O.Hand(hand), O.Object(obj), x0.astype(np.float64), host(pc).astype(np.float64), 0.01,
                        I.default_params()["w_d"], 300.0)
    clear = ref["gap"] >= 1e-6 if S > 1 else np.ones(ref["kstar"].shape, bool)
    assert (host(small[4])[clear] == ref["kstar"][clear]).all()
    met = bx.bodex_contact_metrics(H, Ob, x)
    want = O.contact_metrics(O.Hand(hand), O.Object(obj), x0.astype(np.float64))
    np.testing.assert_allclose(host(met["d"]), want["d"], rtol=0, atol=2e-6)
    # the same poses in a batch that fills the GPU
    n = x.shape[0]
    rep = lambda t: t.repeat(-(-BIG // n), *([1] * (t.dim() - 1)))[:BIG].contiguous()
    small = _refine(H, Ob, x, pc, 3)
    big = _refine(H, Ob, rep(x), rep(pc), 3)
    for a, b in zip(small, big):
        assert torch.equal(rep(a), b)
    mb = bx.bodex_contact_metrics(H, Ob, rep(x))
    for k in ("d", "cdc"):
        assert torch.equal(rep(met[k]), mb[k])


@pytest.mark.parametrize("kind", ["grid", "sphere"])
@pytest.mark.parametrize("half", [4, 8, 16, 24, 32])
def test_equal_samples_give_the_lowest_index(kind, half):
    """Every sample twice, `half` apart: on other lanes of the warp and, from
    32 on, in another round of the same lane."""
    hand, obj, x0 = _case("hand5", kind, half)
    twice = dataclasses.replace(hand, tip_samples=np.ascontiguousarray(np.concatenate([hand.tip_samples] * 2, axis=1)))
    Ob = bx.Object(obj)
    H1, H2 = bx.Hand(hand), bx.Hand(twice)
    x = cuda(x0)
    pc = bx.bodex_fk_contacts(H1, Ob, x)["p"]
    for B in (x.shape[0], BIG):
        xb, pb = (t.repeat(-(-B // x.shape[0]), *([1] * (t.dim() - 1)))[:B].contiguous() for t in (x, pc))
        for a, b in zip(_refine(H1, Ob, xb, pb, 2), _refine(H2, Ob, xb, pb, 2)):
            assert torch.equal(a, b)
        assert torch.equal(bx.bodex_contact_metrics(H1, Ob, xb)["d"], bx.bodex_contact_metrics(H2, Ob, xb)["d"])


def test_few_samples_cost_less_than_many():
    """A large batch on a sphere object: a step with one sample a finger takes
    a fraction of the time of one with 64 (0.37 when this was written; 0.87
    with a warp per grasp)."""
    ms = []
    for S in (1, 64):
        hand, obj, x0 = _case("hand5", "sphere", S)
        H, Ob = bx.Hand(hand), bx.Object(obj)
        x = cuda(np.tile(x0, (400, 1)))
        pc = bx.bodex_fk_contacts(H, Ob, x)["p"]
        st = bx.State(H, x.shape[0], 1)
        st.set_pose(x)
        sp, best = bx.step_params(I.default_params()), float("inf")
        for r in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            bx.bodex_refine(H, Ob, st, pc, 100, 0.01, 300.0, sp)
            b.record()
            torch.cuda.synchronize()
            if r:
                best = min(best, a.elapsed_time(b))
        ms.append(best)
    assert ms[0] <= 0.6 * ms[1], ms


@pytest.mark.parametrize("metrics,name,S,B,lanes", [(False, "hand4", 10, 5000, 8), (False, "hand5", 10, 5000, 8), (False, "hand5", 10, 3500, 32),
                                                    (False, "hand3", 20, 10000, 32), (False, "hand3", 20, 20000, 32),
                                                    (True, "hand3", 20, 28000, 32), (True, "hand4", 20, 14000, 32), (True, "hand5", 10, 28000, 8)])
def test_the_faster_form_near_the_crossings(metrics, name, S, B, lanes, tmp_path):
    """Lanes a grasp of the launched kernel where one form was 5 to 30% faster."""
    hand, obj, x0 = _case(name, "grid", S)
    H, Ob = bx.Hand(hand), bx.Object(obj)
    x = cuda(np.tile(x0, (-(-B // len(x0)), 1))[:B])
    pc = bx.bodex_fk_contacts(H, Ob, x)["p"]
    st, sp = bx.State(H, B, 1), bx.step_params(I.default_params())
    st.set_pose(x)
    call = (lambda: bx.bodex_contact_metrics(H, Ob, x)) if metrics else (lambda: bx.bodex_refine(H, Ob, st, pc, 1, 0.01, 300.0, sp))
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g):
        call()
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")  # the dump announces itself
        g.debug_dump(str(tmp_path / "graph.dot"))
    launched = re.findall(r"(?:refine|metrics)_kernel(?:I|<)(?:Li)?\d(?:E|, *)(?:Li)?(\d+)", (tmp_path / "graph.dot").read_text())
    assert launched == [str(lanes)]
