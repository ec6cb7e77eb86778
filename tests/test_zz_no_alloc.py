"""The allocation-free step, bodex_step_noalloc, against the allocating one.

Some callers cannot allocate device memory while they run -- a real-time
robot controller that reserves all of its memory at start-up so its loop has
bounded latency, or a process whose memory pool owns the device.  For them
the library keeps the per-grasp optimiser state (Adam moments, ADMM warm
starts) in a fixed array of its own instead of a bodex_state_t.  This test
calls that entry point through the C ABI twice in a row, on different
poses, and checks each result against bodex_state_set_pose + bodex_step on
the same inputs: the second call also shows that the array's leftovers from
the first call do not leak into the next one.  Free device memory is read
(cudaMemGetInfo) around that second call: once the first call has loaded the
library's code and array onto the device, a call allocates nothing.  It also
checks that a batch larger than the array is refused before any device work.

This file is collected last (test_zz_*) so that a run stopping at its first
failure has already run every other test.
"""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import bodex_inputs as I  # noqa: E402
import paper_2412_16490_gb300 as bx  # noqa: E402
from paper_2412_16490_gb300 import _binding  # noqa: E402

pytestmark = pytest.mark.gpu


def _ptr(t):
    return C.c_void_p(t.data_ptr()) if t is not None else None


def _reference(H, Ob, x, T, n_steps, sp):
    st = bx.State(H, x.shape[0], T.shape[0])
    st.set_pose(x)
    E = torch.empty(x.shape[0], device="cuda")
    bx.bodex_step(H, Ob, st, T, n_steps, sp, E_last=E)
    return st.pose(), E


def test_noalloc_step_matches_allocating_step_on_two_calls():
    lib = bx.load()
    hand, obj, x0, T, P, _, _ = I.workload("tiny")
    H, Ob = bx.Hand(hand), bx.Object(obj)
    sp = bx.step_params(P, qp=bx.qp_params(max_iter=30))
    Tt = torch.as_tensor(T).cuda()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for first, n_steps in ((0, 5), (16, 7)):  # two calls in a row, different poses
        x = torch.as_tensor(x0[first:first + 48]).cuda()
        want_x, want_E = _reference(H, Ob, x.clone(), Tt, n_steps, sp)
        got_x = x.clone()
        got_E = torch.empty(48, device="cuda")
        status = torch.empty(48, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        rc = lib.bodex_step_noalloc(H.handle, Ob.handle, _ptr(got_x), 48, _ptr(Tt), T.shape[0], n_steps,
                                    C.byref(sp), _ptr(got_E), _ptr(status), stream)
        assert rc == _binding.BODEX_OK, lib.bodex_last_error()
        torch.cuda.synchronize()
        if first:  # the second call, after the first loaded the code and the array: no device memory taken
            assert torch.cuda.mem_get_info()[0] == free0
        np.testing.assert_allclose(got_x.cpu().numpy(), want_x.cpu().numpy(), atol=1e-6)
        np.testing.assert_allclose(got_E.cpu().numpy(), want_E.cpu().numpy(), rtol=1e-5, atol=1e-7)
        assert (status.cpu().numpy() & bx.ST_NONFINITE == 0).all()


def test_noalloc_step_refuses_batches_beyond_its_array():
    lib = bx.load()
    hand, obj, x0, T, P, _, _ = I.workload("tiny", batch=2)
    H, Ob = bx.Hand(hand), bx.Object(obj)
    sp = bx.step_params(P)
    Tt = torch.as_tensor(T).cuda()
    big = 1 << 20  # far beyond 4 MiB of per-grasp state; no device work is issued
    x = torch.zeros((1, hand.dof), device="cuda")
    rc = lib.bodex_step_noalloc(H.handle, Ob.handle, _ptr(x), big, _ptr(Tt), T.shape[0], 1, C.byref(sp), None,
                                None, C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == _binding.BODEX_ERR_INVALID
    assert b"scratch" in lib.bodex_last_error()


LAZY = """
import ctypes as C, sys
import numpy as np, torch
import bodex_inputs as I
import paper_2412_16490_gb300 as bx
lib = bx.load()
ptr = lambda t: C.c_void_p(t.data_ptr())
hand, obj = I.hand_template(sys.argv[1]), I.grid_object(3, n=32)
H, Ob = bx.Hand(hand), bx.Object(obj)
x = torch.as_tensor(np.tile(I.initial_poses(hand, obj, 40, seed=5), (40, 1)).astype(np.float32)).cuda()
T = torch.as_tensor(I.wrench_set(12).astype(np.float32)).cuda()
E, status = torch.empty(1600, device="cuda"), torch.empty(1600, dtype=torch.int32, device="cuda")
P = I.default_params()
coll = dict(P, w_pen=100.0, w_self=100.0, w_lim=10.0, eta_pen=0.005, eta_lim=0.05)

def taken(B, s, P, tile=0, **qp):
    sp = bx.step_params(P, qp=bx.qp_params(max_iter=20, **qp), grasps_per_cta=tile)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    rc = lib.bodex_step_noalloc(H.handle, Ob.handle, ptr(x), B, ptr(T), s, 2, C.byref(sp), ptr(E), ptr(status),
                                C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.bodex_last_error()
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]

taken(4, 12, P)  # the warm-up
calls = [(4, 12, P, {}), (1300, 12, P, {}), (4, 12, P, dict(tile=4)), (4, 2, P, {}), (4, 12, P, dict(cone=1)), (1300, 12, P, dict(cone=1, tile=4)),
         (4, 12, P, dict(solver=bx.QP_EXACT)), (4, 12, coll, {}), (700, 12, coll, dict(tile=4))]
for cone in (0, 1):
    for s in (2, 12):
        calls += [(30, s, P, dict(cone=cone, eps_abs=1e-4, adaptive_rho=1)), (30, s, dict(P, energy=bx.ENERGY_DFC), dict(cone=cone))]
got = [taken(B, s, Q, **kw) for B, s, Q, kw in calls]
assert not any(got), list(zip(got, calls))
"""


@pytest.mark.parametrize("name", ["hand3", "hand4x4", "hand5"])
def test_one_small_warm_up_covers_every_step(name):
    """A fresh process under lazy loading: after one small warm-up call no
    batch size, wrench count, solver, cone or energy takes device memory."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, CUDA_MODULE_LOADING="LAZY", PYTHONPATH=root)
    run = subprocess.run([sys.executable, "-c", LAZY, name], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr[-2000:]
