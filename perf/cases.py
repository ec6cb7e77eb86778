"""The work that users of this framework have it do, as cases to be timed and compared.

Each case goes through the package's public calls.  `kind` names the call:

* ``step``        -- ``bodex_step``: a synthesis run of fused upper iterations on one object;
* ``multi``       -- ``bodex_step_multi``: jobs of several hands and objects in one launch;
* ``synthesize``  -- the whole coarse / fine / final schedule;
* ``qp``          -- ``bodex_qp_solve_batch``: lower-level QPs alone;
* ``energy``      -- ``grasp_energy`` forward and backward through autograd;
* ``refine``      -- ``bodex_refine``: the fine stage after a coarse run;
* ``contacts``    -- ``bodex_fk_contacts`` and ``bodex_contact_metrics`` of candidate poses.

Hands, grid sizes, batch sizes and parameters are those of the package's named workloads, benchmark and tests.
"""
import math

import numpy as np
import torch

import bodex_inputs as I
import paper_2412_16490_gb300 as bx
from paper_2412_16490_gb300.autograd import grasp_energy

COLLISION = dict(w_pen=100.0, w_self=100.0, w_lim=10.0, eta_pen=0.005, eta_lim=0.05)
MIXED = (("hand3", 1 / 17), ("hand4x4", 4 / 17), ("hand5", 12 / 17))  # the mixed batch: 512 / 2048 / 6144 grasps
MIXED_GRIDS = (48, 56, 64, 72, 80, 96)


def listed():
    return [
        # the smallest run: one quick plan on an analytic sphere, bound by latency
        dict(name="step_tiny", kind="step", hand="hand4", grid=0, B=64, s=6, steps=50, iters=30, lower="admm", collide=False),
        # the paper's coarse stage, as the benchmark has it
        dict(name="step_paper", kind="step", hand="hand5", grid=64, B=4096, s=12, steps=200, iters=50, lower="admm", collide=False),
        # a ragged batch with the hand-object, self-collision and joint-limit energies on
        dict(name="step_collision", kind="step", hand="hand4x4", grid=64, B=1501, s=12, steps=50, iters=50, lower="admm", collide=True),
        # every QP of every step solved exactly: what a server's accurate jobs run
        dict(name="step_exact", kind="step", hand="hand5", grid=64, B=4096, s=12, steps=25, iters=64, lower="exact", collide=False),
        # several users' jobs sharing a launch: three hands, six objects
        dict(name="multi_mixed", kind="multi", B=8704, s=12, steps=50, iters=50),
        # one object's whole schedule, 300 / 100 / 100 steps
        dict(name="synthesize", kind="synthesize", hand="hand5", grid=64, B=1024, s=12, iters=50, coarse=300, fine=100),
        # the paper's QPs alone, to a residual
        dict(name="qp_paper", kind="qp", hand="hand5", grid=64, B=4096, s=12, lower="admm", iters=5000),
        # a small ragged set of second-order-cone programs
        dict(name="qp_cone_small", kind="qp", hand="hand4", grid=0, B=67, s=6, lower="cone", iters=5000),
        # the paper's QPs, exactly
        dict(name="qp_exact", kind="qp", hand="hand5", grid=64, B=4096, s=12, lower="exact", iters=64),
        # gradients for another optimiser: forward (QPs to a residual) and backward
        dict(name="energy_grad", kind="energy", hand="hand4", grid=0, B=1024, s=6, lower="admm", iters=5000),
        # the fine stage of a coarse batch
        dict(name="refine_paper", kind="refine", hand="hand5", grid=64, B=4096, s=12, steps=100),
        # screening candidate poses: contacts, grasp matrices, fingertip distances
        dict(name="contacts", kind="contacts", hand="hand5", grid=64, B=16384),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "multi", "synthesize", "qp", "qp", "qp", "energy", "refine", "contacts"])
    hand = rng.choice(["hand3", "hand4", "hand4x4", "hand5"])
    grid = rng.choice([0, rng.randint(32, 96), rng.randint(32, 96)])
    s = rng.choice([6, 12])
    where = dict(kind=kind, hand=hand, grid=grid)
    if kind == "step":
        lower = rng.choice(["admm", "admm", "cone", "exact"])
        B = _log(rng, 16, 4096)
        steps = min(200 if lower != "exact" else 25, _log(rng, 1, 200))
        return dict(where, B=B, s=s, steps=steps, iters=64 if lower == "exact" else rng.randint(20, 50), lower=lower, collide=rng.random() < 0.3)
    if kind == "multi":
        return dict(kind=kind, B=_log(rng, 170, 8704), s=12, steps=rng.randint(10, 50), iters=rng.randint(20, 50))
    if kind == "synthesize":
        return dict(where, B=_log(rng, 16, 1024), s=s, iters=rng.randint(20, 50), coarse=rng.randint(100, 300), fine=rng.randint(20, 100))
    if kind == "qp":
        lower = rng.choice(["admm", "cone", "adaptive", "finish", "exact"])
        return dict(where, B=_log(rng, 8, 4096), s=s, lower=lower, iters={"exact": 64, "finish": 200}.get(lower, 5000))
    if kind == "energy":
        lower = rng.choice(["admm", "fixed", "exact"])
        return dict(where, B=_log(rng, 16, 2048), s=s, lower=lower, iters={"exact": 64, "fixed": 50}.get(lower, 5000))
    if kind == "refine":
        return dict(where, B=_log(rng, 16, 4096), s=s, steps=rng.randint(10, 100))
    return dict(where, B=_log(rng, 64, 16384))


# ------------------------------------------------------------------ inputs
def _object(grid, seed):
    return I.grid_object(seed, n=grid) if grid else I.sphere_object()


def _poses(hand, obj, B, rng, gap, flex):
    """bodex_inputs.initial_poses' distribution, all poses at once: the palm a gap outside the object's surface along a
    random direction, facing it, with a random roll and mildly flexed fingers."""
    u = rng.normal(size=(B, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    s = np.full(B, 0.2)
    for _ in range(10):  # sphere tracing from outside
        s -= obj.sdf(s[:, None] * u)
    z = -u
    a = np.cross(z, np.where(np.abs(z[:, :1]) < 0.9, [[1.0, 0.0, 0.0]], [[0.0, 1.0, 0.0]]))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    psi = rng.uniform(0, 2 * math.pi, size=(B, 1))
    x = np.cos(psi) * a + np.sin(psi) * np.cross(z, a)
    R = np.stack([x, np.cross(z, x), z], axis=2)
    out = np.zeros((B, hand.dof))
    out[:, :3] = (s + rng.uniform(*gap, size=B))[:, None] * u
    out[:, 3] = np.arctan2(-R[:, 1, 2], R[:, 2, 2])
    out[:, 4] = np.arcsin(np.clip(R[:, 0, 2], -1, 1))
    out[:, 5] = np.arctan2(-R[:, 0, 1], R[:, 0, 0])
    out[:, 6:] = rng.uniform(0, flex, size=(B, hand.n_joints)) * hand.qmax[6:]
    return out.astype(np.float32)


def _scene(case, seed):
    """Hand template, object and poses: approach poses, or near the surface for the stages after the coarse one."""
    rng = np.random.default_rng(seed)
    hand, obj = I.hand_template(case["hand"]), _object(case["grid"], seed)
    near = case["kind"] in ("refine", "contacts")
    x = _poses(hand, obj, case["B"], rng, (-0.01, 0.005) if near else (0.02, 0.05), 0.8 if near else 0.3)
    return hand, obj, x


def _qp(case):
    lower, it = case["lower"], case["iters"]
    if lower == "exact":
        return bx.qp_params(max_iter=it, solver=bx.QP_EXACT)
    cone = bx.CONE_ELLIPTIC if lower == "cone" else bx.CONE_PYRAMID
    if case["kind"] == "step" or lower == "fixed":
        return bx.qp_params(max_iter=it, cone=cone)
    return bx.qp_params(max_iter=it, eps_abs=1e-5, check_every=10, cone=cone, adaptive_rho=int(lower == "adaptive"), polish=2 * int(lower == "finish"))


def _dev(a):
    return torch.as_tensor(a).cuda()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "multi":
        rng = np.random.default_rng(seed)
        st["T"] = _dev(I.wrench_set(case["s"]))
        st["params"] = bx.step_params(I.default_params(), qp=bx.qp_params(max_iter=case["iters"]))
        st["jobs"], st["x0"] = [], []
        for k, n in enumerate(MIXED_GRIDS):
            name, share = MIXED[k // 2]
            hand, obj = I.hand_template(name), _object(n, seed * 6 + k)
            x = _dev(_poses(hand, obj, max(1, int(case["B"] * share / 2)), rng, (0.02, 0.05), 0.3))
            H = bx.Hand(hand)
            st["x0"].append(x)
            st["jobs"].append(dict(hand=H, obj=bx.Object(obj), state=bx.State(H, len(x), case["s"]), T=st["T"], n_steps=case["steps"],
                                   E_last=torch.empty(len(x), device="cuda"), status=torch.empty(len(x), dtype=torch.int32, device="cuda")))
        return st
    hand, obj, x = _scene(case, seed)
    B = case["B"]
    st.update(hand=bx.Hand(hand), obj=bx.Object(obj), x=_dev(x))
    if kind == "contacts":
        return st
    st["T"] = _dev(I.wrench_set(case["s"]))
    if kind == "qp":
        st["G"] = bx.bodex_fk_contacts(st["hand"], st["obj"], st["x"])["G"]
        st["params"] = _qp(case)
        return st
    P = I.default_params(**(COLLISION if case.get("collide") else {}))
    if kind == "energy":
        st["params"] = bx.step_params(P, qp=_qp(case))
        st["x"].requires_grad_(True)
        return st
    st["params"] = bx.step_params(P, qp=_qp(case) if kind == "step" else bx.qp_params(max_iter=case.get("iters", 50)))
    if kind != "synthesize":
        st.update(state=bx.State(st["hand"], B, case["s"]), E=torch.empty(B, device="cuda"), status=torch.empty(B, dtype=torch.int32, device="cuda"))
    if kind == "refine":
        st["p"] = bx.bodex_fk_contacts(st["hand"], st["obj"], st["x"])["p"] + 0.003
        st["kstar"] = torch.empty((B, hand.n_contacts), dtype=torch.int32, device="cuda")
    return st


# ------------------------------------------------------------------ one pass
def _moments(state):
    m, v, _ = state.adam()
    return dict(m=m, v=v)


def run(st):
    kind = st["case"]["kind"]
    if kind == "step":
        st["state"].set_pose(st["x"])
        bx.bodex_step(st["hand"], st["obj"], st["state"], st["T"], st["case"]["steps"], st["params"], E_last=st["E"], status=st["status"])
        return dict(x=st["state"].pose(), E=st["E"], status=st["status"], **_moments(st["state"]))
    if kind == "multi":
        for job, x in zip(st["jobs"], st["x0"]):
            job["state"].set_pose(x)
        bx.bodex_step_multi(st["jobs"], st["params"])
        return [dict(x=j["state"].pose(), E=j["E_last"], status=j["status"], **_moments(j["state"])) for j in st["jobs"]]
    if kind == "synthesize":
        return bx.synthesize(st["hand"], st["obj"], st["x"], st["T"], st["params"], coarse_steps=st["case"]["coarse"],
                             fine_steps=st["case"]["fine"], final_steps=st["case"]["fine"])
    if kind == "qp":
        return bx.bodex_qp_solve_batch(st["G"], st["T"], st["params"])
    if kind == "energy":
        E = grasp_energy(st["x"], st["hand"], st["obj"], st["T"], st["params"])
        (g,) = torch.autograd.grad(E.sum(), st["x"])
        return dict(E=E, grad=g)
    if kind == "refine":
        st["state"].set_pose(st["x"])
        bx.bodex_refine(st["hand"], st["obj"], st["state"], st["p"], st["case"]["steps"], 0.01, 1000.0, st["params"], E_last=st["E"],
                        kstar=st["kstar"], status=st["status"])
        return dict(x=st["state"].pose(), E=st["E"], kstar=st["kstar"], status=st["status"], **_moments(st["state"]))
    return dict(contacts=bx.bodex_fk_contacts(st["hand"], st["obj"], st["x"]), metrics=bx.bodex_contact_metrics(st["hand"], st["obj"], st["x"]))


# ------------------------------------------------------------------ what a pass cannot do without
def _iteration_flops(m, cone):
    """One ADMM iteration: the products with A and its transpose, with K^-1, and the rows' projections and updates."""
    nv, nnz, nc = 3 * m, (5 if cone else 26) * m, (4 if cone else 9) * m + 1
    return 4 * nnz + 2 * nv * nv + 6 * nv + 10 * nc


def _step_flops(hand, s, iters, lower):
    """One grasp's upper iteration: kinematics, query, G, K^-1, the QPs, the energy's gradient, Adam."""
    m, nv = hand.n_contacts, 3 * hand.n_contacts
    qps = s * (4000 if lower == "exact" else iters * _iteration_flops(m, lower == "cone"))
    return qps + 6 * nv * (nv + 1) + 2 * nv ** 3 + 72 * hand.dof + 150 * m + 1000 + s * 24 * nv


def _refine_flops(hand, S=32):
    return hand.n_contacts * (S * 60 + 300) + 72 * hand.dof


def work(case):
    kind = case["kind"]
    if kind == "multi":
        f = b = 0
        for name, share in MIXED:
            hand, n = I.hand_template(name), int(case["B"] * share)
            f += n * case["steps"] * _step_flops(hand, case["s"], case["iters"], "admm")
            b += 4 * n * 4 * hand.dof
        return dict(bytes=b + 4 * sum(n ** 3 for n in MIXED_GRIDS), flops=f)
    hand, B, s = I.hand_template(case["hand"]), case["B"], case.get("s", 0)
    m, D = hand.n_contacts, hand.dof
    grid = 4 * case["grid"] ** 3
    if kind == "step":
        return dict(bytes=4 * B * (4 * D + 2) + grid, flops=B * case["steps"] * _step_flops(hand, s, case["iters"], case["lower"]))
    if kind == "synthesize":
        return dict(bytes=4 * B * (4 * D + m + 2) + grid,
                    flops=B * (case["coarse"] * _step_flops(hand, s, case["iters"], "admm") + 2 * case["fine"] * _refine_flops(hand)))
    if kind == "qp":
        nc = (4 if case["lower"] == "cone" else 9) * m + 1
        # the iterations that such QPs take in the mean, or the minimum-norm-point method's 13 or so calls
        f = 13 * 1000 if case["lower"] == "exact" else {"cone": 250, "finish": 180}.get(case["lower"], 600) * _iteration_flops(m, case["lower"] == "cone")
        return dict(bytes=4 * B * (18 * m + s * (3 * m + 2 * nc + 5)), flops=B * s * f)
    if kind == "energy":
        it = {"exact": 10, "fixed": 50}.get(case["lower"], 600)
        return dict(bytes=4 * B * (2 * D + 1) + grid, flops=B * 2 * _step_flops(hand, s, it, case["lower"]))
    if kind == "refine":
        return dict(bytes=4 * B * (4 * D + 4 * m + 2) + grid, flops=B * case["steps"] * _refine_flops(hand))
    return dict(bytes=4 * B * (D + 13 * m + 18 * m + 1 + m + 1) + grid, flops=B * (2 * 72 * D + _refine_flops(hand)))


# ------------------------------------------------------------------ the same in 64 bits
def _t(a):
    return torch.as_tensor(np.asarray(a, np.float64), device="cuda")


def _rot(axis, q):
    """Rodrigues' rotation about a unit axis [3] by q [B]."""
    x, y, z = (float(v) for v in axis)
    K = _t([[0, -z, y], [z, 0, -x], [-y, x, 0]])
    s, c = torch.sin(q)[:, None, None], torch.cos(q)[:, None, None]
    return torch.eye(3, dtype=torch.float64, device="cuda") + s * K + (1 - c) * (K @ K)


def _links(hand, x):
    """World frames (R [B,3,3], t [B,3]) of every joint."""
    R = _rot((1, 0, 0), x[:, 3]) @ _rot((0, 1, 0), x[:, 4]) @ _rot((0, 0, 1), x[:, 5])
    root, out = (R, x[:, :3]), []
    for j in range(hand.n_joints):
        R, t = root if hand.parent[j] < 0 else out[hand.parent[j]]
        off = _t(hand.offset[j].reshape(3, 4))
        out.append((R @ off[:, :3] @ _rot(hand.axis[j], x[:, 6 + j]), t + R @ off[:, 3]))
    return out


def _sdf(obj, c):
    """phi, its gradient and the voxel cell at points c [..., 3]: the sphere, or the trilinear grid with phi(clamp c) + |c - clamp c|
    outside its box."""
    if obj.kind == "sphere":
        v = c - _t(obj.center)
        L = v.norm(dim=-1)
        return L - float(np.float32(obj.radius)), v / L[..., None]
    N, h, V, org = obj.n, float(np.float32(obj.h)), _t(obj.values).reshape(-1), _t(obj.origin)
    lo, hi = org, org + h * (N - 1)
    cl = torch.minimum(torch.maximum(c, lo), hi)
    u = (cl - org) / h
    k = u.detach().floor().clamp(0, N - 2).long()
    t = u - k
    base = (k[..., 2] * N + k[..., 1]) * N + k[..., 0]
    v = [[[V[base + (dz * N + dy) * N + dx] for dx in (0, 1)] for dy in (0, 1)] for dz in (0, 1)]
    tx, ty, tz = t[..., 0], t[..., 1], t[..., 2]
    lerp = lambda a, b, w: a + w * (b - a)  # noqa: E731
    a = [[lerp(v[z][y][0], v[z][y][1], tx) for y in (0, 1)] for z in (0, 1)]
    d = [[v[z][y][1] - v[z][y][0] for y in (0, 1)] for z in (0, 1)]
    g = torch.stack([lerp(lerp(d[0][0], d[0][1], ty), lerp(d[1][0], d[1][1], ty), tz), lerp(a[0][1] - a[0][0], a[1][1] - a[1][0], tz),
                     lerp(a[1][0], a[1][1], ty) - lerp(a[0][0], a[0][1], ty)], -1) / h
    dv = c - cl
    out = (c < lo) | (c > hi)
    far = out.any(-1)
    dl = torch.where(far[..., None], dv, torch.ones_like(dv)).norm(dim=-1)
    phi = lerp(lerp(a[0][0], a[0][1], ty), lerp(a[1][0], a[1][1], ty), tz) + torch.where(far, dl, torch.zeros_like(dl))
    return phi, torch.where(out, dv / dl[..., None], g)


def _centre(obj):
    if obj.kind == "sphere":
        return _t(obj.center)
    iz, iy, ix = np.nonzero(obj.values < 0)
    return _t(obj.origin) + float(np.float32(obj.h)) * _t([ix.mean(), iy.mean(), iz.mean()])


def _contacts(hand, obj, x):
    """Contact points, nearest points, inward normals, distances and grasp matrices."""
    F = _links(hand, x)
    c = torch.stack([F[L][1] + F[L][0] @ _t(p) for L, p in zip(hand.contact_link, hand.contact_local)], 1)
    phi, g = _sdf(obj, c)
    no = g / g.norm(dim=-1, keepdim=True)
    p, n = c - phi[..., None] * no, -no
    sg = torch.where(n[..., 2].detach() >= 0, 1.0, -1.0).to(n.dtype)
    a = -1 / (sg + n[..., 2])  # Duff et al.'s basis, as the package documents it
    b = n[..., 0] * n[..., 1] * a
    d = torch.stack([1 + sg * n[..., 0] ** 2 * a, sg * b, -sg * n[..., 0]], -1)
    e = torch.stack([b, sg + n[..., 1] ** 2 * a, -n[..., 1]], -1)
    cols = torch.stack([n, d, e], 2)  # [B, m, 3 columns, 3]
    W = torch.cat([cols, torch.linalg.cross((p - _centre(obj))[:, :, None].expand_as(cols), cols)], -1)
    return c, p, n, phi, W.reshape(len(x), -1, 6).transpose(1, 2)


def _tips(hand, obj, x):
    F = _links(hand, x)
    return torch.stack([_sdf(obj, F[L][1][:, None] + _t(tip) @ F[L][0].transpose(1, 2))[0].amin(1) for L, tip in zip(hand.contact_link, hand.tip_samples)], 1)


def _rows(m, mu, cone):
    """The QP's constraint matrix A: per contact f_n, then 8 facets or the cone's rows; the sum row last."""
    per = 4 if cone else 9
    A = np.zeros((per * m + 1, 3 * m))
    for i in range(m):
        A[per * i, 3 * i] = 1
        if cone:
            A[per * i + 1:per * i + 4, 3 * i:3 * i + 3] = np.diag([mu, 1, 1])
        for k in range(0 if cone else 8):
            f = (2 * k + 1) * math.pi / 8
            A[9 * i + 1 + k, 3 * i:3 * i + 3] = (-mu * math.cos(math.pi / 8), math.cos(f), math.sin(f))
    A[-1, 0::3] = 1
    return _t(A)


def _project(w, m, gamma, cone):
    z = torch.empty_like(w)
    v = w[:, :-1].reshape(len(w), m, -1)
    out = z[:, :-1].view(len(w), m, -1)
    out[..., 0] = v[..., 0].clamp(0, 1)
    if cone:
        s, u = v[..., 1], v[..., 2:]
        r = u.norm(dim=-1)
        k = torch.where(r <= s, torch.ones_like(s), torch.where(r <= -s, torch.zeros_like(s), 0.5 * (s + r) / r.clamp_min(1e-300)))
        out[..., 1] = torch.where(r <= s, s, torch.where(r <= -s, torch.zeros_like(s), 0.5 * (s + r)))
        out[..., 2:] = k[..., None] * u
    else:
        out[..., 1:] = v[..., 1:].clamp(max=0)
    z[:, -1] = w[:, -1].clamp(min=gamma)
    return z


def _admm(G, T, p, m):
    """The documented ADMM of every QP in 64 bits: y, z, lam [B*s, ...]."""
    B, s = len(G), len(T)
    cone = p.cone == bx.CONE_ELLIPTIC
    A = _rows(m, p.mu, cone)
    P = 2 * G.transpose(1, 2) @ G
    Ki = torch.linalg.inv(P + p.sigma * torch.eye(3 * m, dtype=P.dtype, device="cuda") + p.rho * A.T @ A)
    q = (-2 * p.beta * T @ G).reshape(B * s, -1)  # [B, s, nv]
    y, w = torch.zeros_like(q), torch.zeros((B * s, len(A)), dtype=q.dtype, device="cuda")
    run_, it = torch.arange(B * s, device="cuda"), 0
    while len(run_) and it < p.max_iter:
        yr, wr, qr, Kr, Pr = y[run_], w[run_], q[run_], Ki[run_ // s], P[run_ // s]
        for _ in range(min(p.check_every if p.eps_abs > 0 else p.max_iter, p.max_iter - it)):
            z = _project(wr, m, p.gamma, cone)
            ys = torch.bmm(Kr, (p.sigma * yr - qr + p.rho * (2 * z - wr) @ A)[..., None])[..., 0]
            wr = wr + p.alpha * (ys @ A.T - z)
            yr = p.alpha * ys + (1 - p.alpha) * yr
            it += 1
        y[run_], w[run_] = yr, wr
        z = _project(wr, m, p.gamma, cone)
        rp = (yr @ A.T - z).abs().amax(1)
        rd = (torch.bmm(Pr, yr[..., None])[..., 0] + qr + p.rho * (wr - z) @ A).abs().amax(1)
        if p.eps_abs > 0:
            run_ = run_[(rp > p.eps_abs) | (rd > p.eps_abs)]
    z = _project(w, m, p.gamma, cone)
    return y, z, p.rho * (w - z)


def _optimum(G, T, p, m):
    """Q* = min |beta t - G y|^2 over the pyramids, by Wolfe's minimum-norm-point method on all QPs at once."""
    s = len(T)
    b = (p.beta * T).repeat(len(G), 1)
    Gq = G.repeat_interleave(s, 0)
    n, K = len(b), 8
    k = torch.arange(8, dtype=torch.float64, device="cuda") * math.pi / 4
    E = torch.stack([torch.ones_like(k), p.mu * torch.cos(k), p.mu * torch.sin(k)], 1)  # the pyramid's edge tips
    tips = torch.einsum("qric,kc->qikr", Gq.reshape(n, 6, m, 3), E)  # [n, m, 8, 6]

    def oracle(x):
        best, at = (tips @ x[:, None, :, None])[..., 0].min(-1)  # [n, m]
        f, order = torch.empty_like(best), best.argsort(1)
        left = torch.full((n,), float(p.gamma), dtype=torch.float64, device="cuda")
        for j in range(m):
            i = order[:, j:j + 1]
            take = torch.where(best.gather(1, i)[:, 0] < 0, torch.ones_like(left), left.clamp(0, 1))
            f.scatter_(1, i, take[:, None])
            left = left - take
        tip = tips.gather(2, at[..., None, None].expand(-1, -1, 1, 6))[:, :, 0]
        return (f[..., None] * tip).sum(1) - b

    P, lam, on = torch.zeros((n, K, 6), dtype=torch.float64, device="cuda"), torch.zeros((n, K), dtype=torch.float64, device="cuda"), torch.zeros((n, K), dtype=torch.bool, device="cuda")
    P[:, 0], lam[:, 0], on[:, 0] = oracle(-b), 1, True
    eye, done = torch.eye(K, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.bool, device="cuda")
    for _ in range(60):
        x = (lam[..., None] * P).sum(1)
        q = oracle(x)
        done = done | ((x * x).sum(1) - (x * q).sum(1) <= 1e-13) | on.all(1)
        if bool(done.all()):
            break
        slot = (~on).long().argmax(1)
        new = ~done
        P[new, slot[new]] = q[new]
        on[new, slot[new]] = True
        open_ = new.clone()
        for _ in range(K + 1):
            mask = on.double()
            M = mask[:, :, None] * mask[:, None, :] * (1 + P @ P.transpose(1, 2)) + (1 - mask)[..., None] * eye + 1e-15 * eye
            al = torch.linalg.solve(M, mask[..., None])[..., 0] * mask
            al = al / al.sum(1, keepdim=True)
            bad = on & (al <= 0)
            th = torch.where(bad, lam / (lam - al).clamp_min(1e-300), torch.ones_like(lam)).amin(1).clamp(0, 1)
            nl = torch.where(on, lam + th[:, None] * (al - lam), torch.zeros_like(lam))
            drop = bad & (nl <= 1e-14)
            lam = torch.where(open_[:, None], nl.clamp_min(0), lam)
            on = torch.where(open_[:, None], on & ~drop, on)
            lam = lam * on
            lam = lam / lam.sum(1, keepdim=True)
            open_ = open_ & bad.any(1)
            if not bool(open_.any()):
                break
    x = (lam[..., None] * P).sum(1)
    return (x * x).sum(1).reshape(len(G), s)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "multi", "synthesize", "refine"):
        return None  # Adam divides by its second moment: over many steps, rounding alone ends at other poses
    hand, obj, x32 = _scene(case, seed)
    x, m = _t(x32), hand.n_contacts
    if kind == "contacts":
        c, p, n, phi, G = _contacts(hand, obj, x)
        d = _tips(hand, obj, x)
        return dict(contacts=dict(c=c, p=p, n=n, phi=phi, G=G, cell=None, status=None), metrics=dict(d=d, cdc=d.amax(1) - d.amin(1)))
    T, p = _t(I.wrench_set(case["s"])), _qp(case)
    if kind == "qp":
        if case["lower"] in ("adaptive", "finish"):
            return None  # which penalty, or which of the two methods, a QP gets hangs on rounding
        G = bx.bodex_fk_contacts(bx.Hand(hand), bx.Object(obj), _dev(x32))["G"].double()  # the input that prepare() makes
        none = dict(iters=None, status=None, res=None)
        if case["lower"] == "exact":
            return dict(y=None, z=None, lam=None, Q=_optimum(G, T, p, m), **none)  # the minimiser is not unique, its value is
        y, z, lam = (v.reshape(len(G), len(T), -1) for v in _admm(G, T, p, m))
        return dict(y=y, z=z, lam=lam, Q=(p.beta * T - y @ G.transpose(1, 2)).square().sum(-1), **none)
    P = I.default_params()
    x.requires_grad_(True)
    _, _, _, phi, G = _contacts(hand, obj, x)
    dist = P["w_d"] * (phi - float(np.float32(hand.contact_radius)) - P["delta"]).square().sum(1)
    if case["lower"] == "exact":
        return dict(E=P["w_q"] * _optimum(G.detach(), T, p, m).sum(1) + dist.detach(), grad=None)  # no gradient where y is not unique
    y = _admm(G.detach(), T, p, m)[0].reshape(len(x), len(T), -1)
    E = P["w_q"] * (p.beta * T - y @ G.transpose(1, 2)).square().sum((1, 2)) + dist
    (g,) = torch.autograd.grad(E.sum(), x)
    return dict(E=E.detach(), grad=g)
