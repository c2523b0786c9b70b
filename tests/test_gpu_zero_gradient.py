"""Contacts where the SDF's gradient is zero: n = 0, so the normal correction vanishes and the whole displacement is
tangential (t = D/|D|, w_t = 1/m + |d x t|^2/I).  A field that is 0 throughout the object has such contacts at every
point inside it (C = r).  Every form of the metric against the FP64 oracle.

Tolerances as for the other parity tests: loss 1e-4 relative, gradient, update and wrench 1e-3 relative per candidate,
on candidates whose every decision sits outside the guard band."""

import numpy as np
import pytest
import torch

import synth
from oracle import fastgraspd_oracle as O

pytestmark = pytest.mark.gpu

LOSS_TOL = 1e-4
GRAD_TOL = 1e-3
R = 0.004          # sigma = dt V = 1 mm: static friction at mu = 0.5 (mu C = 2 mm), kinetic at 0.05


@pytest.fixture(scope="module")
def fg():
    from paper_2306_08132_gb300.build import build_library
    build_library()
    import paper_2306_08132_gb300 as m
    return m


class Case:
    def __init__(self, fg, n_cand=24):
        self.w = synth.tiny_sphere_workload(n_cand=n_cand)
        obj = synth.sphere_grid(0.06, 64, 0.003)
        obj["grid"] = obj["grid"].clamp(min=0.0)
        self.obj = obj
        self.hand = fg.Hand.from_synth(self.w.hand)
        self.scene = fg.Scene([fg.Sdf.from_synth(obj)])
        self.q = torch.tensor(self.w.q0, device="cuda:0")

    def reference(self, params):
        """The oracle's results, and the clean candidates that have zero-gradient contacts."""
        S = O.Setup(self.w.hand, [self.obj], params)
        ref = O.batch_loss_and_grad(S, self.w.q0, np.zeros(len(self.w.q0), dtype=np.int32), R, chunk=len(self.w.q0))
        clean = O.clean_candidates(S.hand, S.objs[0], self.w.q0, R, S.prm)
        qd = torch.tensor(self.w.q0.astype(np.float64))
        _, g = O.sdf_query(S.objs[0], O.hand_points(S.hand, *O.forward_kinematics(S.hand, qd)), R)
        flat = ((g * g).sum(-1) == 0).sum(-1).numpy()
        idx = np.nonzero(clean & (flat > 0))[0]
        assert len(idx) >= 5
        return ref, idx


@pytest.fixture(scope="module")
def case(fg):
    return Case(fg)


def _check(loss, grad, ref, idx):
    L = loss.cpu().numpy().astype(np.float64)[idx]
    G = grad.cpu().numpy().astype(np.float64)[idx]
    lrel = np.abs(L - ref["L"][idx]) / np.maximum(np.abs(ref["L"][idx]), 1e-6)
    grel = np.linalg.norm(G - ref["grad"][idx], axis=1) / np.maximum(np.linalg.norm(ref["grad"][idx], axis=1), 1e-6)
    assert lrel.max() < LOSS_TOL, (idx[np.argmax(lrel)], lrel.max())
    assert grel.max() < GRAD_TOL, (idx[np.argmax(grel)], grel.max())


def _check_wrench(W, N, ref, idx):
    assert np.array_equal(N.cpu().numpy()[idx], ref["N"][idx].astype(np.int32))
    a, b = W.cpu().numpy().astype(np.float64)[idx].reshape(len(idx), -1), ref["W"][idx].reshape(len(idx), -1)
    rel = np.linalg.norm(a - b, axis=1) / np.maximum(np.linalg.norm(b, axis=1), 1e-9)
    assert rel.max() < GRAD_TOL, (idx[np.argmax(rel)], rel.max())


@pytest.mark.parametrize("mu", [0.5, 0.05])
@pytest.mark.parametrize("T", [1, 2])
def test_zero_gradient_contacts_tstep(fg, case, T, mu):
    params = dict(case.w.params, sim_steps=T, mu=mu)
    ref, idx = case.reference(params)
    loss, grad = fg.loss_and_grad(case.hand, case.scene, case.q, params, R)
    _check(loss, grad, ref, idx)


@pytest.mark.parametrize("mu", [0.5, 0.05])
def test_zero_gradient_contacts_gauss_seidel(fg, case, mu):
    params = dict(case.w.params, gauss_seidel=1, mu=mu)
    ref, idx = case.reference(params)
    loss, grad = fg.loss_and_grad(case.hand, case.scene, case.q, params, R)
    _check(loss, grad, ref, idx)
    W, N, _ = fg.contact_wrench(case.hand, case.scene, case.q, params, R)
    _check_wrench(W, N, ref, idx)


@pytest.mark.parametrize("mu", [0.5, 0.05])
def test_zero_gradient_contacts_averaged(fg, case, mu):
    params = dict(case.w.params, mu=mu)
    ref, idx = case.reference(params)
    try:
        for i in [-1] + list(range(len(fg.fused_configs()))):
            fg.fused_config_select(i)
            _check(*fg.loss_and_grad(case.hand, case.scene, case.q, params, R), ref, idx)
    finally:
        fg.fused_config_select(-1)
    W, N, _ = fg.contact_wrench(case.hand, case.scene, case.q, params, R)
    _check_wrench(W, N, ref, idx)


@pytest.mark.parametrize("mu", [0.5, 0.05])
def test_zero_gradient_contacts_per_stage(fg, case, mu):
    params = dict(case.w.params, mu=mu, r0=R)
    ref, idx = case.reference(params)
    q = case.q.clone()
    loss = fg.optimize_step_plain(case.hand, case.scene, q, params, 0, 10, 1)
    _check(loss, (case.q - q) / params["lr"], ref, idx)


def test_zero_gradient_contacts_in_the_queue_and_in_mixed_scenes(fg, case):
    """The request queue steps such an object as fg_optimize_step does, and another object's candidates keep their
    results, bit for bit, in a scene and in a round with it."""
    params = dict(case.w.params, r0=R)
    flat, plain = fg.Sdf.from_synth(case.obj), fg.Sdf.from_synth(case.w.objects[0])
    expected = []
    for sdf in (flat, plain):
        q = case.q.clone()
        loss = fg.optimize_step(case.hand, fg.Scene([sdf]), q, params, 0, 3, 1)
        expected.append((q.cpu().numpy(), loss.cpu().numpy()))
    q = torch.cat([case.q, case.q])
    oc = torch.arange(2, device=q.device, dtype=torch.int32).repeat_interleave(len(case.q))
    loss = fg.optimize_step(case.hand, fg.Scene([flat, plain]), q, params, 0, 3, 1, obj_of_cand=oc)
    np.testing.assert_array_equal(q.cpu().numpy(), np.concatenate([expected[0][0], expected[1][0]]))
    np.testing.assert_array_equal(loss.cpu().numpy(), np.concatenate([expected[0][1], expected[1][1]]))
    queue = fg.Queue(1 << 30)
    try:
        ids = [queue.submit(case.hand, s, case.w.q0, 1, params) for s in (flat, plain)]
        for rid, (qe, le) in zip(ids, expected):
            queue.wait(rid, 120000)
            qg, lg, _ = queue.result(rid)
            np.testing.assert_array_equal(qg, qe)
            np.testing.assert_array_equal(lg, le)
    finally:
        queue.close()


def test_zero_gradient_cell_anywhere_in_the_grid(fg):
    """One constant cell at each place of small odd and even grids, a hand of one point in it."""
    hand_d = {"parent": np.array([-1]), "T_fix": np.eye(3, 4)[None], "axis": np.zeros((1, 3)), "q_low": np.zeros(0),
              "q_up": np.zeros(0), "pts_local": np.array([[0.003, -0.002, 0.001]]), "link_of_point": np.array([0])}
    hand = fg.Hand.from_synth(hand_d)
    params = synth.tiny_sphere_workload(n_cand=1).params
    rng = np.random.default_rng(4)
    pitch = 0.02
    for dims in ((4, 3, 5), (2, 5, 4)):                                    # nodes along z, y, x
        cells = [(k, j, i) for k in range(dims[0] - 1) for j in range(dims[1] - 1) for i in range(dims[2] - 1)]
        objs, q = [], np.zeros((len(cells), 6), dtype=np.float32)
        for n, (k, j, i) in enumerate(cells):
            g = rng.uniform(-0.02, 0.02, size=dims).astype(np.float32)
            g[k:k + 2, j:j + 2, i:i + 2] = 0.0
            objs.append({"kind": "cell", "grid": torch.tensor(g), "origin": np.array([-0.03, -0.02, -0.04], dtype=np.float32),
                         "pitch": float(np.float32(pitch)), "mass": 0.7, "inertia": 4e-4, "bound_radius": 0.05, "params": {}})
            q[n, :3] = objs[-1]["origin"] + pitch * (np.array([i, j, k]) + rng.uniform(0.3, 0.7, 3)) - hand_d["pts_local"][0]
        oc = np.arange(len(cells), dtype=np.int32)
        S = O.Setup(dict(hand_d, L=1, J=0, D=6, P=1), objs, params)
        ref = O.batch_loss_and_grad(S, q, oc, R)
        assert (ref["N"] == 1).all()
        loss, grad = fg.loss_and_grad(hand, fg.Scene([fg.Sdf.from_synth(o) for o in objs]), torch.tensor(q, device="cuda:0"),
                                      params, R, obj_of_cand=torch.tensor(oc, device="cuda:0"))
        _check(loss, grad, ref, oc)


@pytest.mark.parametrize("form", [{}, {"gauss_seidel": 1}, {"sim_steps": 1}])
def test_zero_gradient_contacts_in_a_scene_with_a_mesh(fg, case, form):
    import synth.meshes
    params = dict(case.w.params, **form)
    ref, idx = case.reference(params)
    scene = fg.Scene([fg.Sdf.from_synth(synth.meshes.icosphere(0.04, 1)), fg.Sdf.from_synth(case.obj)])
    oc = torch.ones(len(case.q), device=case.q.device, dtype=torch.int32)
    _check(*fg.loss_and_grad(case.hand, scene, case.q, params, R, obj_of_cand=oc), ref, idx)


@pytest.mark.parametrize("points_per_link", [21, 1300])
def test_zero_gradient_contacts_of_ragged_and_large_hands(fg, case, points_per_link):
    """Chunks that span links, and 13,000 points (more chunks than are flagged, two parts of the adjoint sweep): the
    fused step against the per-stage form, which takes the same decisions at every point."""
    h = synth.make_hand(3, points_per_link)
    hand = fg.Hand.from_synth(h)
    q0 = torch.tensor(synth.sample_candidates(np.random.default_rng(5), h, 24, 0.1), device="cuda:0")
    for mu in (0.5, 0.05):
        params = dict(case.w.params, r0=R, mu=mu)
        a, b = q0.clone(), q0.clone()
        la = fg.optimize_step(hand, case.scene, a, params, 0, 10, 1)
        lb = fg.optimize_step_plain(hand, case.scene, b, params, 0, 10, 1)
        assert torch.allclose(la, lb, rtol=LOSS_TOL, atol=1e-6)
        ga, gb = (q0 - a).double(), (q0 - b).double()
        rel = (ga - gb).norm(dim=1) / gb.norm(dim=1).clamp(min=1e-9)
        assert float(rel.max()) < GRAD_TOL, rel
