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
