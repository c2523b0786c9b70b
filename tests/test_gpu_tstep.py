"""GPU parity of the T-step metric (params.sim_steps = T >= 1: each simulation
runs T PBD steps with the SDF re-queried at the predicted object pose) against
the FP64 oracle's evaluate_tstep, through the C ABI.

Tolerances as for the one-step path: loss 1e-4 relative, gradient and update
1e-3 relative per candidate, compared on candidates whose every decision (over
all steps and simulations) sits outside the guard band."""

import ctypes as C

import numpy as np
import pytest
import torch

import synth
from oracle import fastgraspd_oracle as O

pytestmark = pytest.mark.gpu

LOSS_TOL = 1e-4
GRAD_TOL = 1e-3


@pytest.fixture(scope="module")
def fg():
    from paper_2306_08132_gb300.build import build_library
    build_library()
    import paper_2306_08132_gb300 as m
    return m


def _dev():
    return torch.device("cuda:0")


class Case:
    def __init__(self, fg, w):
        self.w = w
        self.hand = fg.Hand.from_synth(w.hand)
        self.sdfs = [fg.Sdf.from_synth(o) for o in w.objects]
        self.scene = fg.Scene(self.sdfs)
        self.oc = torch.tensor(w.obj_of_cand, device=_dev(), dtype=torch.int32)

    def oracle(self, params):
        return O.Setup(self.w.hand, self.w.objects, params)

    def clean(self, S, q, r):
        mask = np.zeros(len(q), dtype=bool)
        for k in np.unique(self.w.obj_of_cand):
            idx = np.nonzero(self.w.obj_of_cand == k)[0]
            mask[idx] = O.clean_candidates(S.hand, S.objs[int(k)], q[idx], r, S.prm)
        return mask


def _rel_rows(a, b, floor=1e-6):
    return np.linalg.norm(a - b, axis=1) / np.maximum(np.linalg.norm(b, axis=1), floor)


def _compare(loss, grad, ref, clean):
    idx = np.nonzero(clean)[0]
    L = loss.astype(np.float64)[idx]
    lrel = np.abs(L - ref["L"][idx]) / np.maximum(np.abs(ref["L"][idx]), 1e-6)
    grel = _rel_rows(grad.astype(np.float64)[idx], ref["grad"][idx])
    assert lrel.max() < LOSS_TOL, (idx[np.argmax(lrel)], lrel.max())
    assert grel.max() < GRAD_TOL, (idx[np.argmax(grel)], grel.max())


@pytest.fixture(scope="module")
def tiny(fg):
    return Case(fg, synth.tiny_sphere_workload(n_cand=64))


@pytest.mark.parametrize("T,alpha", [(1, 0.1), (2, 0.1), (3, 0.1), (2, 0.0), (8, 0.1)])
def test_tstep_loss_and_grad_match_oracle(fg, tiny, T, alpha):
    w, r = tiny.w, 0.004
    params = dict(w.params, sim_steps=T, alpha_leak=alpha)
    q = torch.tensor(w.q0, device=_dev())
    loss, grad = fg.loss_and_grad(tiny.hand, tiny.scene, q, params, r, obj_of_cand=tiny.oc)
    S = tiny.oracle(params)
    ref = O.batch_loss_and_grad(S, w.q0, w.obj_of_cand, r)
    clean = tiny.clean(S, w.q0, r)
    assert clean.sum() >= 0.5 * len(clean), clean.sum()
    assert (ref["N"].sum(axis=1) > 0).sum() >= 8, "workload must exercise contacts"
    _compare(loss.cpu().numpy(), grad.cpu().numpy(), ref, clean)


def test_tstep_mixed_objects_four_finger(fg):
    w = synth.batched_superquadric_workload(n_obj=3, per_obj=12, grid_n=48, points_per_link=32, steps=50,
                                            device="cuda")
    case = Case(fg, w)
    params = dict(w.params, sim_steps=2)
    S = case.oracle(params)
    r = O.dilation_radius(S.prm, 7, w.steps)
    loss, grad = fg.loss_and_grad(case.hand, case.scene, torch.tensor(w.q0, device=_dev()), params, r,
                                  obj_of_cand=case.oc)
    ref = O.batch_loss_and_grad(S, w.q0, w.obj_of_cand, r)
    clean = case.clean(S, w.q0, r)
    assert clean.sum() >= 0.5 * len(clean)
    _compare(loss.cpu().numpy(), grad.cpu().numpy(), ref, clean)


def test_tstep_optimize_step_matches_oracle_and_is_reproducible(fg, tiny):
    w = tiny.w
    params = dict(w.params, sim_steps=2, r0=0.01, schedule="linear")
    S = tiny.oracle(params)
    K = 20
    q0 = torch.tensor(w.q0, device=_dev())
    q1 = q0.clone()
    loss = fg.optimize_step(tiny.hand, tiny.scene, q1, params, 3, K, 1, obj_of_cand=tiny.oc)
    r = O.dilation_radius(S.prm, 3, K)
    ref = O.batch_loss_and_grad(S, w.q0, w.obj_of_cand, r)
    step = (q1 - q0).cpu().numpy().astype(np.float64)
    _compare(loss.cpu().numpy(), -step / params["lr"], ref, tiny.clean(S, w.q0, r))
    # nsteps in one launch == repeated launches, bit for bit
    qa = q0.clone()
    la = fg.optimize_step(tiny.hand, tiny.scene, qa, params, 3, K, 3, obj_of_cand=tiny.oc)
    qb = q0.clone()
    for s in range(3):
        lb = fg.optimize_step(tiny.hand, tiny.scene, qb, params, 3 + s, K, 1, obj_of_cand=tiny.oc)
    torch.cuda.synchronize()
    assert torch.equal(qa, qb) and torch.equal(la, lb)
    # loss-only call equals the loss of the gradient call
    l1, _ = fg.loss_and_grad(tiny.hand, tiny.scene, q0, params, 0.004, obj_of_cand=tiny.oc)
    l2, none = fg.loss_and_grad(tiny.hand, tiny.scene, q0, params, 0.004, obj_of_cand=tiny.oc, want_grad=False)
    assert none is None and torch.equal(l1, l2)


def test_tstep_one_step_agrees_with_plane_form_on_flat_contact(fg, tiny):
    """On a linear field the plane linearisation is exact: T = 1 on the GPU gives the
    one-step kernel's loss and gradient to float32 rounding."""
    w = tiny.w
    n0 = np.array([0.48, -0.6, 0.64])
    n0 /= np.linalg.norm(n0)
    obj = synth.linear_grid(tuple(n0), -0.07, 80, 0.008)
    sdf = fg.Sdf.from_synth(obj)
    scene = fg.Scene([sdf])
    q = torch.tensor(w.q0, device=_dev())
    l0, g0 = fg.loss_and_grad(tiny.hand, scene, q, w.params, 0.004)
    l1, g1 = fg.loss_and_grad(tiny.hand, scene, q, dict(w.params, sim_steps=1), 0.004)
    torch.cuda.synchronize()
    L0, L1 = l0.cpu().numpy().astype(np.float64), l1.cpu().numpy().astype(np.float64)
    assert np.abs(L1 - L0).max() <= 1e-5 * np.abs(L0).max()
    rel = _rel_rows(g1.cpu().numpy().astype(np.float64), g0.cpu().numpy().astype(np.float64))
    assert np.median(rel) < 1e-4 and rel.max() < 1e-2


def test_tstep_is_refused_where_only_the_one_step_metric_exists(fg, tiny):
    from paper_2306_08132_gb300 import _lib
    w = tiny.w
    q = torch.tensor(w.q0[:4], device=_dev())
    params = dict(w.params, sim_steps=2)
    with pytest.raises(_lib.FgError) as e:
        fg.contact_wrench(tiny.hand, tiny.scene, q, params, 0.004)
    assert e.value.name == "FG_ERR_INVALID"
    with pytest.raises(_lib.FgError):
        fg.optimize_step_plain(tiny.hand, tiny.scene, q.clone(), params, 0, 10, 1)
    for bad in (-1, 9):
        with pytest.raises(_lib.FgError):
            fg.loss_and_grad(tiny.hand, tiny.scene, q, dict(w.params, sim_steps=bad), 0.004)


@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("points_per_link", [21, 100, 1300])
def test_tstep_ragged_and_large_hands(fg, T, points_per_link):
    """Links whose points are not 32-aligned (chunks across links, work units of 21 and 36 points) and a hand of
    13,000 points, more than the first step's unit table and the chunk culling take."""
    w = synth.tiny_sphere_workload(n_cand=12)
    h = synth.make_hand(3, points_per_link)
    qs = synth.sample_candidates(np.random.default_rng(7), h, 12, 0.095)
    case = Case(fg, synth.Workload("ragged", h, w.objects, qs, np.zeros(12, dtype=np.int32), w.params, 10))
    params = dict(w.params, sim_steps=T)
    S = case.oracle(params)
    q = torch.tensor(qs, device=_dev())
    loss, grad = fg.loss_and_grad(case.hand, case.scene, q, params, 0.004)
    ref = O.batch_loss_and_grad(S, qs, case.w.obj_of_cand, 0.004)
    clean = case.clean(S, qs, 0.004)
    assert clean.sum() >= 1
    _compare(loss.cpu().numpy(), grad.cpu().numpy(), ref, clean)
    l2, g2 = fg.loss_and_grad(case.hand, case.scene, q, params, 0.004)
    assert torch.equal(loss, l2) and torch.equal(grad, g2)


@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("nodes,pitch,v_test", [(63, 0.002, 1.0), (126, 0.001003, 1.0), (126, 0.001, 1.0),
                                                (140, 0.0009, 1.0), (63, 0.002, 0.0), (40, 0.002, 1.0)])
def test_tstep_pitch_against_the_displacement(fg, T, nodes, pitch, v_test):
    """The first step's queries lie dt V = 1 mm from the point: below one cell (corners shared by the
    simulations), at one cell, beyond it, at zero velocity, and on a grid smaller than the hand (clamped axes)."""
    w = synth.tiny_sphere_workload(n_cand=24)
    obj = synth.sphere_grid(0.03, nodes, pitch)
    case = Case(fg, synth.Workload("pitch", w.hand, [obj], w.q0, w.obj_of_cand, w.params, 10))
    params = dict(w.params, sim_steps=T, v_test=v_test)
    S = case.oracle(params)
    q = torch.tensor(w.q0, device=_dev())
    loss, grad = fg.loss_and_grad(case.hand, case.scene, q, params, 0.012)
    ref = O.batch_loss_and_grad(S, w.q0, w.obj_of_cand, 0.012)
    clean = case.clean(S, w.q0, 0.012)
    if v_test == 0.0:        # a candidate at rest without contacts has no stability gradient: nothing to divide by
        clean &= ref["N"].reshape(len(clean), -1).sum(axis=1) > 0
    assert clean.sum() >= 3
    _compare(loss.cpu().numpy(), grad.cpu().numpy(), ref, clean)


@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_tstep_contacts_past_an_upper_face(fg, T, axis):
    """A hand past a grid's last plane along one axis, where the field is that plane's value plus the excess
    distance.  The plane before it (1e6) must not enter the value, whose rounding would be 0.03 m against contacts
    of 0.02 m: the reverse sweep would miss contacts of the forward sweep."""
    w = synth.tiny_sphere_workload(n_cand=24)
    n, pitch = 200, 0.002
    wide, o = pitch * np.arange(n), [a for a in range(3) if a != axis]
    origin = np.array([-0.1995, -0.2003, -0.1998])
    origin[axis] = -0.0055
    plane = -0.02 + 0.15 * (wide + origin[o[0]])[:, None] - 0.1 * (wide + origin[o[1]])[None, :]
    g = np.full((4, n, n), 1e6)
    g[-1] = plane
    g = np.moveaxis(g, 0, axis)                                              # [x, y, z]
    obj = {"kind": "top", "grid": torch.tensor(np.ascontiguousarray(g.transpose(2, 1, 0)), dtype=torch.float32),
           "origin": origin.astype(np.float32), "pitch": float(np.float32(pitch)), "mass": 1.0, "inertia": 1e-3,
           "bound_radius": 0.05, "params": {}}
    params = dict(w.params, sim_steps=T)
    S = O.Setup(w.hand, [obj], params)
    q = w.q0.copy()
    q[:, :3] = 0.0
    pts = O.hand_points(S.hand, *O.forward_kinematics(S.hand, torch.tensor(q.astype(np.float64)))).numpy()
    q[:, axis] = float(obj["origin"][axis]) + 3 * obj["pitch"] + 0.004 - pts[..., axis].min(axis=1)
    loss, grad = fg.loss_and_grad(fg.Hand.from_synth(w.hand), fg.Scene([fg.Sdf.from_synth(obj)]),
                                  torch.tensor(q, device=_dev()), params, 0.004)
    ref = O.batch_loss_and_grad(S, q, np.zeros(len(q), dtype=np.int32), 0.004, chunk=len(q))
    clean = O.clean_candidates(S.hand, S.objs[0], q, 0.004, S.prm)
    assert clean.sum() >= 0.25 * len(clean) and (ref["N"].sum(axis=1) > 0).all()
    _compare(loss.cpu().numpy(), grad.cpu().numpy(), ref, clean)


def test_tstep_queries_of_a_frame_far_from_its_origin(fg):
    """300 m from the origin a position is a multiple of 2^-15 m, 0.0305 cells, so dt V = 0.9979 cells moves a query
    by 33 of them, 1.007 cells, and some queries land two cells away.  A displacement of 0.9981 cells moves every
    query by the same 33 multiples: the two gradients differ by the displacement's 2e-4 in friction and test
    velocity only (2e-3 allowed, and two candidates in which a contact's friction regime changes)."""
    w = synth.tiny_sphere_workload(n_cand=24)
    rng = np.random.default_rng(3)
    centre = np.array([300.0, -290.0, 310.0])
    base = synth.sphere_grid(0.05, 160, 0.001)
    rough = torch.tensor(rng.standard_normal((160, 160, 160)), dtype=torch.float32)
    obj = dict(base, grid=base["grid"] + 0.0015 * rough,
               origin=(base["origin"].astype(np.float64) + centre).astype(np.float32))
    q = w.q0.copy()
    q[:, :3] += centre.astype(np.float32)
    hand, scene = fg.Hand.from_synth(w.hand), fg.Scene([fg.Sdf.from_synth(obj)])
    G = []
    for v_test in (0.9979, 0.9981):
        _, g = fg.loss_and_grad(hand, scene, torch.tensor(q, device=_dev()),
                                dict(w.params, sim_steps=1, v_test=v_test), 0.004)
        G.append(g.cpu().numpy().astype(np.float64))
    rel = np.sort(_rel_rows(G[0], G[1]))
    assert rel[-3] < 2e-3, rel
