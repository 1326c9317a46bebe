"""Receiver-misfit gradients on meshes above the sizes at which a degree's solvers switch to the tile kernels, whose adjoint
forms (the spatial operator alone, the stage's pre-kernel, the kept brackets) small meshes do not reach. FP64: the directional
derivatives in c^2 and in the initial state against central differences of forward runs. FP32: against FP64, which runs the team
kernels at N = 6. Bounds as in the other gradient tests on meshes of this size: 1e-6 of the derivative, 1e-3 (c^2) and
1e-4 (state) in FP32.
"""
import numpy as np
import pytest

from oracle import bernstein as bb
from paper_1808_08645_gb300 import binding as B
from paper_1808_08645_gb300 import inputs
from parity_util import rel_l2, rounded

pytestmark = pytest.mark.gpu

XR = np.random.default_rng(97).uniform(0.05, 0.95, (60, 3))
AMP = np.random.default_rng(98).uniform(-1.0, 1.0, 20)


def case(hexes, N, M, prec):
    v, e = inputs.cube_mesh(hexes, jitter=0.1, shuffle=True, seed=N)
    rng = np.random.default_rng(N + 7)
    c2 = rounded(rng.uniform(0.5, 2.0, (len(e), bb.np_count(M))), prec)
    q0 = rounded(rng.standard_normal((4, len(e), bb.np_count(N))) * 0.1, prec)
    return v, e, c2, q0, rng


def run(mesh, N, prec, c2, q0, data, every, grad=True):
    """Misfit against data, and its gradients."""
    steps = len(data)
    with B.Solver(*mesh, N, 1, prec) as s:
        s.set_c2(c2)
        s.set_state(q0)
        s.set_point_source([0.5, 0.5, 0.5], AMP)
        s.set_receivers(XR)
        tr = s.record(DT, steps, every)
        J = 0.5 * np.sum((tr - data) ** 2)
        return (J, *s.adjoint(tr - data, want_q0=True)) if grad else J


DT = 2e-3


@pytest.mark.parametrize("N,hexes", [(1, 12), (2, 14), (3, 12)])
def test_gradient_against_finite_differences(N, hexes):
    v, e, c2, q0, rng = case(hexes, N, 1, 32)
    data = rng.standard_normal((2, len(XR))) * 1e-3
    J, gc, gq = run((v, e), N, 64, c2, q0, data, 0)
    J1, gc1, gq1 = run((v, e), N, 64, c2, q0, data, 1)  # brackets recomputed from checkpoints
    assert J1 == J and np.array_equal(gc1, gc) and np.array_equal(gq1, gq)
    d = rng.uniform(-0.1, 0.1, c2.shape)
    w = rng.uniform(-0.1, 0.1, q0.shape)
    eps = 1e-6
    fd = (run((v, e), N, 64, c2 + eps * d, q0, data, 0, False) - run((v, e), N, 64, c2 - eps * d, q0, data, 0, False)) / (2 * eps)
    assert abs(fd - np.sum(gc * d)) <= 1e-6 * abs(fd)
    eps = 1e-5
    fd = (run((v, e), N, 64, c2, q0 + eps * w, data, 0, False) - run((v, e), N, 64, c2, q0 - eps * w, data, 0, False)) / (2 * eps)
    assert abs(fd - np.sum(gq * w)) <= 1e-6 * abs(fd)
    _, g32, q32 = run((v, e), N, 32, c2, q0, data, 0)
    assert rel_l2(g32, gc) <= 1e-3 and rel_l2(q32, gq) <= 1e-4


def test_degree_6_against_the_team_kernels():
    v, e, c2, q0, rng = case(24, 6, 1, 32)
    data = rng.standard_normal((1, len(XR))) * 1e-3
    _, gc, gq = run((v, e), 6, 64, c2, q0, data, 0)
    _, g32, q32 = run((v, e), 6, 32, c2, q0, data, 0)
    assert rel_l2(g32, gc) <= 1e-3 and rel_l2(q32, gq) <= 1e-4
