"""The elastic kernels with one element per lane (FP32 solvers above a size per degree) against the library's FP64 team kernels,
which the parity tests check against the oracle: one stage from a random state on meshes of at least the switching size
whose element count is no multiple of 32 (ragged last warp), every face orientation, all media degrees.

Tolerance: an FP32 stage agrees with the FP64 oracle to 1e-5 (the parity tests' bound) and the FP64 one to 1e-11.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_08645_gb300 import binding as B  # noqa: E402
from paper_1808_08645_gb300 import inputs  # noqa: E402
from parity_util import rel_l2  # noqa: E402

_meshes = {}


def mesh(n):
    if n not in _meshes:
        _meshes[n] = inputs.cube_mesh(n, jitter=0.1, shuffle=True, seed=n)
    return _meshes[n]


def rounded(rng, lo, hi, shape):
    return rng.uniform(lo, hi, shape).astype(np.float32).astype(np.float64)


def stage(prec, v, e, N, M, media, q, r, s):
    with B.ElasticSolver(v, e, N, M, prec) as solver:
        solver.set_media(*media)
        solver.set_params(0.5, 2.0)
        solver.set_state(q, r)
        solver.stage(s, 1e-3)
        qo, ro, _ = solver.get_state(with_res=True)
        solver.sync()
    return np.concatenate([qo.ravel(), 1e3 * ro.ravel()])


@pytest.mark.parametrize("N,n", [(2, 11), (3, 11), (4, 9), (5, 9), (6, 9), (7, 7)])
@pytest.mark.parametrize("M,s", [(1, 0), (2, 2), (3, 4)])
def test_elastic_stage(N, n, M, s):
    v, e = mesh(n)
    rng = np.random.default_rng(200 * N + M)
    Np, Mp = (N + 1) * (N + 2) * (N + 3) // 6, (M + 1) * (M + 2) * (M + 3) // 6
    media = [rounded(rng, 0.5, 1.5, (len(e), Mp)) for _ in range(3)]
    q, r = (rounded(rng, -1, 1, (9, len(e), Np)) for _ in range(2))
    a, b = (stage(p, v, e, N, M, media, q, r, s) for p in (B.F32, B.F64))
    assert rel_l2(a, b) <= 1e-5


@pytest.mark.parametrize("N,M,n", [(2, 0, 15), (2, 1, 12), (2, 2, 12), (3, 0, 11), (4, 0, 11), (5, 0, 9), (6, 0, 10), (7, 0, 7)])
def test_elastic_step(N, M, n):
    """Constant media, and the media degrees of N = 2 above their own switching sizes; five stages in turn, whose error is at
    most the five stages', each below the stage's bound."""
    v, e = mesh(n)
    assert len(e) >= B.lib().bbw_internal_lane_min(1, N, M, 32)
    rng = np.random.default_rng(300 * N + M)
    Np, Mp = (N + 1) * (N + 2) * (N + 3) // 6, (M + 1) * (M + 2) * (M + 3) // 6
    media = [rounded(rng, 0.5, 1.5, (len(e), Mp)) for _ in range(3)]
    q = rounded(rng, -1, 1, (9, len(e), Np))
    out = []
    for prec in (B.F32, B.F64):
        with B.ElasticSolver(v, e, N, M, prec) as solver:
            solver.set_media(*media)
            solver.set_state(q)
            solver.step(1e-4, 1)
            out.append(solver.get_state()[0])
    assert rel_l2(*out) <= 5e-5
