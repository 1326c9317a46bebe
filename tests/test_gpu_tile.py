"""The acoustic tile kernels (one element per lane, chosen by size and degree) perform the operations of the team kernels in
their order. A batch bucket goes by its total size and a solo solver by its own, so instances that run the tile kernels in
the bucket and the team kernels alone (and padded sizes that leave a ragged last tile) must agree bit by bit: no tolerance.
Degrees whose solo solvers run the tile kernels at every size are compared with the FP64 solver instead, to the parity
tests' bound of an FP32 stage (1e-5) over a few steps from a random state.
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


def rounded(rng, lo, hi, shape):
    return rng.uniform(lo, hi, shape).astype(np.float32).astype(np.float64)


def case(n, N, M, seed):
    v, e = inputs.cube_mesh(n, jitter=0.1, shuffle=True, seed=seed)
    rng = np.random.default_rng(seed)
    Np, Mp = (N + 1) * (N + 2) * (N + 3) // 6, (M + 1) * (M + 2) * (M + 3) // 6
    return v, e, rounded(rng, 0.5, 2.0, (len(e), Mp)), rounded(rng, -1, 1, (4, len(e), Np))


# hexes per side of three instances: two small ones, and one that takes the bucket over its degree's switching size
@pytest.mark.parametrize("prec,N,ns", [(32, 2, (3, 5, 12)), (32, 3, (3, 5, 12)), (32, 6, (3, 5, 24)), (64, 2, (3, 5, 9)),
                                       (64, 3, (3, 5, 9)), (64, 5, (3, 5, 10))])
@pytest.mark.parametrize("M", [0, 1, 3])
def test_tile_and_team_bits(prec, N, ns, M):
    insts = [case(n, N, M, 10 * N + n) for n in ns]
    amp = np.linspace(100.0, 300.0, 10)
    with B.Batch([(v, e) for v, e, _, _ in insts], [N] * 3, M, prec) as b:
        b.set_params(0.7, 1.3)
        for i, (v, e, c2, q) in enumerate(insts):
            b.set_c2(i, c2)
            b.set_state(i, q)
            b.set_point_source(i, [0.4, 0.5, 0.6], amp)
        dts, steps = np.array([1e-3, 2e-3, 5e-4]), np.array([2, 1, 2])
        b.set_instance_steps(dts, steps)
        b.step(1e-3, 2)
        b.sync()
        got = [b.get_state(i, with_res=True) for i in range(3)]
    for i, (v, e, c2, q) in enumerate(insts[:2]):
        with B.Solver(v, e, N, M, prec) as s:
            s.set_c2(c2)
            s.set_params(0.7, 1.3)
            s.set_state(q)
            s.set_point_source([0.4, 0.5, 0.6], amp)
            s.step(dts[i], int(steps[i]))
            qs, rs, _ = s.get_state(with_res=True)
        assert np.array_equal(got[i][0], qs) and np.array_equal(got[i][1], rs)


@pytest.mark.parametrize("N,n", [(1, 3), (1, 7), (4, 3), (4, 7), (5, 3), (5, 7)])
@pytest.mark.parametrize("M", [0, 1, 2, 3])
def test_tile_against_fp64(N, n, M):
    v, e, c2, q = case(n, N, M, 7 * N + n)
    out = []
    for prec in (B.F32, B.F64):
        with B.Solver(v, e, N, M, prec) as s:
            s.set_c2(c2)
            s.set_state(q)
            s.set_forcing([0, len(e) // 2, len(e) - 1], np.ones((3, s.Np)), np.linspace(100.0, 300.0, 10))
            s.step(1e-3, 2)
            out.append(s.get_state()[0])
    assert rel_l2(out[0], out[1]) <= 1e-5
