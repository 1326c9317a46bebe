"""Every degree that has both kinds of acoustic kernels, at every media degree: an instance runs the team kernels alone (its own
size is below the switch) and the tile kernels in a batch (the bucket's size is above), and the results are the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_08645_gb300 import binding as B  # noqa: E402
from paper_1808_08645_gb300 import inputs  # noqa: E402
from parity_util import rounded  # noqa: E402

np3 = lambda n: (n + 1) * (n + 2) * (n + 3) // 6  # noqa: E731


def lane_min(N, M, prec):
    return B.lib().bbw_internal_lane_min(0, N, M, prec)


@pytest.mark.parametrize("prec,N", [(32, 1), (32, 2), (32, 3), (32, 6), (64, 2), (64, 3), (64, 5)])
@pytest.mark.parametrize("M", [0, 1, 2, 3])
def test_the_two_kernels_give_the_same_bits(prec, N, M):
    switch = lane_min(N, M, prec)
    if switch == 0:
        pytest.skip("the tile kernels at every size")
    small = inputs.cube_mesh(5, jitter=0.1, shuffle=True, seed=N)
    big = inputs.cube_mesh(int(np.ceil((switch / 6) ** (1 / 3))), seed=0)
    K = len(small[1])
    assert K < switch <= len(big[1])
    rng = np.random.default_rng(40 * N + M)
    c2 = rounded(rng.uniform(0.5, 2.0, (K, np3(M))), 32)
    q, r = (rounded(rng.uniform(-1, 1, (4, K, np3(N))), 32) for _ in range(2))
    amp = np.linspace(100.0, 300.0, 10)
    # the padding and the instance before it put the instance's elements on ragged tiles
    with B.Batch([(small[0], small[1][:7]), small, big], [N] * 3, M, prec) as b:
        b.set_params(0.7, 1.3)
        b.set_c2(1, c2)
        b.set_state(1, q, r)
        b.set_point_source(1, [0.4, 0.5, 0.6], amp)
        b.step(1e-3, 2)
        b.sync()
        got = b.get_state(1, with_res=True)
    with B.Solver(*small, N, M, prec) as s:
        s.set_params(0.7, 1.3)
        s.set_c2(c2)
        s.set_state(q, r)
        s.set_point_source([0.4, 0.5, 0.6], amp)
        s.step(1e-3, 2)
        want = s.get_state(with_res=True)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_the_rule():
    """Degrees above 6 (5 in FP64) have the team kernels alone, N = 4 the tile kernels alone."""
    assert all(lane_min(N, M, 32) == 2**63 - 1 for N in (7, 8, 9) for M in range(4))
    assert all(lane_min(N, M, 64) == 2**63 - 1 for N in (6, 7, 8, 9) for M in range(4))
    assert all(lane_min(4, M, p) == 0 for M in range(4) for p in (32, 64))
