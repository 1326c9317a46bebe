"""Instances of a batch that have used up their step budgets cost one copy per stage, on the tile kernels as on the team
kernels: a step in which a large finished instance rides beside a small live one takes well under the large one's own step.

The copy reads and writes q once; a stage reads and writes q and res, gathers traces and computes: at least 2.5 times the
copy's bytes. The bound (half the live step's time) leaves room for the launches of the small instance.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_08645_gb300 import binding as B  # noqa: E402
from paper_1808_08645_gb300 import inputs  # noqa: E402


def step_ms(b, stream, budgets):
    b.set_instance_steps(None, budgets)
    b.step(1e-6, 2)  # both parities' graphs
    best = float("inf")
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        b.step(1e-6, 4)
        e1.record(stream)
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1) / 4)
    return best


# the tile kernels with the projection inside (FP32, FP64) and apart (N = 6); N = 7 runs the team kernel
@pytest.mark.parametrize("prec,N,n", [(32, 5, 22), (64, 4, 16), (32, 6, 24), (32, 7, 16)])
def test_finished_instances_cost_a_copy(prec, N, n):
    stream = torch.cuda.Stream()
    big, small = inputs.cube_mesh(n), inputs.cube_mesh(2)
    with B.Batch([big, small], [N, N], 2, prec, stream=stream.cuda_stream) as b:
        q = np.random.default_rng(1).uniform(-1, 1, (4, len(big[1]), b.np_(0)))
        b.set_state(0, q)
        live = step_ms(b, stream, np.array([10**9, 10**9]))
        before = b.get_state(0)
        done = step_ms(b, stream, np.array([0, 10**9]))
        assert np.array_equal(b.get_state(0), before)
    assert done <= 0.5 * live, (done, live)
