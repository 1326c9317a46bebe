"""Device memory of elastic solvers on the kernels with one element per lane: the face fluxes and one trace beside the state,
and, where not even that fits, the team kernel, which needs no scratch, instead of a refusal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_08645_gb300 import binding as B  # noqa: E402
from paper_1808_08645_gb300 import inputs  # noqa: E402
from parity_util import rel_l2  # noqa: E402


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def state_bytes(K, N, Mp):
    """Three state copies in FP32, the FP64 staging, media, geometry (13 rows) and connectivity."""
    Np = (N + 1) * (N + 2) * (N + 3) // 6
    return K * (4 * (27 * Np + 3 * Mp + 13) + 8 * 9 * Np + 16)


@pytest.mark.parametrize("N", [2, 3, 5, 6, 7])
def test_scratch_is_the_fluxes_and_one_trace(N):
    v, e = inputs.cube_mesh(20)
    K, Np, Nfp = len(e), (N + 1) * (N + 2) * (N + 3) // 6, (N + 1) * (N + 2) // 2
    B.ElasticSolver(v, e, N, 2, 32).close()  # code and tables of the degree are on the device
    before = free()
    with B.ElasticSolver(v, e, N, 2, 32):
        used = before - free()
    # 2 MiB granules for the ten arrays, and two more for the status words and the context
    assert used <= state_bytes(K, N, 10) + 4 * K * (24 * Nfp + Np) + 12 * 2**21


def test_a_mesh_whose_scratch_does_not_fit_runs_on_the_team_kernel():
    N, M = 5, 2
    v, e = inputs.cube_mesh(24)  # 82,944 tets: 167 MB of fluxes, 19 MB of trace
    K, Np = len(e), 56
    rng = np.random.default_rng(0)
    q = rng.uniform(-1, 1, (9, K, Np)).astype(np.float32).astype(np.float64)

    def stage():
        with B.ElasticSolver(v, e, N, M, 32) as s:
            s.set_state(q)
            s.stage(0, 1e-3)
            return s.get_state()[0]

    want = stage()
    torch.cuda.empty_cache()
    hold = torch.empty(free() - state_bytes(K, N, 10) - (80 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = stage()
    finally:
        del hold
        torch.cuda.empty_cache()
    # two FP32 kernels of the same stage, each within 1e-5 of FP64 (the parity tests' bound)
    assert rel_l2(got, want) <= 2e-5
