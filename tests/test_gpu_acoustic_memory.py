"""Device memory of acoustic solvers whose projection of p runs apart from the tile kernel: the bracket waits in p's place of
the stage's output and takes no memory of its own."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_08645_gb300 import binding as B  # noqa: E402
from paper_1808_08645_gb300 import inputs  # noqa: E402


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("N,prec", [(6, 32), (5, 64)])
def test_the_bracket_takes_no_memory_of_its_own(N, prec):
    v, e = inputs.cube_mesh(28)
    K, Np, size = len(e), (N + 1) * (N + 2) * (N + 3) // 6, prec // 8
    B.Solver(v, e, N, 2, prec).close()  # code and tables of the degree are on the device
    before = free()
    with B.Solver(v, e, N, 2, prec):
        used = before - free()
    # three states, c^2, geometry, connectivity and the numbering both ways; 2 MiB granules
    assert used <= K * (size * (12 * Np + 10 + 9) + 16 + 16) + 10 * 2**21 < K * size * 13 * Np
