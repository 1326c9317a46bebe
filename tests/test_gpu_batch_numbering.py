"""The numbering of a batch's union mesh does not depend on the kernels that its buckets run: every instance starts at a
multiple of the degree's group width, with detached padding elements in between, and the totals count them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1808_08645_gb300 import binding as B  # noqa: E402
from paper_1808_08645_gb300 import inputs  # noqa: E402

#: elements per group of the team kernels, by precision and degree (1..9)
WIDTH = {32: (2, 2, 4, 4, 4, 2, 2, 2, 2), 64: (2, 2, 2, 2, 1, 1, 1, 1, 1)}


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("N", range(1, 10))
def test_members_start_on_group_boundaries(N, prec):
    """Two meshes of 5 tetrahedra (a cube's) and one of 6: the paddings are inert, also with budgets and steps of their own."""
    w = WIDTH[prec][N - 1]
    v, e = inputs.cube_mesh(1)
    meshes = [(v, e[:5]), (v, e[:5]), (v, e)]
    with B.Batch(meshes, [N] * 3, 1, prec) as b:
        starts = [b.member(i)["first"] for i in range(3)]
        assert starts == [0, -(-5 // w) * w, 2 * -(-5 // w) * w]
        assert b.info()[2] == starts[2] + -(-6 // w) * w
        q = [np.random.default_rng(i).uniform(-1, 1, (4, len(m[1]), b.np_(i))) for i, m in enumerate(meshes)]
        for i in range(3):
            b.set_state(i, q[i])
        b.set_instance_steps(np.array([1e-3, 2e-3, 1e-3]), np.array([2, 1, 2]))
        b.step(1e-3, 2)
        b.sync()
        got = [b.get_state(i) for i in range(3)]
    for i, (dt, n) in enumerate(((1e-3, 2), (2e-3, 1), (1e-3, 2))):
        with B.Solver(*meshes[i], N, 1, prec) as s:
            s.set_state(q[i])
            s.step(dt, n)
            assert np.array_equal(s.get_state()[0], got[i])
