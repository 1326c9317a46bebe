"""Axis transform on both basis layouts in shared memory: rows padded to eight
modes while they fit 48 KB, unpadded beyond, odd pencil counts on either."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# L = 1536 is the last padded size at eight modes; 1537 x 7 and 2048 x 6 are unpadded
@pytest.mark.parametrize("P,L,m,C", [(3, 1536, 8, 5), (5, 1537, 7, 3), (3, 2048, 6, 4), (7, 13, 5, 33), (2, 17, 1, 1)])
def test_axis_transform_padded_and_unpadded_rows(P, L, m, C):
    from paper_1808_08645_gb300 import surrogate as S
    rng = np.random.default_rng(5)
    f32 = dict(dtype=torch.float32, device="cuda")
    basis = rng.standard_normal((L, m)).astype(np.float32)
    x = rng.standard_normal((P, L, C)).astype(np.float32)
    t = rng.standard_normal((P, m, C)).astype(np.float32)
    out = torch.full((P, m, C), float("nan"), **f32)
    S.axis(torch.tensor(basis, **f32), L, m, torch.tensor(x, **f32), out, P, C)
    b64, x64, t64 = (a.astype(np.float64) for a in (basis, x, t))
    # L (or m) products and sums in FP32, each rounded once: |error| <= n 2^-24 sum |w u| (to first order)
    bound = (L + 1) * 2.0**-24 * np.einsum("zk,pzc->pkc", abs(b64), abs(x64))
    assert (abs(out.double().cpu().numpy() - np.einsum("zk,pzc->pkc", b64, x64)) <= 1.01 * bound).all()
    o = torch.full((P, L, C), float("nan"), **f32)
    S.axis(torch.tensor(basis, **f32), L, m, torch.tensor(t, **f32), o, P, C, expand=1)
    bound = (m + 1) * 2.0**-24 * np.einsum("zk,pkc->pzc", abs(b64), abs(t64))
    assert (abs(o.double().cpu().numpy() - np.einsum("zk,pkc->pzc", b64, t64)) <= 1.01 * bound).all()
