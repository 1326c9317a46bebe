"""Sums along the axis on both sides of the sizes at which the number of pencils per thread changes: 152 blocks of 256 threads
with two pencils each (one per SM), 304, 456 and 608, with pencil counts that leave threads a part of their pencils."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [2431, 2433, 3001, 4863, 4865, 7295, 7297, 9727, 9729])
@pytest.mark.parametrize("L,m", [(16, 6), (5, 8), (9, 1)])
def test_sums_at_every_split(P, L, m):
    from paper_1808_08645_gb300 import surrogate as S
    C = 32
    rng = np.random.default_rng(P)
    f32 = dict(dtype=torch.float32, device="cuda")
    basis, x = (rng.standard_normal(s).astype(np.float32) for s in ((L, m), (P, L, C)))
    out = torch.full((P + 1, m, C), float("nan"), **f32)
    S.axis(torch.tensor(basis, **f32), L, m, torch.tensor(x, **f32), out, P, C)
    got = out.double().cpu().numpy()
    assert np.isnan(got[P]).all()
    b64, x64 = basis.astype(np.float64), x.astype(np.float64)
    # L products and sums in FP32, each rounded once
    bound = (L + 1) * 2.0**-24 * np.einsum("zk,pzc->pkc", abs(b64), abs(x64))
    assert (abs(got[:P] - np.einsum("zk,pzc->pkc", b64, x64)) <= 1.01 * bound).all()
