"""fp32 scores beyond the range: a score of +inf gives its token the lse of
torch.logsumexp, +inf, and takes the token out of the other prototypes' sums; one of -inf
is no weight; a NaN reaches the token's lse.

Expected values in 64 bits from the finite tokens; tolerance 1e-4 of the largest, as for
fp32 elsewhere.
"""
import numpy as np
import pytest
import torch

from paper_2609_08443_gb300 import binding

pytestmark = pytest.mark.gpu

N, d = 70, 16


def make(P, j, q):
    g = torch.Generator().manual_seed(P + j)
    K, V = torch.randn(N, 1, d, generator=g), torch.randn(N, 1, d, generator=g)
    Q = torch.randn(1, P, d, generator=g)
    K[33, 0, 0], Q[0, :, 0], Q[0, j, 0] = 1e30, 0., q
    return K, V, Q


def run(K, V, Q):
    cu = torch.tensor([0, N], dtype=torch.int32, device="cuda")
    sketch, lse = binding.sa_sketch_fwd(K.cuda(), V.cuda(), cu, Q.cuda(), 1.0, want_lse=True)
    return sketch[0, 0].double().cpu(), lse[:, 0].double().cpu()


@pytest.mark.parametrize("P,j", [(1, 0), (2, 1), (20, 19), (64, 3), (200, 150)], ids=str)
@pytest.mark.parametrize("q,want", [(1e30, np.inf), (-1e30, None), (float("nan"), np.nan)], ids=["inf", "-inf", "nan"])
def test_one_score(cuda_lib, P, j, q, want):
    K, V, Q = make(P, j, q)
    sketch, lse = run(K, V, Q)
    k, v = K[:, 0].double(), V[:, 0].double()
    s = k @ Q[0].double().T
    if q != q:  # the prototype's scores are NaN for every token
        assert torch.isnan(lse).all()
        return
    s[33, j] = np.inf if q > 0 else -np.inf
    ref = torch.logsumexp(s, 1)
    keep = torch.arange(N) != 33 if q > 0 or P == 1 else torch.ones(N, dtype=torch.bool)
    assert torch.allclose(lse[keep], ref[keep], rtol=1e-4, atol=1e-4)
    if q > 0 or P == 1:
        assert lse[33] == (np.inf if q > 0 else -np.inf)
    w = torch.exp(s[keep] - ref[keep, None])
    out = w.T @ v[keep]
    rows = torch.arange(P) != j if q > 0 or P == 1 else torch.ones(P, dtype=torch.bool)
    assert (sketch[rows] - out[rows]).abs().max() <= 1e-4 * out.abs().max() if rows.any() else True


def test_two_infinite_scores(cuda_lib):
    K, V, Q = make(90, 5, 1e30)
    Q[0, 80, 0] = 1e30
    sketch, lse = run(K, V, Q)
    assert lse[33] == np.inf
    assert torch.isfinite(sketch[[i for i in range(90) if i not in (5, 80)]]).all()
