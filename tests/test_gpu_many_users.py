"""As many (user, head) pairs as an int holds, nearly all without tokens (34 GB of sketch):
the CUDA-core kernels launch a block per tile there can be, not per user."""
import pytest
import torch

from paper_2609_08443_gb300 import binding

pytestmark = pytest.mark.gpu


def test_users_without_tokens_need_no_blocks(cuda_lib):
    B, H, P, d = 2**25 - 1, 64, 1, 4
    cu = torch.zeros(B + 1, dtype=torch.int32, device="cuda")
    cu[1000:] = 5
    cu[B // 2:] = 40
    cu[B:] = 64
    K, V = torch.randn(64, H, d, device="cuda"), torch.randn(64, H, d, device="cuda")
    Q = torch.randn(H, P, d, device="cuda")
    sketch, lse = binding.sa_sketch_fwd(K, V, cu, Q, 0.5, want_lse=True)
    # one prototype: every weight is 1, the lse is the score
    assert torch.allclose(lse, 0.5 * (K * Q[:, 0]).sum(2), rtol=1e-4, atol=1e-5)
    for user, rows in ((999, slice(0, 5)), (B // 2 - 1, slice(5, 40)), (B - 1, slice(40, 64))):
        assert torch.allclose(sketch[user, :, 0], V[rows].sum(0), rtol=1e-4, atol=1e-4)
        sketch[user] = 0
    flat = sketch.view(-1)
    assert not any(bool(x.any()) for x in flat.split(2**28))
    del sketch, flat
    torch.cuda.empty_cache()
