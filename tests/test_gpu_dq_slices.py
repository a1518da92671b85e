"""The dQ slices (csrc/sa_tc_bwd_dq.cu) where their two 64-token halves and their
per-token terms can go wrong: users that end on either side of a half, odd token
offsets (the bulk copy of (lse, D) starts on an even one), many heads, large and
tiny scales, against the fp64 oracle.

Tolerance: the suite's 2e-2 of max|oracle|.
"""
import numpy as np
import pytest
import torch

import harness
from oracle import sa_backward
from paper_2609_08443_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu

LENS = [1, 63, 64, 65, 0, 127, 129, 191, 1, 700, 1333]


@pytest.mark.parametrize("P,d,H", [(256, 128, 3), (512, 128, 2), (512, 64, 3), (1024, 128, 1), (2048, 64, 1)],
                         ids=lambda x: str(x))
def test_half_edges(cuda_lib, P, d, H):
    harness.check_spec(wl.custom(LENS, H=H, P=P, d=d, dtype=wl.BF16, seed=P + d + H), bwd=True)


@pytest.mark.parametrize("scale", [0.0, 1e-33, 1e-6, 2.0])
def test_scales(cuda_lib, scale):
    spec = wl.custom(LENS, H=2, P=512, d=64, dtype=wl.BF16, seed=77, q_std=0.3)
    host = wl.make_host(spec)
    t = wl.host_to_torch(spec, host, torch.device("cuda"))
    args = (t["K"], t["V"], t["cu_seqlens"], t["Q"])
    _, lse = binding.sa_sketch_fwd(*args, scale, want_lse=True)
    _, _, dQ = binding.sa_sketch_bwd(*args, t["dsketch"], scale, lse=lse)
    K, V, Q = (wl.host_as_f64(spec, host[k]) for k in ("K", "V", "Q"))
    _, _, ref = sa_backward(K, V, host["cu_seqlens"], Q, scale, host["dsketch"].astype(np.float64))
    got = wl.torch_as_f64(dQ)
    if scale < 1e-30:  # below the fp32 range of s dS^T K
        assert np.all(np.isfinite(got)) and np.max(np.abs(got - ref)) <= 1e-28
    else:
        harness.assert_close("dQ", got, ref, harness.TOL[wl.BF16])
