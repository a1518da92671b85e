"""The key projection's tiled products (csrc/sa_xproj.cu) at sizes that do not
fill their 32 x 32 tiles, and dX summed in the backward's epilogue at the shapes
the other file leaves out, against the fp64 oracle.

Tolerance: the suite's 1e-4 (fp32) and 2e-2 (bf16) of max|oracle|.
"""
import numpy as np
import pytest
import torch

import harness
from oracle import sa_backward_x, sa_forward_x
from paper_2609_08443_gb300 import binding, workloads as wl
from test_gpu_key_projection import _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,d,dt,H", [(1, 8, wl.BF16, 1), (33, 36, wl.F32, 2), (200, 96, wl.BF16, 1),
                                      (512, 64, wl.BF16, 2), (256, 128, wl.BF16, 2), (128, 64, wl.BF16, 3)],
                         ids=lambda x: str(x))
def test_edges(cuda_lib, P, d, dt, H):
    spec, host, t, Wk_host, Wk_t = _case(P, d, dt, H, seed=2 * P + d)
    X, cu_t = t["K"], t["cu_seqlens"]
    sketch, lse = binding.sa_sketch_fwd_x(X, cu_t, t["Q"], Wk_t, spec.scale, want_lse=True)
    dX, dQ, dWk = binding.sa_sketch_bwd_x(X, cu_t, t["Q"], Wk_t, t["dsketch"], spec.scale, lse=lse)
    torch.cuda.synchronize()
    Xf, Qf, Wf = (wl.host_as_f64(spec, a) for a in (host["K"], host["Q"], Wk_host))
    cu = host["cu_seqlens"]
    tol = harness.TOL[spec.dtype]
    harness.assert_close("sketch", wl.torch_as_f64(sketch), sa_forward_x(Xf, cu, Qf, Wf, spec.scale), tol)
    ref = sa_backward_x(Xf, cu, Qf, Wf, spec.scale, host["dsketch"].astype(np.float64))
    for name, got, want in zip(("dX", "dQ", "dWk"), (dX, dQ, dWk), ref):
        if P == 1 and name != "dX":  # one prototype: the weights are 1, so the exact gradient is 0
            want = np.zeros_like(want)
            scale = float(np.max(np.abs(wl.torch_as_f64(dX))))
            assert np.max(np.abs(wl.torch_as_f64(got))) <= tol * scale * X.shape[0]
            continue
        harness.assert_close(name, wl.torch_as_f64(got), want, tol)
