"""How the tensor-core kernels start (read from their source, no GPU): until the CTA's
barriers and tensor memory are set up, no thread leaves on its own reading of the error
word, which another CTA of the same launch may write at any time."""
import glob
import os
import re

import pytest

from paper_2609_08443_gb300 import build

SOURCES = sorted(glob.glob(os.path.join(build.CSRC, "sa_tc*.cu")))


def setups():
    """(file, text) from each kernel's dynamic shared memory to its TMEM allocation."""
    for path in SOURCES:
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"extern __shared__[^;]*;(.*?)tmem_alloc\(", text, flags=re.S):
            yield os.path.basename(path), m.group(1)


def test_every_kernel_is_looked_at():
    assert sum(1 for _ in setups()) == sum(open(p).read().count("tmem_alloc(") for p in SOURCES) == 7


@pytest.mark.parametrize("where,text", list(setups()), ids=lambda x: x[:16] if x.endswith(".cu") else "")
def test_leaves_as_one_block(where, text):
    assert "cta_leaves(a.ws" in text
    assert "ws_failed" not in text, f"{where}: one thread's reading of the error word"
    for line in (x for x in text.splitlines() if re.search(r"\breturn;", x)):
        assert "cta_leaves(" in line or "!PAIR && skip" in line, f"{where}: {line.strip()}"


@pytest.mark.gpu
@pytest.mark.parametrize("P,d,path", [(128, 64, 0), (256, 64, 0), (256, 128, 2), (512, 64, 0), (512, 128, 0),
                                      (512, 128, 2), (512, 128, 3), (1024, 128, 0)], ids=lambda x: str(x))
def test_failed_call_leaves_and_the_next_is_clean(cuda_lib, P, d, path):
    """Offsets that the planner refuses: every kernel of the call leaves, forward, backward
    and token-wise, and the next call on the same workspace gives the bits of a first one."""
    import torch

    from paper_2609_08443_gb300 import binding, workloads as wl

    spec = wl.custom([700, 0, 129, 3000], H=2, P=P, d=d, dtype=wl.BF16, seed=P + d)
    t = wl.host_to_torch(spec, wl.make_host(spec), torch.device("cuda"))
    N, H, _ = t["K"].shape
    B = t["cu_seqlens"].numel() - 1
    need = max(binding.sa_workspace_size(B, N, H, P, d, binding.SA_BF16, 1),
               binding.load().sa_workspace_size_tokenwise(B, N, H, P, d, binding.SA_BF16, 1))
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")

    def calls(cu):
        a = (t["K"], t["V"], cu, t["Q"])
        yield binding.sa_sketch_fwd(*a, spec.scale, want_lse=True, ws=ws)
        yield binding.sa_sketch_bwd(*a, t["dsketch"], spec.scale, ws=ws)
        yield binding.sa_sketch_fwd_tokenwise(*a, spec.scale, want_lse=True, ws=ws)
        yield binding.sa_sketch_bwd_tokenwise(*a, t["dsketch"], spec.scale, ws=ws)

    try:
        binding.sa_select_path(path)
        want = [[x.clone() for x in out] for out in calls(t["cu_seqlens"])]
        bad = t["cu_seqlens"].clone()
        bad[1] = N  # then falls
        for _ in calls(bad):
            assert binding.sa_get_device_error(ws) == 6
        for out, ref in zip(calls(t["cu_seqlens"]), want):
            assert binding.sa_get_device_error(ws) == 0
            assert all(torch.equal(x, y) for x, y in zip(out, ref))
    finally:
        binding.sa_select_path(0)


def kernels():
    """(file, text) of each tensor-core kernel from its set-up to its TMEM release."""
    for path in SOURCES:
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"extern __shared__[^;]*;(.*?)tmem_dealloc\(", text, flags=re.S):
            yield os.path.basename(path), m.group(1)


@pytest.mark.parametrize("where,text", list(kernels()), ids=lambda x: x[:16] if x.endswith(".cu") else "")
def test_abort_waits_for_every_copy(where, text):
    """A role that gives up waits for its copies in flight: every barrier that a copy into
    shared memory completes has its bounded wait (the peer's pushes, x_full and r_full,
    are no copies of the waiting CTA)."""
    full = set(re.findall(r"mbar_arrive_expect_tx\((\w+)", text)) - {"x_full", "r_full"}
    if "full" in full:  # a streamed block's barrier, one of q_full
        full = full - {"full"} | {"q_full"}
    assert full, where
    assert full <= set(re.findall(r"mbar_wait_bounded\((\w+)", text)), where


def test_slot_parity_stays_that_of_the_last_load():
    text = open(os.path.join(build.CSRC, "sa_tc_bwd.cu")).read()
    load = re.search(r"auto load = .*?used \|= 1u << s;", text, flags=re.S).group(0)
    assert re.search(r"mbar_wait\(empty_bar\(s\)[^;]*;\s*if \(!ok\) return;[^\n]*\n\s*par \^= 1u << s;", load)
