"""Host checks of the key projection's entry points: what the host can see is returned
before the prototype fold is enqueued (fake, never-dereferenced addresses)."""
import ctypes

import pytest

from paper_2609_08443_gb300 import binding, build

vp = ctypes.c_void_p


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load()


def fwd(lib, X=256, cu=768, Q=1024, Wk=2048, scale=0.125, sketch=4096):
    n = lib.sa_launch_count()
    st = lib.sa_sketch_fwd_x(vp(X), vp(cu), 2, 100, vp(Q), vp(Wk), 2, 64, 64, scale, 1, vp(sketch), None, vp(1 << 20),
                             1 << 30, None)
    assert lib.sa_launch_count() == n
    return st


def bwd(lib, X=256, cu=768, Q=1024, Wk=2048, scale=0.125, dsketch=4096, dX=8192):
    n = lib.sa_launch_count()
    st = lib.sa_sketch_bwd_x(vp(X), vp(cu), 2, 100, vp(Q), vp(Wk), 2, 64, 64, scale, 1, vp(dsketch), None, vp(dX),
                             vp(16384), vp(32768), vp(1 << 20), 1 << 30, None)
    assert lib.sa_launch_count() == n
    return st


@pytest.mark.parametrize("bad", [dict(X=256 + 2), dict(cu=0), dict(scale=float("inf"))], ids=str)
def test_refused_before_the_fold(lib, bad):
    assert fwd(lib, **bad) == 1
    assert bwd(lib, **bad) == 1


def test_null_outputs(lib):
    assert fwd(lib, sketch=0) == 1
    assert bwd(lib, dsketch=0) == 1
    assert bwd(lib, dX=0) == 1
