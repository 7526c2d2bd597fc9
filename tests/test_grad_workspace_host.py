"""The adjoint's workspace: `ckpt` bounds it, the whole trace is kept where that
allows it, and the segments cover the horizon."""
import ctypes as C

import pytest

from paper_2603_20525_gb300 import atp


class GradPlan(C.Structure):
    _fields_ = [("seg", C.c_int), ("n_seg", C.c_int)] + [(n, C.c_size_t) for n in
                                                         ("rec", "ckpt", "fin", "lam", "ints", "total")]


@pytest.fixture(scope="module")
def grad_plan():
    f = getattr(atp.load(), "_ZN3atp9grad_planEiiii")
    f.argtypes, f.restype = [C.c_int] * 4, GradPlan
    return f


MIB = 1 << 20


@pytest.mark.parametrize("K", [1, 64, 4096, 7297, 16384, 131072, 1 << 21, 1 << 28])
@pytest.mark.parametrize("H,n_sub", [(1, 1), (7, 3), (100, 4), (101, 20), (1000, 1), (150, 50)])
def test_workspace(grad_plan, K, H, n_sub):
    for ckpt in sorted({min(c, H) for c in (1, 2, 5, 7, 10, 31, 100, H)}):
        g = grad_plan(K, H, n_sub, ckpt)
        one, two = (320 * (-(-H // ckpt) + b * ckpt * n_sub) for b in (1, 2))
        bound = max(one, min(two, (16 << 10) * MIB // K))
        small = 64 * H * n_sub * K <= 128 * MIB
        assert g.total <= (max(bound * K, 128 * MIB + 24 * K) if small else bound * K) + 2048
        assert (g.n_seg - 1) * g.seg < H <= g.n_seg * g.seg
        if small or 64 * H * n_sub + 24 <= bound:
            assert g.n_seg == 1
        if g.n_seg > 1:
            # one segment fewer would not have fitted
            seg = -(-H // (g.n_seg - 1))
            assert 64 * seg * n_sub + 24 + (0 if g.n_seg == 2 else 64 + 80 * (g.n_seg - 1)) > bound
        sizes = [64 * g.seg * n_sub * K, 80 * g.n_seg * K if g.n_seg > 1 else 0, 16 * K, 64 * K if g.n_seg > 1 else 0, 8 * K]
        at = [g.rec, g.ckpt, g.fin, g.lam, g.ints, g.total]
        assert all(a % 256 == 0 and a + n <= e for a, n, e in zip(at, sizes, at[1:]))


def test_a_caller_can_ask_for_less(grad_plan):
    """16384 candidates of 400 steps: 419 MB for the whole trace at the default
    interval, 214 MB at a shorter one."""
    assert grad_plan(16384, 100, 4, 10).n_seg == 1
    assert grad_plan(16384, 100, 4, 4).total < 215e6
