"""sin and cos without branches (sincos_g), which every rollout's steps use, have
the bits of the form with them (sincos_r), whose accuracy test_gpu_math.py
bounds and which the adjoint takes at the rollout's recorded angles:
atp_math_check gives NaN where the two differ.  Around every quadrant's edge, up
to the end of the reduction's range and beyond, both signs, zeros, denormals,
infinities and NaN."""
import numpy as np
import pytest

from test_gpu_math import run

pytestmark = pytest.mark.gpu


def around(x):
    x = np.asarray(x, np.float32)
    lo, hi = np.nextafter(x, np.float32(-np.inf)), np.nextafter(x, np.float32(np.inf))
    return np.concatenate([x, lo, hi, np.nextafter(lo, np.float32(-np.inf)), np.nextafter(hi, np.float32(np.inf))])


def test_both_forms_have_the_same_bits():
    rng = np.random.default_rng(2)
    k = np.concatenate([np.arange(1, 4001), rng.integers(4001, 166886, 20000)])
    edges = around((k * (np.pi / 4)).astype(np.float32))          # up to 131072
    top = around(np.array([131072.0, 1e6, 3.4e38], np.float32))
    small = np.array([0.0, 1e-45, 1e-40, 1e-30, 1e-8, 0.785398163], np.float32)
    wide = np.exp(rng.uniform(np.log(1e-6), np.log(2e5), 200000)).astype(np.float32)
    a = np.concatenate([edges, top, small, wide])
    a = a[np.isfinite(a)]
    a = np.concatenate([a, -a])
    o = run(a, np.ones_like(a))
    assert not np.any(np.isnan(o[:, :4]))
    o = run(np.array([np.inf, -np.inf, np.nan, -np.nan], np.float32), np.ones(4, np.float32))
    assert np.all(np.isnan(o[:, :4]))
