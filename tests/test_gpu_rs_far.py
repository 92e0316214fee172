"""FP32 direct sum: pairs whose path difference is so many wavelengths that FP32
holds no phase, beside pairs that it resolves."""
import numpy as np
import pytest

import oracle as O
from test_gpu_rs import rs_gpu

pytestmark = pytest.mark.gpu

LAM, Z = 500e-9, 8e-3


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1308_6644_gb300 as pkg
    return pkg


@pytest.mark.parametrize("far", [1.2, 14.0, 1e3, 1e8])
@pytest.mark.parametrize("m1", [300, 2000])
def test_far_sources_beside_near_ones(P, m1, far):
    """50 sources of a tenth the amplitude at `far` (path differences of 2^21
    wavelengths and more) among m1 near ones: theirs is at most 0.1 z^2 / r^2 =
    4.4e-6 of a near one's share, so the FP32 bound of 1e-5 holds whatever their
    phases."""
    rng = np.random.default_rng(64)
    x1, y1 = rng.uniform(-1e-4, 1e-4, m1), rng.uniform(-1e-4, 1e-4, m1)
    t = rng.uniform(0, 2 * np.pi, 50)
    at = rng.choice(m1, 50, replace=False)
    x1[at], y1[at] = far * np.cos(t), far * np.sin(t)
    c = (rng.normal(size=m1) + 1j * rng.normal(size=m1)).astype(np.complex64)
    c[at] *= 0.1
    area = rng.uniform(0.5, 1.5, m1) * 1e-11
    x2, y2 = rng.uniform(-1e-4, 1e-4, 130), rng.uniform(-1e-4, 1e-4, 130)
    got = rs_gpu(P, "f32", x1, y1, c, area, x2, y2, LAM, Z)
    assert O.rel_l2(got, O.rs_direct(x1, y1, c, area, x2, y2, LAM, Z)) < 1e-5


@pytest.mark.parametrize("far", [1.2, 14.0, 1e3, 1e8])
def test_far_points_keep_their_magnitude(P, far):
    """Far from everything the phases are lost, the magnitudes are not: no sum
    exceeds that of its terms' magnitudes (1 + 1e-5: the FP32 bound)."""
    rng = np.random.default_rng(65)
    x1, y1 = rng.uniform(-1e-4, 1e-4, 400), rng.uniform(-1e-4, 1e-4, 400)
    t = rng.uniform(0, 2 * np.pi, 70)
    x2, y2 = far * np.cos(t), far * np.sin(t)
    x2[::7], y2[::7] = x2[::7] * 1e-5, y2[::7] * 1e-5   # and some near ones
    c = (rng.normal(size=400) + 1j * rng.normal(size=400)).astype(np.complex64)
    area = rng.uniform(0.5, 1.5, 400) * 1e-11
    got = rs_gpu(P, "f32", x1, y1, c, area, x2, y2, LAM, Z)
    r = np.sqrt((x2[:, None] - x1) ** 2 + (y2[:, None] - y1) ** 2 + Z * Z)
    top = (np.abs(c) * area * (Z / r) * np.hypot(1, 2 * np.pi / LAM * r) / (2 * np.pi * r * r)).sum(axis=1)
    assert (np.abs(got) <= top * (1 + 1e-5)).all()
    assert got.any()
