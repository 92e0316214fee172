"""FP32 spreading's integer sums: tiles whose records crowd a few cells (batches
of a quantum each) and tiles with one quantum, at magnitudes where the quantum
underflows or the values are not finite, whole and split over CTAs."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1308_6644_gb300 as pkg
    return pkg


def _solve(P, n, pitch, x, y, c, tile, chunk):
    import torch
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.01, tile=tile, spread_chunk=chunk),
                        torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    try:
        u = torch.zeros(n * n, dtype=torch.complex64, device="cuda")
        P.nuasm1_execute(plan, torch.from_numpy(c.astype(np.complex64)).cuda(), u)
        torch.cuda.synchronize()
        return u.cpu().numpy()
    finally:
        plan.destroy()


@pytest.mark.parametrize("tile,chunk", [(16, 0), (16, 64), (32, -1), (64, 0)])
@pytest.mark.parametrize("crowd", [0, 40, 3000])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e30])
def test_one_quantum_or_batches(P, tile, chunk, crowd, scale):
    """300 scattered records and `crowd` in one cell (3000: above the load a
    single quantum serves), 1e-5 as every FP32 solve."""
    n, pitch = 64, 10e-6
    rng = np.random.default_rng(91)
    h = 0.5 * n * pitch * (1 - 1e-9)
    x = np.concatenate([rng.uniform(-h, h, 300), 33e-6 + rng.uniform(0, 1e-6, crowd)])
    y = np.concatenate([rng.uniform(-h, h, 300), -57e-6 + rng.uniform(0, 1e-6, crowd)])
    c = rng.normal(size=len(x)) + 1j * rng.normal(size=len(x))
    got = _solve(P, n, pitch, x, y, c * scale, tile, chunk)
    ref = O.nuasm1(x, y, (c * scale).astype(np.complex64) / scale, dict(n=n, pitch=pitch, lam=633e-9, z=0.01))
    assert O.rel_l2(got.astype(np.complex128) / scale, ref.ravel()) < 1e-5


@pytest.mark.parametrize("crowd", [0, 3000])
def test_values_that_are_not_finite_propagate(P, crowd):
    n, pitch = 64, 10e-6
    rng = np.random.default_rng(92)
    x = np.concatenate([rng.uniform(-3e-4, 3e-4, 200), np.full(crowd, 1e-5)])
    y = np.concatenate([rng.uniform(-3e-4, 3e-4, 200), np.full(crowd, 1e-5)])
    for bad in (np.inf, np.nan):
        c = np.ones(len(x), np.complex64)
        c[-1] = bad
        assert not np.isfinite(_solve(P, n, pitch, x, y, c, 16, 0)).all()
