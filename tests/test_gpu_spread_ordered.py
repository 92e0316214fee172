"""FP32 spreading of ordered points on tiles of side 16: warp-private copies where no
warp takes two records of one cell together, the integer sums elsewhere."""
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


def _points(kind, n, pitch, density):
    k = int(n * density)
    h = 0.5 * n * pitch
    g = (np.arange(k) + 0.3) * (2 * h / k) - h
    y, x = (v.ravel() for v in np.meshgrid(g, g, indexing="ij"))
    if kind == "repeated":     # one cell twice: the warps that meet there
        x, y = np.append(x, x[k]), np.append(y, y[k])
    elif kind == "shuffled":
        p = np.random.default_rng(96).permutation(len(x))
        x, y = x[p], y[p]
    return x, y


def _solve(P, n, pitch, x, y, c, w, **kw):
    import torch
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.01, **kw), *(torch.from_numpy(v).cuda() for v in (x, y)),
                        None if w is None else torch.from_numpy(w).cuda())
    try:
        u = torch.full((n * n,), 5 - 5j, dtype=torch.complex64, device="cuda")
        P.nuasm1_execute(plan, torch.from_numpy(c).cuda(), u)
        torch.cuda.synchronize()
        return u.cpu().numpy()
    finally:
        plan.destroy()


# tiles of side 16: up to 304 (n <= 128) and more, of up to 128 records and more
@pytest.mark.parametrize("kind", ["lattice", "repeated", "shuffled"])
@pytest.mark.parametrize("n,density", [(16, 1.0), (32, 0.7), (64, 2.0), (128, 1.0), (256, 1.0), (256, 1.9)])
@pytest.mark.parametrize("weighted", [False, True])
def test_ordered_points(P, kind, n, density, weighted):
    """Against tiles of side 32, which always take the integer sums (equal to
    roundings: 1e-6), and on small planes against the oracle (1e-5)."""
    pitch, rng = 10e-6, np.random.default_rng(97)
    x, y = _points(kind, n, pitch, density)
    c = (rng.normal(size=len(x)) + 1j * rng.normal(size=len(x))).astype(np.complex64)
    w = rng.uniform(0.5, 1.5, len(x)) if weighted else None
    got = _solve(P, n, pitch, x, y, c, w, tile=16)
    assert O.rel_l2(got, _solve(P, n, pitch, x, y, c, w, tile=32)) < 1e-6
    if n <= 64:
        ref = O.nuasm1(x, y, c, dict(n=n, pitch=pitch, lam=633e-9, z=0.01), w)
        assert O.rel_l2(got, ref.ravel()) < 1e-5


@pytest.mark.parametrize("tol", [1e-3, 1e-4, 1e-5, 1e-7])
def test_every_width(P, tol):
    n, pitch, rng = 64, 10e-6, np.random.default_rng(98)
    x, y = _points("lattice", n, pitch, 1.0)
    c = (rng.normal(size=len(x)) + 1j * rng.normal(size=len(x))).astype(np.complex64)
    a, b = (_solve(P, n, pitch, x, y, c, None, tile=t, tol=tol) for t in (16, 32))
    assert O.rel_l2(a, b) < 1e-6


@pytest.mark.parametrize("chunk", [-1, 0, 64])
def test_values_that_are_zero_or_not_finite(P, chunk):
    n, pitch = 64, 10e-6
    x, y = _points("lattice", n, pitch, 1.0)
    for bad in (np.inf, np.nan):
        c = np.ones(len(x), np.complex64)
        c[33] = bad
        assert not np.isfinite(_solve(P, n, pitch, x, y, c, None, tile=16, spread_chunk=chunk)).all()
    assert not _solve(P, n, pitch, x, y, np.zeros(len(x), np.complex64), None, tile=16, spread_chunk=chunk).any()
