"""FP32 spreading where one sample, or a few, outshine a dense tile's others: the
integer sums' quantum follows the tile's values, not its largest one alone."""
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


@pytest.mark.parametrize("tile,chunk", [(16, -1), (16, 0), (32, -1), (32, 0), (64, 0)])
@pytest.mark.parametrize("count", [2700, 9000, 22500])
@pytest.mark.parametrize("every", [0, 300])
def test_bright_samples_among_faint_ones(P, tile, chunk, count, every):
    """`count` samples over 30 x 30 fine-grid cells (loads of about 30, 100 and
    250), of magnitude 1e-3 but one, or one in 300, of magnitude 1.  A solve is
    linear and so are the kernel's own errors, so the solve of the sum differs
    from the sum of the bright and the faint samples' solves by roundings alone:
    1e-6 for the three of them, 16 units of 2^-24."""
    import torch
    n, pitch = 64, 10e-6
    rng = np.random.default_rng(93)
    x, y = (torch.from_numpy(rng.uniform(-7.5, 7.5, count) * pitch).cuda() for _ in range(2))
    phase = np.exp(2j * np.pi * rng.uniform(size=count))
    at = np.zeros(count, bool)
    at[count // 2 if every == 0 else slice(None, None, every)] = True
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.01, tile=tile, spread_chunk=chunk), x, y)
    try:
        def solve(c):
            u = torch.zeros(n * n, dtype=torch.complex64, device="cuda")
            P.nuasm1_execute(plan, torch.from_numpy(c.astype(np.complex64)).cuda(), u)
            torch.cuda.synchronize()
            return u.cpu().numpy().astype(complex)
        bright, faint = np.where(at, phase, 0), np.where(at, 0, 1e-3 * phase)
        assert O.rel_l2(solve(bright + faint), solve(bright) + solve(faint)) < 1e-6
    finally:
        plan.destroy()


@pytest.mark.parametrize("tile,chunk", [(16, -1), (32, 64), (64, 0)])
def test_batches_that_hold_no_values(P, tile, chunk):
    """A dense tile whose first and last records are zero, one whose values all are."""
    import torch
    n, pitch, count = 64, 10e-6, 9000
    rng = np.random.default_rng(94)
    x, y = (torch.from_numpy(rng.uniform(-7.5, 7.5, count) * pitch).cuda() for _ in range(2))
    c = np.zeros(count, np.complex64)
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.01, tile=tile, spread_chunk=chunk), x, y)
    try:
        u = torch.full((n * n,), 7 + 7j, dtype=torch.complex64, device="cuda")
        P.nuasm1_execute(plan, torch.from_numpy(c).cuda(), u)
        torch.cuda.synchronize()
        assert not u.cpu().numpy().any()
        c[4000:5000] = 1e-4
        c[4500] = 1
        P.nuasm1_execute(plan, torch.from_numpy(c).cuda(), u)
        torch.cuda.synchronize()
        ref = O.nuasm1(x.cpu().numpy(), y.cpu().numpy(), c, dict(n=n, pitch=pitch, lam=633e-9, z=0.01))
        assert O.rel_l2(u.cpu().numpy(), ref.ravel()) < 1e-5
    finally:
        plan.destroy()


@pytest.mark.parametrize("tile", [16, 64])
def test_a_bright_sample_that_is_not_finite(P, tile):
    import torch
    n, pitch, count = 64, 10e-6, 9000
    rng = np.random.default_rng(95)
    x, y = (torch.from_numpy(rng.uniform(-7.5, 7.5, count) * pitch).cuda() for _ in range(2))
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.01, tile=tile), x, y)
    try:
        for bad in (np.inf, np.nan, complex(np.nan, 1), complex(0, -np.inf)):
            c = np.full(count, 1e-3, np.complex64)
            c[7000] = bad
            u = torch.zeros(n * n, dtype=torch.complex64, device="cuda")
            P.nuasm1_execute(plan, torch.from_numpy(c).cuda(), u)
            torch.cuda.synchronize()
            assert not np.isfinite(u.cpu().numpy()).all()
    finally:
        plan.destroy()
