"""The double-float FFT passes' scales (FP64, N' >= 512): strips of columns of
different magnitude, tables far from 1, and no values at all."""
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


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _points(rng, n, pitch, m):
    h = 0.5 * n * pitch * (1 - 1e-9)
    return rng.uniform(-h, h, m), rng.uniform(-h, h, m)


@pytest.mark.parametrize("span", [40, 300])
def test_type2_columns_of_different_magnitude(P, span):
    """Columns scaled by 2^0 .. 2^-span: the solve's scale is the largest strip's."""
    import torch
    n, pitch, m = 256, 5e-6, 500
    rng = np.random.default_rng(81)
    x, y = _points(rng, n, pitch, m)
    u1 = (rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))) * 2.0 ** -rng.integers(0, span, n)[None, :]
    plan = P.nuasm_plan(P.make_params(n, pitch, 500e-9, 8e-3, prec="f64"), _dev(x), _dev(y))
    try:
        v = torch.zeros(m, dtype=torch.complex128, device="cuda")
        P.nuasm2_execute(plan, _dev(u1.ravel()), v)
        torch.cuda.synchronize()
        assert O.rel_l2(v.cpu().numpy(), O.nuasm2(u1, x, y, dict(n=n, pitch=pitch, lam=500e-9, z=8e-3))) < 1e-10
    finally:
        plan.destroy()


@pytest.mark.parametrize("unit", [2.0 ** -100, 2.0 ** 100])
@pytest.mark.parametrize("type_", [1, 2, 3])
def test_fresnel_does_not_depend_on_the_unit_of_length(P, type_, unit):
    """NU-FRE is dimensionless; its factor 1/(lambda z) pitch^2 reaches the tables as 2^+-100 and more."""
    import torch
    n, pitch, m = 256, 5e-6, 400
    rng = np.random.default_rng(82)
    x, y = _points(rng, n, pitch, m)
    src = _dev(rng.normal(size=n * n if type_ == 2 else m) + 0j)
    out = []
    for k in (1.0, unit):
        plan = P.nuasm_plan(P.make_params(n, pitch * k, 500e-9 * k, 8e-3 * k, kind="fresnel", prec="f64"),
                            _dev(x * k), _dev(y * k))
        try:
            v = torch.zeros(n * n if type_ == 1 else m, dtype=torch.complex128, device="cuda")
            if type_ == 3:
                P.nufresnel3_execute(plan, plan, src, v)
            else:
                P.nufresnel_execute(plan, type_, src, v)
            torch.cuda.synchronize()
            out.append(v.cpu().numpy())
        finally:
            plan.destroy()
    assert O.rel_l2(out[1], out[0]) < 1e-12


@pytest.mark.parametrize("m", [0, 3])
def test_zero_sources(P, m):
    import torch
    n = 256
    x = np.zeros(m)
    plan = P.nuasm_plan(P.make_params(n, 5e-6, 500e-9, 8e-3, prec="f64"), _dev(x), _dev(x))
    try:
        u = torch.full((n * n,), 7 + 7j, dtype=torch.complex128, device="cuda")
        P.nuasm1_execute(plan, torch.zeros(m, dtype=torch.complex128, device="cuda"), u)
        torch.cuda.synchronize()
        assert not u.cpu().numpy().any()
    finally:
        plan.destroy()


@pytest.mark.parametrize("tol,bound", [(0.0, 1e-10), (1e-14, 1e-13)])
@pytest.mark.parametrize("n", [16, 64, 128])
@pytest.mark.parametrize("type_", [1, 2])
def test_small_planes_in_both_arithmetics(P, n, type_, tol, bound):
    """N' <= 256: double-float passes at the default tolerance, FP64 ones below
    1e-12 (1e-13: the kernel's error at 1e-14 with some margin)."""
    import torch
    pitch, m = 5e-6, 301
    rng = np.random.default_rng(83)
    x, y = _points(rng, n, pitch, m)
    p = dict(n=n, pitch=pitch, lam=500e-9, z=2e-3)
    plan = P.nuasm_plan(P.make_params(n, pitch, 500e-9, 2e-3, prec="f64", tol=tol), _dev(x), _dev(y))
    try:
        if type_ == 1:
            c = rng.normal(size=m) + 1j * rng.normal(size=m)
            out = torch.zeros(n * n, dtype=torch.complex128, device="cuda")
            P.nuasm1_execute(plan, _dev(c), out)
            ref = O.nuasm1(x, y, c, p).ravel()
        else:
            u1 = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
            out = torch.zeros(m, dtype=torch.complex128, device="cuda")
            P.nuasm2_execute(plan, _dev(u1.ravel()), out)
            ref = O.nuasm2(u1, x, y, p)
        torch.cuda.synchronize()
        assert O.rel_l2(out.cpu().numpy(), ref) < bound
    finally:
        plan.destroy()
