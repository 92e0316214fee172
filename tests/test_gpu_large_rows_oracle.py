"""The FP32 passes of N' = 4096 and 8192 at a distance against the direct oracle:
type 1 at some of its samples, type 3 at its points, type 2 as type 3's second
half (paired row and column passes with the factors of the transfer function)."""
import functools

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


PITCH, LAM, Z, OX, OY = 4e-6, 633e-9, 0.05, 40e-6, -25e-6


@functools.lru_cache(maxsize=2)
def transfer(n):
    return O.asm_transfer(n, 2 * n, PITCH, LAM, Z, OX, OY)


@pytest.mark.parametrize("n", [2048, 4096])
def test_types_1_and_3_at_a_distance(P, n):
    """A type-1 sample is the type-3 value at the sample's position, so one direct
    evaluation serves both.  1e-5: the FP32 bound."""
    import torch
    pitch, rng = PITCH, np.random.default_rng(74)
    h = 0.5 * n * pitch * (1 - 1e-9)
    m, k = 301, 60
    src = [rng.uniform(-h, h, m) for _ in range(2)]
    dst = [rng.uniform(-h, h, k) for _ in range(2)]
    flat = rng.choice(n * n, k, replace=False)
    lat = [(flat % n - n // 2) * pitch, (flat // n - n // 2) * pitch]
    c = (rng.normal(size=m) + 1j * rng.normal(size=m)).astype(np.complex64)
    params = P.make_params(n, pitch, LAM, Z, ox=OX, oy=OY)
    a, b = (P.nuasm_plan(params, *(torch.from_numpy(v).cuda() for v in pts)) for pts in (src, dst))
    try:
        dc = torch.from_numpy(c).cuda()
        u = torch.zeros(n * n, dtype=torch.complex64, device="cuda")
        v = torch.zeros(k, dtype=torch.complex64, device="cuda")
        P.nuasm1_execute(a, dc, u)
        P.nuasm3_execute(a, b, dc, v)
        torch.cuda.synchronize()
        u = u[torch.from_numpy(flat).cuda()].cpu().numpy()
        v = v.cpu().numpy()
    finally:
        a.destroy()
        b.destroy()
    ref = O.diffraction_type3(*src, c, np.concatenate([lat[0], dst[0]]), np.concatenate([lat[1], dst[1]]),
                              dict(n=n, pitch=pitch), h=transfer(n))
    assert O.rel_l2(u, ref[:k]) < 1e-5
    assert O.rel_l2(v, ref[k:]) < 1e-5


@pytest.mark.parametrize("n", [2048, 4096])
def test_type_2_at_a_distance(P, n):
    """A plane of 301 single samples is a type-3 source at their positions."""
    import torch
    pitch, rng = PITCH, np.random.default_rng(75)
    h = 0.5 * n * pitch * (1 - 1e-9)
    m, k = 301, 60
    flat = rng.choice(n * n, m, replace=False)
    dst = [rng.uniform(-h, h, k) for _ in range(2)]
    c = (rng.normal(size=m) + 1j * rng.normal(size=m)).astype(np.complex64)
    plan = P.nuasm_plan(P.make_params(n, pitch, LAM, Z, ox=OX, oy=OY),
                        *(torch.from_numpy(v).cuda() for v in dst))
    try:
        u = torch.zeros(n * n, dtype=torch.complex64, device="cuda")
        u[torch.from_numpy(flat).cuda()] = torch.from_numpy(c).cuda()
        v = torch.zeros(k, dtype=torch.complex64, device="cuda")
        P.nuasm2_execute(plan, u, v)
        torch.cuda.synchronize()
        v = v.cpu().numpy()
    finally:
        plan.destroy()
    ref = O.diffraction_type3((flat % n - n // 2) * pitch, (flat // n - n // 2) * pitch, c, *dst,
                              dict(n=n, pitch=pitch), h=transfer(n))
    assert O.rel_l2(v, ref) < 1e-5
