"""The FP32 row passes of N' = 4096 and 8192 (pairs of sequences per thread):
types 1, 2 and 3 on ragged point counts."""
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


@pytest.mark.parametrize("n", [2048, 4096])
def test_types_1_2_3_at_zero_distance_on_lattice_points(P, n):
    """z = 0: the transfer function is 1, so a source at a lattice point gives
    that plane sample alone, and the plane is read back unchanged (1e-5: the
    FP32 kernel tolerance 1e-6 with its sums)."""
    import torch
    pitch, rng, m = 4e-6, np.random.default_rng(71), 777
    flat = rng.choice(n * n, m, replace=False)
    x = torch.from_numpy((flat % n - n // 2) * pitch).cuda()
    y = torch.from_numpy((flat // n - n // 2) * pitch).cuda()
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.0), x, y)
    try:
        c = torch.from_numpy((rng.normal(size=m) + 1j * rng.normal(size=m)).astype(np.complex64)).cuda()
        u = torch.zeros(n * n, dtype=torch.complex64, device="cuda")
        v, w = torch.zeros_like(c), torch.zeros_like(c)
        P.nuasm1_execute(plan, c, u)
        P.nuasm2_execute(plan, u, v)
        P.nuasm3_execute(plan, plan, c, w)
        torch.cuda.synchronize()
        ref = np.zeros(n * n, np.complex64)
        ref[flat] = c.cpu().numpy()
        assert O.rel_l2(u.cpu().numpy(), ref) < 1e-5
        assert O.rel_l2(v.cpu().numpy(), c.cpu().numpy()) < 1e-5
        assert O.rel_l2(w.cpu().numpy(), c.cpu().numpy()) < 1e-5
    finally:
        plan.destroy()


@pytest.mark.parametrize("n", [2048, 4096])
@pytest.mark.parametrize("type_", [1, 3])
def test_adjoint_at_a_distance(P, n, type_):
    """<T c, v> = <c, T* v>, T* the opposite type (or type 3 back) over -z, -o."""
    import torch
    pitch, rng = 4e-6, np.random.default_rng(72)
    h = 0.5 * n * pitch * (1 - 1e-9)

    def cplx(k):
        return torch.from_numpy((rng.normal(size=k) + 1j * rng.normal(size=k)).astype(np.complex64)).cuda()

    def plan(z, o, pts):
        return P.nuasm_plan(P.make_params(n, pitch, 633e-9, z, ox=o, oy=-o), *pts)

    m = 1001
    src = [torch.from_numpy(rng.uniform(-h, h, m)).cuda() for _ in range(2)]
    dst = [torch.from_numpy(rng.uniform(-h, h, m + 30)).cuda() for _ in range(2)]
    z, o = 0.05, 50e-6
    plans = [plan(z, o, src), plan(-z, -o, src), plan(z, o, dst), plan(-z, -o, dst)]
    try:
        c = cplx(m)
        v = cplx(n * n if type_ == 1 else m + 30)
        a, b = torch.zeros_like(v), torch.zeros_like(c)
        if type_ == 1:
            P.nuasm1_execute(plans[0], c, a)
            P.nuasm2_execute(plans[1], v, b)
        else:
            P.nuasm3_execute(plans[0], plans[2], c, a)
            P.nuasm3_execute(plans[3], plans[1], v, b)
        torch.cuda.synchronize()
        # the transforms carry 1/N'^2 in the plane -> points direction (type 2) as in type 1, so
        # both sides scale alike; compared against the product of the norms
        lhs, rhs = torch.vdot(v.to(torch.complex128), a.to(torch.complex128)), \
            torch.vdot(b.to(torch.complex128), c.to(torch.complex128))
        scale = float(v.norm() * a.norm())
        assert abs(lhs - rhs).item() < 1e-5 * scale
    finally:
        for p in plans:
            p.destroy()


def test_arrays_off_the_16_byte_alignment_at_n_4096(P):
    """The paired column passes of N' = 8192 need 16-byte aligned arrays; others
    take the one-column passes (equal to FP32 rounding of another order of
    operations: 2e-6)."""
    import torch
    n, pitch, rng, m = 4096, 4e-6, np.random.default_rng(73), 500
    h = 0.5 * n * pitch * (1 - 1e-9)
    plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.05),
                        *(torch.from_numpy(rng.uniform(-h, h, m)).cuda() for _ in range(2)))
    try:
        c = torch.from_numpy((rng.normal(size=m) + 1j * rng.normal(size=m)).astype(np.complex64)).cuda()
        buf = torch.zeros(n * n + 1, dtype=torch.complex64, device="cuda")
        out = [buf[:-1], torch.zeros(n * n + 1, dtype=torch.complex64, device="cuda")[1:]]
        for u in out:
            P.nuasm1_execute(plan, c, u)
        src = torch.zeros(n * n + 1, dtype=torch.complex64, device="cuda")[1:]
        src.copy_(out[0])
        v = [torch.zeros_like(c) for _ in range(2)]
        P.nuasm2_execute(plan, out[0], v[0])
        P.nuasm2_execute(plan, src, v[1])
        torch.cuda.synchronize()
        assert out[1].data_ptr() % 16 == 8 and src.data_ptr() % 16 == 8
        assert O.rel_l2(out[1].cpu().numpy(), out[0].cpu().numpy()) < 2e-6
        assert O.rel_l2(v[1].cpu().numpy(), v[0].cpu().numpy()) < 2e-6
    finally:
        plan.destroy()
