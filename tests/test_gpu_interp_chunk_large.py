"""Interpolation chunks at the ends of their range: every value from the number of
points up means one CTA per tile."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1308_6644_gb300 as pkg
    return pkg


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("m", [1, 65, 30000])
@pytest.mark.parametrize("tile", [0, 16])
def test_chunks_of_any_size_give_equal_bits(P, prec, m, tile):
    import torch
    n, pitch = 64, 10e-6
    rng = np.random.default_rng(48)
    x, y = (torch.from_numpy(np.clip(rng.normal(0, 40e-6, m), -3e-4, 3e-4)).cuda() for _ in range(2))
    cdt = torch.complex64 if prec == "f32" else torch.complex128
    u = torch.randn(n * n, dtype=cdt, device="cuda", generator=torch.Generator("cuda").manual_seed(6))
    out = []
    for chunk in (0, 64, 30000, (1 << 31) - 64, (1 << 31) - 1):
        plan = P.nuasm_plan(P.make_params(n, pitch, 633e-9, 0.02, prec=prec, tile=tile, interp_chunk=chunk), x, y)
        try:
            v = torch.zeros(m, dtype=cdt, device="cuda")
            P.nuasm2_execute(plan, u, v)
            torch.cuda.synchronize()
            out.append(v)
        finally:
            plan.destroy()
    assert out[0].abs().max() > 0
    for v in out[1:]:
        assert torch.equal(v, out[0])
