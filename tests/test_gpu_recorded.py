"""Solves recorded into a caller's CUDA graph, whose launches keep their order,
against the same solves launched on a stream, where the kernels of small FP32
chains start early."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1308_6644_gb300 as pkg
    return pkg


@pytest.mark.parametrize("n", [16, 256, 512, 1024])
@pytest.mark.parametrize("typ", [1, 2])
def test_recorded_solve_matches_stream(P, n, typ):
    """Type 2 is the same arithmetic in the same order: equal bits.  Type 1 may
    add split tiles in another order: a few roundings of 2^-24 (1e-6)."""
    import torch
    rng = np.random.default_rng(95)
    m, h = 4 * n * 16, 0.5 * n * 10e-6 * (1 - 1e-9)
    x, y = (torch.from_numpy(rng.uniform(-h, h, m)).cuda() for _ in range(2))
    gen = torch.Generator("cuda").manual_seed(3)
    num = (m, n * n) if typ == 1 else (n * n, m)
    src = [torch.randn(num[0], dtype=torch.complex64, device="cuda", generator=gen) for _ in range(3)]
    out = torch.zeros(num[1], dtype=torch.complex64, device="cuda")
    execute = P.nuasm1_execute if typ == 1 else P.nuasm2_execute
    plan = P.nuasm_plan(P.make_params(n, 10e-6, 633e-9, 0.01), x, y)
    try:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            held = src[0].clone()
            execute(plan, held, out)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                execute(plan, held, out)
                execute(plan, held, out)
        torch.cuda.synchronize()
        for s in src:
            execute(plan, s, out)
            torch.cuda.synchronize()
            direct = out.clone()
            held.copy_(s)
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            if typ == 2:
                assert torch.equal(out, direct)
            else:
                assert torch.linalg.vector_norm(out - direct) <= 1e-6 * torch.linalg.vector_norm(direct)
    finally:
        plan.destroy()
