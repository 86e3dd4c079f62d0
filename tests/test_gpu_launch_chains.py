"""Kernels launched before their predecessor has ended: solves issued back to
back with changing inputs, each reading what the one before wrote, give the same
bits on the default stream, on a stream of their own and (ordinary launches)
replayed from a captured graph."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 8, 8), (48, 32, 72), (128, 64, 64), (18, 243, 16)])
def test_poisson_chain(gpu_lib, shape):
    import torch
    ek = gpu_lib
    nx, ny, nz = shape
    q = torch.from_numpy(np.random.default_rng(5).standard_normal(nx * ny * nz)).cuda()
    spec = torch.empty(ek.poisson_scratch_bytes(nx, ny, nz) // 8, dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()

    def chain(stream):
        # phi_1 of q, phi_2 of phi_1, ...: in place from the second on
        phi = torch.empty_like(q)
        ek.poisson_solve(q, phi, shape, 0.7, spec, stream=stream)
        for _ in range(4):
            ek.poisson_solve(phi, phi, shape, 0.7, spec, stream=stream)
        return phi

    a = chain(None).cpu()
    with torch.cuda.stream(side):
        b = chain(side)
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        c = chain(side)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(a, b.cpu())
    assert torch.equal(a, c.cpu())


@pytest.mark.parametrize("shape", [(16, 16, 16), (64, 96, 32), (36, 54, 72)])
@pytest.mark.parametrize("solver", ["mg", "cg"])
def test_iterative_chain(gpu_lib, solver, shape):
    import torch
    ek = gpu_lib
    nx, ny, nz = shape
    q = torch.from_numpy(np.random.default_rng(6).standard_normal(nx * ny * nz)).cuda()
    q -= q.mean()

    def solve(stream):
        phi = torch.zeros_like(q)
        if solver == "mg":
            scratch = torch.empty(ek.poisson_mg_scratch_bytes(shape) // 8 + 1, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            ek.poisson_solve_mg(q, phi, shape, 0.7, scratch, stream=stream)
        else:
            scratch = torch.empty(ek.poisson_cg_scratch_bytes(shape) // 8 + 1, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            ek.poisson_solve_cg(q, phi, shape, 0.7, scratch, stream=stream)
        torch.cuda.synchronize()
        return phi.cpu()

    a = solve(None)
    assert torch.equal(a, solve(torch.cuda.Stream()))
    assert torch.equal(a, solve(None))
