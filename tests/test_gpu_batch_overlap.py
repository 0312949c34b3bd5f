"""Batched solves whose arrays overlap across the branches of the graph.

Every right-hand side and guess is taken before any solution is written, and of
two solutions written to one place the later one stays: the same bits as with
arrays apart.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 2, 5])
def test_overlapping_arrays_give_the_results_of_separate_ones(gen, nrhs):
    from paper_1410_2153_gb300 import asmg
    meshes = [gen.grid2d(33, 1 + i) for i in range(2)]
    solvers = [asmg.Solver(m) for m in meshes]
    nv, k = meshes[0].nv, 2 * nrhs
    batch = asmg.amg_batch_create([s.h for s in solvers], nrhs, 1e-8)
    f = torch.from_numpy(gen.nodal_uniform(meshes[0], 3, k).reshape(k, -1)).cuda()
    b = torch.stack([solvers[j // nrhs].mass_apply(f[j]) for j in range(k)])

    def apart(guess):
        us = [g.clone() for g in guess]
        asmg.amg_batch_solve(batch, [b[j].clone() for j in range(k)], us)
        return us

    # each solution on the next right-hand side, the last on the first
    shared = b.clone()
    asmg.amg_batch_solve(batch, list(shared), [shared[(j + 1) % k] for j in range(k)])
    for j, u in enumerate(apart([b[(j + 1) % k] for j in range(k)])):
        assert torch.equal(shared[(j + 1) % k], u), j
    # one array for every solution, and solutions on their own right-hand sides
    one = torch.zeros(nv, dtype=torch.float64, device="cuda")
    asmg.amg_batch_solve(batch, list(b), [one] * k)
    assert torch.equal(one, apart([torch.zeros_like(one)] * k)[-1])
    own = b.clone()
    asmg.amg_batch_solve(batch, list(own), list(own))
    for j, u in enumerate(apart(b)):
        assert torch.equal(own[j], u), j
    asmg.amg_batch_destroy(batch)
    for s in solvers:
        s.close()
