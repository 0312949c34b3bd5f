"""A coefficient update that fails in the rebuild, and the update after it.

Coefficients of 1.7e308 are positive and finite, but their element matrices add
up to infinities: the coarsest matrix has no Cholesky factor.  The handle then
refuses every call until an update succeeds, and equals a new handle after that.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_calls_are_refused_until_an_update_succeeds(gen, precision):
    from paper_1410_2153_gb300 import asmg
    m = gen.grid2d(40, 5)
    a = np.exp(np.random.default_rng(2).uniform(-1, 1, m.ne))
    s = asmg.Solver(m, precision=precision)
    batch = asmg.amg_batch_create([s.h], 2, 1e-9)
    b = s.mass_apply(torch.from_numpy(gen.nodal_uniform(m, 1)).cuda())
    u = torch.zeros(2 * m.nv, dtype=torch.float64, device="cuda")
    its = s.solve(b)[2]
    assert its > 0 and s.precond(b).norm() > 0          # graphs of both exist
    with pytest.raises(asmg.AsmgError):
        asmg.amg_update_coefficients(s.h, np.full(m.ne, 1.7e308))
    for call in (lambda: s.solve(b), lambda: s.precond(b), lambda: s.spmv(b), lambda: s.mass_apply(b),
                 lambda: asmg.amg_solve_multi(s.h, 2, torch.cat([b, b]), u, 1e-9),
                 lambda: asmg.amg_batch_solve(batch, [b, b], [u[:m.nv], u[m.nv:]])):
        with pytest.raises(asmg.AsmgError) as e:
            call()
        assert e.value.code == asmg.ASMG_ERR_INVALID_ARG
    asmg.amg_batch_destroy(batch)
    asmg.amg_update_coefficients(s.h, a)
    m2 = gen.grid2d(40, 5)
    m2.coeff = a
    fresh = asmg.Solver(m2, precision=precision)
    assert torch.equal(s.precond(b), fresh.precond(b))
    assert torch.equal(s.solve(b)[0], fresh.solve(b)[0])
    s.close()
    fresh.close()
