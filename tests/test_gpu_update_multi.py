"""Multiple right-hand sides after a coefficient update.

The work state of earlier solves points at the operators it was made for: after
an update, amg_solve_multi makes new state (and equals a handle set up with the
new coefficients), and a batch captured before the update is refused.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_multi_solves_follow_a_coefficient_update(gen, precision):
    from paper_1410_2153_gb300 import asmg
    m = gen.grid2d(70, 5)
    a = np.exp(np.random.default_rng(2).uniform(-1, 1, m.ne))
    s = asmg.Solver(m, precision=precision)
    b = torch.cat([s.mass_apply(torch.from_numpy(gen.nodal_uniform(m, c)).cuda()) for c in range(2)])
    u = torch.zeros_like(b)
    asmg.amg_solve_multi(s.h, 2, b, u, 1e-9)
    batch = asmg.amg_batch_create([s.h], 2, 1e-9)
    asmg.amg_update_coefficients(s.h, a)
    u.zero_()
    asmg.amg_solve_multi(s.h, 2, b, u, 1e-9)
    bs = [b[: m.nv].clone(), b[m.nv:].clone()]
    with pytest.raises(asmg.AsmgError) as e:
        asmg.amg_batch_solve(batch, bs, [torch.zeros_like(v) for v in bs])
    assert e.value.code == asmg.ASMG_ERR_INVALID_ARG
    asmg.amg_batch_destroy(batch)
    m2 = gen.grid2d(70, 5)
    m2.coeff = a
    fresh = asmg.Solver(m2, precision=precision)
    v = torch.zeros_like(b)
    asmg.amg_solve_multi(fresh.h, 2, b, v, 1e-9)
    assert torch.equal(u, v)
    s.close()
    fresh.close()
