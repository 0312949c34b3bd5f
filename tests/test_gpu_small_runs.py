"""Fused runs of small auxiliary levels, at the sizes where they begin and end.

The sides put the level sizes on both sides of the runs' row limits (512 rows
in FP64, 1,024 in FP32), make the whole hierarchy one run, and (graded) add a
run at the finest levels.  One preconditioner application is held to the
oracle (FP64: 1e-11 as in the parity tests; the FP32 V-cycle: 1e-5, some
hundred roundings of 6e-8 per entry), and the four-column solve to single
solves (1e-9).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402


@pytest.mark.parametrize("nside,graded", [(6, False), (18, False), (33, False), (47, False), (70, False), (65, True)])
@pytest.mark.parametrize("precision", [0, 1])
def test_runs_match_oracle_and_multi(gen, nside, graded, precision):
    from paper_1410_2153_gb300 import asmg
    m = gen.grid2d(nside, 4, graded=graded)
    o = oracle.Oracle(m, coarse_max=20)
    s = asmg.Solver(m, precision=precision, coarse_max_dofs=20)
    vf = o.vertex_of_free()
    r = np.zeros(m.nv)
    r[vf] = np.random.default_rng(3).standard_normal(vf.size)
    z = s.precond(torch.from_numpy(r).cuda()).cpu().numpy()[vf]
    z_ref = o.precond(r[vf])
    assert np.linalg.norm(z - z_ref) <= (1e-11 if precision == 0 else 1e-5) * np.linalg.norm(z_ref)
    k = 3
    b = torch.cat([s.mass_apply(torch.from_numpy(gen.nodal_uniform(m, 20 + c)).cuda()) for c in range(k)])
    u = torch.zeros_like(b)
    rc, its, _ = asmg.amg_solve_multi(s.h, k, b, u, 1e-10)
    assert rc == asmg.ASMG_OK
    for c in range(k):
        u1, _, it1, _ = s.solve(b[c * m.nv:(c + 1) * m.nv], rtol=1e-10)
        assert abs(int(its[c]) - it1) <= 1
        d = (u[c * m.nv:(c + 1) * m.nv] - u1).norm() / u1.norm()
        assert d <= 1e-9, float(d)
    s.close()
