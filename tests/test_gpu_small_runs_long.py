"""Fused runs of small levels whose rows are longer than a run's ELL part.

Locally refined 3D grids (a cube's vertices mapped by x -> x^p) have rows of 19
to 25 entries on their small levels; those levels run fused all the same.  One
preconditioner application is held to the oracle (FP64: 1e-11; FP32: 1e-5, some
hundred roundings of 6e-8; BF16 level values: 5e-2, 2^-9 per entry over some ten
levels), and the four-column solve to single solves (1e-7 at rtol 1e-12: twice
rtol times a condition number of up to 5e4).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402


@pytest.fixture(scope="module", params=[(17, 2), (13, 3)])
def case(request, gen):
    n, power = request.param
    m = gen.grid3d(n, 1)
    m.verts = np.ascontiguousarray(m.verts ** power)
    o = oracle.Oracle(m, n_min=6)
    vf = o.vertex_of_free()
    r = np.zeros(m.nv)
    r[vf] = np.random.default_rng(3).standard_normal(vf.size)
    return m, vf, r, o.precond(r[vf])


@pytest.mark.parametrize("precision,level_bf16,tol", [(0, 0, 1e-11), (1, 0, 1e-5), (1, 1, 5e-2)])
def test_long_rows_run_fused(gen, case, precision, level_bf16, tol):
    from paper_1410_2153_gb300 import asmg
    m, vf, r, z_ref = case
    s = asmg.Solver(m, precision=precision, level_bf16=level_bf16, n_min=6)
    z = s.precond(torch.from_numpy(r).cuda()).cpu().numpy()[vf]
    assert np.linalg.norm(z - z_ref) <= tol * np.linalg.norm(z_ref)
    # the finest level has long rows and no launch of its own
    rows = s.export("level_rows", s.info("J"))["row"]
    assert np.unique(rows, return_counts=True)[1].max() > 16
    b = s.mass_apply(torch.from_numpy(gen.nodal_uniform(m, 20)).cuda())
    res, levels, its = asmg.amg_profile_levels(s.h, b, 1e-8)
    assert sum(p["launches"] for d in levels[-1].values() for p in d.values()) == 0
    assert res["aux_small"]["launches"] >= 2 * its
    k = 3
    b = torch.cat([s.mass_apply(torch.from_numpy(gen.nodal_uniform(m, 20 + c)).cuda()) for c in range(k)])
    u = torch.zeros_like(b)
    rc, its, _ = asmg.amg_solve_multi(s.h, k, b, u, 1e-12)
    assert rc == asmg.ASMG_OK
    for c in range(k):
        u1, _, it1, _ = s.solve(b[c * m.nv:(c + 1) * m.nv], rtol=1e-12)
        assert abs(int(its[c]) - it1) <= 2
        d = (u[c * m.nv:(c + 1) * m.nv] - u1).norm() / u1.norm()
        assert d <= 1e-7, float(d)
    s.close()
