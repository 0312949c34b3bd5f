"""The algorithmic bytes of one PCG step (amg_info) against the profiler's count of the launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(), dict(precision=1), dict(precision=1, level_bf16=1), dict(precision=1, tile_rows=-1),
                                  dict(fine_sweeps=2), dict(smoother=1), dict(additive=1), dict(iteration=1)])
@pytest.mark.parametrize("mesh", ["graded129", "kuhn13"])
def test_bytes_of_a_step_are_those_of_its_launches(gen, mesh, opts):
    from paper_1410_2153_gb300 import asmg
    m, o = (gen.grid2d(129, 2, graded=True), {}) if mesh == "graded129" else (gen.grid3d(13, 2), {"n_min": 6})
    s = asmg.Solver(m, max_iter=6, **opts, **o)
    b = s.mass_apply(torch.from_numpy(gen.nodal_uniform(m, 1)).cuda())
    totals = []
    for rtol in (0.5, 1e-12):                # a few steps, and (to the cap of 6) some more
        res, its = asmg.amg_profile(s.h, b, rtol)
        totals.append((its, sum(c["bytes"] for c in res.values())))
    (i0, b0), (i1, b1) = totals
    assert i1 > i0 and b1 - b0 == (i1 - i0) * s.info("bytes_iter")
    # an update keeps the figure: same sizes
    asmg.amg_update_coefficients(s.h, np.ones(m.ne))
    assert s.info("bytes_iter") == (b1 - b0) / (i1 - i0)
    s.close()
