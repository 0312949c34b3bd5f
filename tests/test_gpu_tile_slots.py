"""Tiles of every slot count against the class-by-class launches.

The tile kernels are compiled per rows a thread holds (1 to 4) and per row
width; a requested tile size beyond what a block holds is cut in half until
its tiles fit.  Small, odd and oversized tile sizes reach each of these; the
preconditioner must not change by a bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_rows", [32, 333, 700, 65536])
@pytest.mark.parametrize("precision,level_bf16", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("mesh", ["graded193", "kuhn25"])
def test_any_tile_size_equals_class_launches(gen, mesh, tile_rows, precision, level_bf16):
    from paper_1410_2153_gb300 import asmg
    if mesh == "kuhn25":
        m, opts = gen.grid3d(25, 3), {"n_min": 6}
    else:
        m, opts = gen.grid2d(193, 2, graded=True), {}
    ref = asmg.Solver(m, precision=precision, level_bf16=level_bf16, tile_rows=-1, **opts)
    til = asmg.Solver(m, precision=precision, level_bf16=level_bf16, tile_rows=tile_rows, **opts)
    r = torch.from_numpy(np.random.default_rng(7).standard_normal(m.nv)).cuda()
    z0, z1 = ref.precond(r).cpu().numpy(), til.precond(r).cpu().numpy()
    ref.close()
    til.close()
    assert np.array_equal(z0, z1), np.abs(z0 - z1).max()
