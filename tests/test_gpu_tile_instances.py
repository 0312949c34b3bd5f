"""Which tile kernels the tile sizes of test_gpu_tile_slots.py reach, and their four-column forms.

A tile kernel is compiled per rows a thread holds and per row width.  The sizes
must reach every count of rows, down and up; there a preconditioner application
and a four-column solve equal the class-by-class launches bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,level_bf16", [(0, 0), (1, 0), (1, 1)])
def test_tiles_of_every_slot_count_run(gen, precision, level_bf16):
    from paper_1410_2153_gb300 import asmg
    reached = set()
    for mesh, sizes in ((gen.grid2d(193, 2, graded=True), (32, 100, 333, 65536)), (gen.grid3d(17, 3), (32, 100))):
        opts = dict(precision=precision, level_bf16=level_bf16, **({"n_min": 6} if mesh.dim == 3 else {}))
        for nu in (1, 2):
            ref = asmg.Solver(mesh, tile_rows=-1, nu_pre=nu, nu_post=nu, **opts)
            r = torch.from_numpy(np.random.default_rng(7).standard_normal(mesh.nv)).cuda()
            b = torch.cat([ref.mass_apply(torch.from_numpy(gen.nodal_uniform(mesh, c)).cuda()) for c in range(4)])
            z, u = ref.precond(r), torch.zeros_like(b)
            its = asmg.amg_solve_multi(ref.h, 4, b, u, 1e-6)[1]
            for rows in sizes:
                s = asmg.Solver(mesh, tile_rows=rows, nu_pre=nu, nu_post=nu, **opts)
                levels = range(s.info("coarse") + 1, s.info("J") + 1)
                slots = [s.info("tile_slots", level) for level in levels]
                widths = [s.info("tile_width", level) for level in levels]
                assert any(slots) and all((n > 0) == (w > 0) for n, w in zip(slots, widths))
                assert all(w % 256 <= 16 and w // 256 <= 16 for w in widths)
                reached |= {("down", n % 16) for n in slots if n} | {("up", n // 16) for n in slots if n}
                assert torch.equal(s.precond(r), z), (mesh.dim, nu, rows)
                v = torch.zeros_like(b)
                assert np.array_equal(asmg.amg_solve_multi(s.h, 4, b, v, 1e-6)[1], its)
                assert torch.equal(v, u), (mesh.dim, nu, rows)
                s.close()
            ref.close()
    assert reached == {(d, n) for d in ("down", "up") for n in (1, 2, 3, 4)}
