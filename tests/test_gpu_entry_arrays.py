"""Where the entry points take their arrays: in place, staged, or overlapping.

Device arrays are read and written in place, host arrays (and device arrays at
an address not aligned for doubles never occur in torch) are staged; the input
and output of one call may be the same array.  Every combination must give the
bits of the separate device arrays.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", ["jitter37", "kuhn11"])
@pytest.mark.parametrize("precision", [0, 1])
def test_host_device_and_in_place_arrays_agree(gen, mesh, precision):
    from paper_1410_2153_gb300 import asmg
    m, opts = (gen.grid2d(37, 2), {}) if mesh == "jitter37" else (gen.grid3d(11, 2), {"n_min": 6})
    s = asmg.Solver(m, precision=precision, **opts)
    rng = np.random.default_rng(1)
    x, y = rng.uniform(-1, 1, (2, m.nv))     # Dirichlet entries too: ignored, but for the mass product
    dev = torch.from_numpy(x).cuda()
    for name in ("spmv", "precond", "mass_apply"):
        ref = getattr(s, name)(dev)
        assert np.array_equal(getattr(s, name)(x), ref.cpu().numpy()), name
        same = dev.clone()
        call = {"spmv": asmg.amg_spmv, "precond": asmg.amg_precond_apply, "mass_apply": asmg.amg_mass_apply}[name]
        call(s.h, same, same)
        assert torch.equal(same, ref), name
    shifted = torch.empty(m.nv + 1, dtype=torch.float64, device="cuda")   # half-overlapping input and output
    shifted[:-1] = dev
    asmg.amg_mass_apply(s.h, shifted[:-1], shifted[1:])
    assert torch.equal(shifted[1:], s.mass_apply(dev))
    g = s.element_grad(dev, torch.from_numpy(y).cuda())
    assert np.array_equal(s.element_grad(x, y), g.cpu().numpy())
    b = s.mass_apply(dev)
    u, rc, it, hist = s.solve(b)
    uh, rch, ith, histh = s.solve(b.cpu().numpy())
    assert (rc, it) == (rch, ith) and np.array_equal(uh, u.cpu().numpy()) and np.array_equal(hist, histh)
    both = b.clone()                          # right-hand side and initial guess the same array
    asmg.amg_solve(s.h, both, both, 1e-8)
    apart, guess = b.clone(), b.clone()
    asmg.amg_solve(s.h, apart, guess, 1e-8)
    assert torch.equal(both, guess)
    k = 3
    bk = torch.cat([b * (c + 1) for c in range(k)])
    ud, uk = torch.zeros_like(bk), np.zeros(k * m.nv)
    asmg.amg_solve_multi(s.h, k, bk, ud, 1e-8)
    asmg.amg_solve_multi(s.h, k, bk.cpu().numpy(), uk, 1e-8)
    assert np.array_equal(uk, ud.cpu().numpy())
    for nrhs in (1, k):                       # one branch per right-hand side, and interleaved columns
        batch = asmg.amg_batch_create([s.h], nrhs, 1e-8)
        bs = [bk[c * m.nv:(c + 1) * m.nv].clone() for c in range(nrhs)]
        us = [torch.zeros_like(v) for v in bs]
        asmg.amg_batch_solve(batch, bs, us)
        hs = [np.zeros(m.nv) for _ in bs]
        asmg.amg_batch_solve(batch, [v.cpu().numpy() for v in bs], hs)
        mixed = [torch.zeros_like(bs[0])] + [np.zeros(m.nv) for _ in bs[1:]]
        asmg.amg_batch_solve(batch, bs, mixed)
        for c in range(nrhs):
            ref = us[c].cpu().numpy()
            assert np.array_equal(hs[c], ref)
            assert np.array_equal(mixed[c] if c else mixed[0].cpu().numpy(), ref)
        asmg.amg_batch_destroy(batch)
    s.close()
