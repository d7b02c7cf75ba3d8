"""Kernel builds held to their work space: fields without mirrors on grids that fill their
padding (two fields a table, then the third; one or two components a launch), alone and beside
mirrored ones, open and periodic in y, in both storage types, against the FP64 direct sum of
Eq. 10.  Bound: the FP32 evaluation's 1e-5 relative L2 per component (FP16 spectra: 5e-4)."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

A, C = W.A_LATT, W.C_LATT
Z, ANY = [0, 0, 1], [1, 2, 2]
CART = [[A, 0, 0], [0, A, 0], [0, 0, C]]
FAMILIES = {"unmirrored": ([ANY] * 3, CART), "beside mirrored": ([Z] * 3 + [ANY] * 3, CART * 2)}


@pytest.mark.parametrize("kind", list(FAMILIES))
@pytest.mark.parametrize("shape,periodic", [((16, 16, 8), False), ((32, 32, 8), False), ((16, 32, 4), True),
                                            ((32, 32, 8), True)])
@pytest.mark.parametrize("fp16", [False, True])
def test_matches_direct_sum(kind, shape, periodic, fp16):
    import paper_1804_01830_gb300 as dds
    t, b = (np.array(v, dtype=float) for v in FAMILIES[kind])
    t /= np.linalg.norm(t, axis=1)[:, None]
    shells = 1 if periodic else 0
    p = W.random_problem(W.Geometry(*shape, 0.2e-6, 0.3e-6, 0.08e-6), t, b, seed=sum(shape) + shells)
    g = p.geom
    ctx = dds.StressContext(0)
    ctx.set_geometry(g.nx, g.ny, g.nz, g.dx, g.dy, g.dz, g.mu, g.nu).set_families(p.t, p.b)
    ctx.set_option(dds.DDS_OPT_PBC_SHELLS, shells)
    ctx.set_option(dds.DDS_OPT_PBC_PERIODIC, int(periodic))
    ctx.set_option(dds.DDS_OPT_SPECTRA_FP16, int(fp16))
    ctx.build_kernels()
    got = ctx.stress(torch.from_numpy(p.rho.astype(np.float32)).cuda()).cpu().numpy().astype(float).reshape(6, -1)
    ctx.close()
    tg = np.unique(np.linspace(0, g.n_cells - 1, 300).astype(int))
    ref = oracle.stress_direct(g, p.t, p.b, p.rho, targets=tg, n_shells=shells, periodic=periodic).T
    top = max(np.linalg.norm(r) for r in ref)
    err = [np.linalg.norm(got[c, tg] - ref[c]) / max(np.linalg.norm(ref[c]), 1e-6 * top) for c in range(6)]
    assert max(err) <= (5e-4 if fp16 else 1e-5), err
