"""GPU parity of built contexts over the symmetry classes of the coefficient table: fields
with both mirrors, one or none, one to three fields of a line direction sharing a table,
classes mixed in one context, replica sums with few and many images per offset, and FP16
storage of folded spectra, on ragged grids against the FP64 direct sum of Eq. 10.
Bound: the FP32 evaluation's 1e-5 relative L2 per component (FP16 spectra: 5e-4)."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

A, C = W.A_LATT, W.C_LATT
Z, X, Y, TILT = [0, 0, 1], [1, 0, 0], [0, 1, 0], [0, 0.6, 0.8]
FAMILIES = {
    "both mirrors": ([Z, Z, Z], [[A, 0, 0], [0, A, 0], [0, 0, C]]),
    "x mirror": ([TILT] * 4, [[A, 0, 0], [0, A, 0], [0, 0, C], [A, A, C]]),
    "y mirror": ([[0.6, 0, 0.8], X], [[0, A, 0], [0, 0, C]]),
    "no mirror": ([TILT, [1, 2, 2]], [[A, A, C], [A, -A, 0.3 * C]]),
    "mixed": ([Z, Z, Y, TILT, Z], [[A, 0, 0], [0.5 * A, A, 0], [A, 0, 0], [A, 0, 0], [0, A, C]]),
}


@pytest.mark.parametrize("kind", list(FAMILIES))
@pytest.mark.parametrize("shape,shells,periodic,fp16", [((9, 7, 5), 0, False, False), ((17, 20, 33), 0, False, False),
                                                        ((7, 5, 4), 1, False, False), ((6, 9, 3), 3, False, True),
                                                        ((9, 32, 3), 3, True, False), ((5, 32, 2), 1, True, False)])
def test_built_context_matches_direct_sum(kind, shape, shells, periodic, fp16):
    import paper_1804_01830_gb300 as dds
    t, b = (np.array(v, dtype=float) for v in FAMILIES[kind])
    t /= np.linalg.norm(t, axis=1)[:, None]
    p = W.random_problem(W.Geometry(*shape, 0.2e-6, 0.3e-6, 0.08e-6), t, b, seed=sum(shape) + shells)
    ctx = dds.StressContext(0)
    g = p.geom
    ctx.set_geometry(g.nx, g.ny, g.nz, g.dx, g.dy, g.dz, g.mu, g.nu).set_families(p.t, p.b)
    ctx.set_option(dds.DDS_OPT_PBC_SHELLS, shells)
    ctx.set_option(dds.DDS_OPT_PBC_PERIODIC, int(periodic))
    ctx.set_option(dds.DDS_OPT_SPECTRA_FP16, int(fp16))
    ctx.build_kernels()
    got = ctx.stress(torch.from_numpy(p.rho.astype(np.float32)).cuda()).cpu().numpy().astype(float).reshape(6, -1)
    ctx.close()
    tg = np.unique(np.linspace(0, g.n_cells - 1, 400).astype(int)) if g.n_cells > 3000 else np.arange(g.n_cells)
    ref = oracle.stress_direct(g, p.t, p.b, p.rho, targets=tg, n_shells=shells, periodic=periodic).T
    top = max(np.linalg.norm(r) for r in ref)
    err = [np.linalg.norm(got[c, tg] - ref[c]) / max(np.linalg.norm(ref[c]), 1e-6 * top) for c in range(6)]
    assert max(err) <= (5e-4 if fp16 else 1e-5), err
