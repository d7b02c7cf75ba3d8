"""The three-stage z pass at the padded z sizes the planner adds to 128 and 256: 512 (1 to 5
combined fields), 64 and 32 (5 and 6 fields), at the smallest, ragged and largest nz of each,
against the FP64 direct sum of Eq. 10 (relative L2 1e-5 per component; FP16 spectra 5e-4) and
against the shared-memory schedule (1e-6, both FP32 roundings of the same sum)."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def families(n):
    t, b = W.gan_families()
    if n == 6:        # five Cartesian fields of the 18 families and an x-directed edge family
        return np.concatenate([t, [[1.0, 0.0, 0.0]]]), np.concatenate([b, [[0.0, W.A_LATT, 0.0]]])
    pick = {1: [0], 2: [0, 9], 3: [0, 7, 8], 4: [0, 1, 2, 9, 10], 5: list(range(18))}[n]
    return t[pick], b[pick]


def rel(got, ref):
    top = max(np.linalg.norm(r) for r in ref)
    return max(np.linalg.norm(g - r) / max(np.linalg.norm(r), 1e-6 * top) for g, r in zip(got, ref))


@pytest.mark.parametrize("nx,ny,nz,fields,fp16,bf16", [
    (9, 6, 129, 1, False, False), (6, 5, 200, 2, False, True), (7, 6, 256, 3, False, False),
    (6, 5, 131, 4, True, False), (5, 6, 150, 5, False, False), (6, 4, 256, 5, False, True),
    (33, 20, 17, 5, False, False), (40, 17, 32, 6, False, False), (37, 9, 25, 5, True, True),
    (35, 20, 9, 5, False, False), (64, 11, 16, 6, False, True), (20, 18, 12, 5, False, False)])
def test_sizes(nx, ny, nz, fields, fp16, bf16):
    import paper_1804_01830_gb300 as dds
    t, b = families(fields)
    p = W.random_problem(W.Geometry(nx, ny, nz, 0.2e-6, 0.3e-6, 0.1e-6), t, b, seed=nx + ny + nz)
    rho = torch.from_numpy(p.rho.astype(np.float32)).cuda()
    rho = rho.to(torch.bfloat16) if bf16 else rho
    out = []
    for lanes in (0, -1):
        ctx = dds.StressContext(0)
        g = p.geom
        ctx.set_geometry(g.nx, g.ny, g.nz, g.dx, g.dy, g.dz, g.mu, g.nu).set_families(t, b)
        ctx.set_option(dds.DDS_OPT_Z_LANES, lanes)
        ctx.set_option(dds.DDS_OPT_SPECTRA_FP16, int(fp16))
        ctx.build_kernels()
        sets = torch.stack([rho, torch.flip(rho, dims=[1]), rho])      # a batch: sets share the tiles' spectra
        multi = ctx.stress_multi(sets).cpu().numpy().astype(float)
        assert rel(multi[2].reshape(6, -1), multi[0].reshape(6, -1)) == 0.0
        out.append(multi[0].reshape(6, -1))
        ctx.close()
    tg = np.unique(np.linspace(0, p.geom.n_cells - 1, 300).astype(int))
    ref = oracle.stress_direct(p.geom, t, b, rho.float().cpu().numpy().astype(float), targets=tg).T
    assert rel(out[0][:, tg], ref) <= (5e-4 if fp16 else 1e-5)
    assert rel(out[0], out[1]) <= (2e-4 if fp16 else 1e-6)
