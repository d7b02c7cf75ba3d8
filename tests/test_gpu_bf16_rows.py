"""Forward x pass on BF16 rows of 65 to 128 cells summed over families: runs of eight values a
thread (nx a multiple of 4), with lines that end inside a run's stride and line counts that
leave CTAs partly empty, and the value-by-value kernel beside it (other nx).  Single sets, a
batch and a subset, against the FP64 direct sum of Eq. 10 of the same
(BF16) densities, 1e-5 relative L2 per component; batch and subset against the single set 1e-6."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rel(got, ref):
    got, ref = (np.asarray(v, dtype=float).reshape(6, -1) for v in (got, ref))
    top = max(np.linalg.norm(r) for r in ref)
    return max(np.linalg.norm(g - r) / max(np.linalg.norm(r), 1e-6 * top) for g, r in zip(got, ref))


@pytest.mark.parametrize("shape", [(68, 3, 3), (72, 1, 1), (100, 7, 5), (124, 5, 2), (128, 9, 4), (128, 8, 4),
                                   (101, 7, 5), (102, 5, 3), (67, 3, 2), (127, 4, 3)])
def test_summed_families(shape):
    import paper_1804_01830_gb300 as dds
    t, b = W.gan_families()
    g = W.Geometry(*shape, 0.2e-6, 0.3e-6, 0.08e-6)
    p = W.random_problem(g, t, b, seed=sum(shape))
    rho = torch.from_numpy(p.rho.astype(np.float32)).cuda().to(torch.bfloat16)
    ctx = dds.StressContext(0)
    ctx.set_geometry(g.nx, g.ny, g.nz, g.dx, g.dy, g.dz, g.mu, g.nu).set_families(t, b).build_kernels()
    one = ctx.stress(rho).cpu().numpy()
    tg = np.unique(np.linspace(0, g.n_cells - 1, 300).astype(int))
    ref = oracle.stress_direct(g, t, b, rho.float().cpu().numpy().astype(float), targets=tg).T
    assert rel(one.reshape(6, -1)[:, tg], ref) <= 1e-5
    sets = torch.stack([torch.flip(rho, dims=[3]), rho]).contiguous()
    assert rel(ctx.stress_multi(sets)[1].cpu().numpy(), one) <= 1e-6
    fams = [4, 1, 16, 9]
    part = torch.zeros_like(rho)
    part[fams] = rho[fams]
    sub = ctx.stress_subset(fams, rho[fams].contiguous()).cpu().numpy()
    assert rel(sub, ctx.stress(part).cpu().numpy()) <= 1e-6
    ctx.close()
