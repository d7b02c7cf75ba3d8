"""The relaxation's march in chunks of one and two layers (grids whose chunks are all resident at
once), between them and longer ones, with a last chunk shorter than the others: against the
FP64 oracle with the bounds of the step-for-step test (1e-6 + K 2^-24 relative L2 after K steps;
the total stress relative to its largest component)."""
import numpy as np
import pytest

import oracle.relax as R
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H = (0.2e-6, 0.2e-6, 0.05e-6)
STEPS = 3
TOL = 1e-6 + STEPS * 2.0 ** -24


@pytest.mark.parametrize("shape", [(2, 3, 5), (4, 16, 16), (3, 500, 33),      # one layer a chunk
                                   (64, 64, 64), (63, 61, 60), (200, 17, 17), (151, 16, 33),   # two
                                   (76, 64, 64), (80, 64, 64)])       # at and beyond one wave of them (152 SMs)
def test_against_oracle(shape):
    import paper_1804_01830_gb300 as dds
    nz, ny, nx = shape
    rng = np.random.default_rng(sum(shape))
    sig = (1e8 * rng.standard_normal((6,) + shape)).astype(np.float32)
    ctx = dds.StressContext(0).set_geometry(nx, ny, nz, *H, W.MU_GAN, W.NU_GAN)
    sig_d = torch.from_numpy(sig).cuda()
    u_d = torch.zeros((3,) + shape, device="cuda")
    tot_d = torch.empty_like(sig_d)
    dds.dds_relax(ctx.handle, sig_d.data_ptr(), u_d.data_ptr(), STEPS, tot_d.data_ptr())
    torch.cuda.synchronize()
    s64 = sig.astype(np.float64)
    u = R.relax(s64, H, W.MU_GAN, W.NU_GAN, STEPS, u0=np.zeros((3,) + shape))
    tot = R.total_stress(u, s64, H, W.MU_GAN, W.NU_GAN)
    for got, ref in ((u_d, u), (tot_d, tot)):
        top = max(np.linalg.norm(c) for c in ref)
        for g, r in zip(got.cpu().numpy().astype(float), ref):
            assert np.linalg.norm(g - r) <= TOL * top
    ctx.close()
