"""The relaxation's march at the edges of its tiles (64 x 8 and 32 x 16 columns), chunks (4, 8 and 16
layers) and copies (16-byte, 8-byte and single values): every shape against the FP64
oracle after a few steps, with the bounds of the step-for-step test (1e-6 + K 2^-24
relative L2 after K steps; the total stress relative to its largest component)."""
import numpy as np
import pytest

import oracle.relax as R
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H = (0.2e-6, 0.2e-6, 0.05e-6)
STEPS = 3
TOL = 1e-6 + STEPS * 2.0 ** -24


@pytest.mark.parametrize("shape", [(2, 8, 64), (4, 9, 65), (5, 7, 63), (16, 16, 128), (17, 1, 1), (18, 3, 2), (33, 8, 68),
                                   (9, 8, 60), (65, 72, 192), (40, 90, 100), (17, 200, 512),
                                   (6, 16, 32), (9, 17, 31), (4, 33, 96), (21, 15, 160)])
@pytest.mark.parametrize("shift", [0, 1])            # first value of u, load and total off 16-byte alignment
def test_tile_edges(shape, shift):
    import paper_1804_01830_gb300 as dds
    nz, ny, nx = shape
    rng = np.random.default_rng(sum(shape))
    sig = (1e8 * rng.standard_normal((6,) + shape)).astype(np.float32)
    u0 = (1e-10 * rng.standard_normal((3,) + shape)).astype(np.float32)
    ctx = dds.StressContext(0).set_geometry(nx, ny, nz, *H, W.MU_GAN, W.NU_GAN)

    def on_device(a):
        flat = torch.empty(a.size + 4, dtype=torch.float32, device="cuda")
        t = flat[shift:shift + a.size].view(a.shape)
        t.copy_(torch.from_numpy(a))
        return t

    sig_d, u_d, tot_d = on_device(sig), on_device(u0), on_device(np.zeros_like(sig))
    dds.dds_relax(ctx.handle, sig_d.data_ptr(), u_d.data_ptr(), STEPS, tot_d.data_ptr())
    torch.cuda.synchronize()
    s64 = sig.astype(np.float64)
    u = R.relax(s64, H, W.MU_GAN, W.NU_GAN, STEPS, u0=u0.astype(np.float64))
    tot = R.total_stress(u, s64, H, W.MU_GAN, W.NU_GAN)
    top = max(np.linalg.norm(c) for c in u)
    for got, ref in zip(u_d.cpu().numpy().astype(float), u):
        assert np.linalg.norm(got - ref) <= TOL * max(np.linalg.norm(ref), 1e-6 * top)
    top = max(np.linalg.norm(c) for c in tot)
    for got, ref in zip(tot_d.cpu().numpy().astype(float), tot):
        assert np.linalg.norm(got - ref) <= TOL * top
    # the total stress may replace the load
    dds.dds_relax(ctx.handle, sig_d.data_ptr(), u_d.data_ptr(), 0, sig_d.data_ptr())
    assert torch.equal(sig_d, tot_d)
    ctx.close()
