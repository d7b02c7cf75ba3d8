"""Work space of the kernel build: its stream-ordered allocations at their highest stay within
a full padded FP64 table of one field and one complex spectrum, for directions alone and for
directions with different mirrors in one context, open and periodic in y.  Allowance: the
index and scalar buffers beside it, and 2 MiB of rounding for each of five allocations."""
import ctypes

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8           # CU_MEMPOOL_ATTR_USED_MEM_HIGH
A, C = W.A_LATT, W.C_LATT
Z, X, TILT, ANY = [0, 0, 1], [1, 0, 0], [0, 0.6, 0.8], [1, 2, 2]
CART = [[A, 0, 0], [0, A, 0], [0, 0, C]]
FAMILIES = {
    "gan": None,
    "unmirrored": ([ANY] * 3, CART),
    "mirrored and not": ([Z] * 3 + [ANY] * 3, CART * 2),
    "all kinds": ([Z] * 3 + [TILT] * 3 + [[0.6, 0, 0.8]] * 3 + [ANY] * 3, CART * 4),
}


def pool():
    cu = ctypes.CDLL("libcuda.so.1")
    h = ctypes.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(h), 0) == 0
    return cu, h


@pytest.mark.parametrize("kind", list(FAMILIES))
@pytest.mark.parametrize("shape,periodic", [((128, 128, 64), False), ((128, 128, 64), True), ((200, 128, 33), False)])
def test_within_one_table_and_spectrum(kind, shape, periodic):
    import paper_1804_01830_gb300 as dds
    t, b = W.gan_families() if FAMILIES[kind] is None else (np.array(v, dtype=float) for v in FAMILIES[kind])
    t = t / np.linalg.norm(t, axis=1)[:, None]
    nx, ny, nz = shape
    ctx = dds.StressContext(0)
    ctx.set_geometry(nx, ny, nz, 0.2e-6, 0.2e-6, 0.1e-6, 68e9, 0.23).set_families(t, b)
    if periodic:
        ctx.set_option(dds.DDS_OPT_PBC_SHELLS, 1)
        ctx.set_option(dds.DDS_OPT_PBC_PERIODIC, 1)
    torch.cuda.synchronize()
    cu, h = pool()
    high = ctypes.c_uint64(0)
    assert cu.cuMemPoolSetAttribute(h, USED_MEM_HIGH, ctypes.byref(high)) == 0
    ctx.build_kernels()
    assert cu.cuMemPoolGetAttribute(h, USED_MEM_HIGH, ctypes.byref(high)) == 0
    q = ctx.query()
    ctx.close()
    px, py, pz = q["px"], q["py"], q["pz"]
    limit = 48 * px * py * pz + 16 * (px // 2 + 1) * py * pz
    assert 0 < high.value <= limit + 5 * (2 << 20), high.value / limit
