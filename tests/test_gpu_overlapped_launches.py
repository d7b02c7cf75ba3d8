"""Evaluations enqueued back to back, whose kernels may start before the ones ahead of them
have finished: each result equals the same evaluation alone (bit for bit), with densities
overwritten on the stream between the calls, outputs reused, two contexts in turn, the Eq. 20
statistics, and inside a captured graph.  Sizes: one CTA wave, ragged lines, several waves."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def context(dds, shape, fams):
    t, b = W.gan_families()
    p = W.random_problem(W.Geometry(*shape, 0.2e-6, 0.2e-6, 0.05e-6), t[fams], b[fams], seed=sum(shape))
    return dds.context_for(p), torch.from_numpy(p.rho.astype(np.float32)).cuda()


@pytest.mark.parametrize("shape,fams", [((32, 32, 8), [0]), ((33, 17, 9), [0, 7, 8]), ((20, 30, 40), list(range(18))),
                                        ((300, 40, 20), [0, 1, 2, 9]), ((128, 200, 70), list(range(18)))])
def test_back_to_back_equals_alone(shape, fams):
    import paper_1804_01830_gb300 as dds
    a, rho_a = context(dds, shape, fams)
    b, rho_b = context(dds, tuple(max(1, n // 2) for n in shape), fams)
    scales = [1.0, 0.5, -2.0, 3.0, 0.25, 1.5]
    alone = []
    for s in scales:
        torch.cuda.synchronize()
        x = a.stress(rho_a * s)
        torch.cuda.synchronize()
        y = b.stress(rho_b * s)
        torch.cuda.synchronize()
        alone.append((x.clone(), y.clone()))
    _, stat = a.stress_stats(rho_a * scales[1])
    torch.cuda.synchronize()
    for _ in range(5):
        cur_a, cur_b = torch.empty_like(rho_a), torch.empty_like(rho_b)
        out_a, out_b = torch.empty_like(alone[0][0]), torch.empty_like(alone[0][1])
        keep = []
        for s in scales:                     # nothing synchronises inside this loop
            torch.mul(rho_a, s, out=cur_a)
            a.stress(cur_a, out_a)
            torch.mul(rho_b, s, out=cur_b)
            b.stress(cur_b, out_b)
            a.stress(cur_a, out_a)
            keep.append((out_a.clone(), out_b.clone()))
        torch.mul(rho_a, scales[1], out=cur_a)
        sig, st = a.stress_stats(cur_a)
        torch.cuda.synchronize()
        for got, ref in zip(keep, alone):
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        assert torch.equal(sig, alone[1][0])
        assert torch.allclose(st, stat, rtol=1e-6, atol=0)      # FP64 atomics: order of the sums only
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a.stress(cur_a, out_a)
        b.stress(cur_b, out_b)
    for s, ref in zip(scales, alone):
        torch.mul(rho_a, s, out=cur_a)
        torch.mul(rho_b, s, out=cur_b)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out_a, ref[0]) and torch.equal(out_b, ref[1])
    a.close()
    b.close()
