"""The fused training step at the edges of its shape -- one point, a CTA's 128
points and one more, all 32 CTAs and a second share for some -- against the
float64 oracle, with an unaligned scratch buffer, and the steps of one call
against the same steps in several calls (the arrival counter starts over)."""
import numpy as np
import pytest

from oracle import cdf_mlp as M

pytestmark = pytest.mark.gpu


def _points(n, seed):
    g = np.random.Generator(np.random.Philox(key=[seed, 77]))
    keys = np.sort(np.minimum(np.exp(g.standard_normal(n) * 2.0 - 12.0), 1.0) * 9.0e18).astype(np.uint64)
    return keys, np.arange(n, dtype=np.uint64)


def _dev(a):
    import torch
    return torch.from_numpy(a.view(np.int64)).cuda()


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 4095, 4096, 4097, 9000])
def test_step_gradient_edges(n):
    import torch

    from paper_1803_01237_gb300 import hss
    keys, ranks = _points(n, 3)
    lo, hi = 1, (1 << 63) - 1
    m = hss.CDFModel().init(6, "log", lo, hi)
    theta = M.init(6) + 0.05 * np.random.default_rng(n).standard_normal(M.NPARAM)
    m.theta.copy_(torch.from_numpy(theta.astype(np.float32)))
    m._work = torch.empty(m._ws(n).numel() + 4, dtype=torch.uint8, device="cuda")[4:]  # scratch off a 16-byte boundary
    g, loss = m.grad(_dev(keys), _dev(ranks), n)
    x = M.feature(keys, M.LOG, np.log2(2.0), np.log2(float(1 << 63)))
    gref, lref = M.grad(m.theta.cpu().numpy().astype(np.float64), x, ranks.astype(np.float64) / n)
    # sums of at most 9000 float32 terms of one sign or less: relative error far below 1e-3 of the largest entry
    assert np.allclose(g.cpu().numpy(), gref, rtol=1e-3, atol=1e-4 * np.abs(gref).max())
    assert float(loss.item()) == pytest.approx(lref, rel=1e-4)


@pytest.mark.parametrize("n", [100, 4097])
def test_steps_of_one_call_equal_steps_of_several(n):
    import torch

    from paper_1803_01237_gb300 import hss
    keys, ranks = _points(n, 4)
    a = hss.CDFModel().init(8, "log", 1, (1 << 63) - 1)
    b = hss.CDFModel().init(8, "log", 1, (1 << 63) - 1)
    a.train(_dev(keys), _dev(ranks), n, 6, 0.01)
    for steps in (1, 2, 3):
        b.train(_dev(keys), _dev(ranks), n, steps, 0.01)
    assert a.step == b.step == 6 and torch.equal(a.theta, b.theta)
