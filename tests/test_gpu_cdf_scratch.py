"""Training with scratch that was sized for fewer points: a partial for every
256 points, 32 at most, is enough whatever the number of points.  Gradients and
losses against the float64 oracle, a step of Adam against the same step with
all the scratch it asks for, and one byte less refused."""
import numpy as np
import pytest

from oracle import cdf_mlp as M

pytestmark = pytest.mark.gpu

PARTIAL = 4624  # bytes: 1153 gradients, the loss, padding


def _points(n, seed):
    g = np.random.Generator(np.random.Philox(key=[seed, 78]))
    keys = np.sort(np.minimum(np.exp(g.standard_normal(n) * 2.0 - 12.0), 1.0) * 9.0e18).astype(np.uint64)
    return keys, np.arange(n, dtype=np.uint64)


def _dev(a):
    import torch
    return torch.from_numpy(a.view(np.int64)).cuda()


# one CTA, a second one, their last points; 32 CTAs, and the scratch of 8192 points for more
@pytest.mark.parametrize("offset", [0, 4])
@pytest.mark.parametrize("n", [1, 128, 256, 257, 4097, 8192, 20001])
def test_least_scratch(n, offset):
    import torch

    from paper_1803_01237_gb300 import hss
    lib = hss.load()
    assert int(lib.hss_cdf_work_bytes(n)) > PARTIAL * min(32, -(-n // 256))
    keys, ranks = _points(n, 3)
    dk, dr = _dev(keys), _dev(ranks)
    a = hss.CDFModel().init(6, "log", 1, (1 << 63) - 1)
    theta = M.init(6) + 0.05 * np.random.default_rng(n).standard_normal(M.NPARAM)
    a.theta.copy_(torch.from_numpy(theta.astype(np.float32)))
    b = hss.CDFModel()
    b.buf.copy_(a.buf)
    nb = PARTIAL * min(32, -(-n // 256))
    ws = torch.full((nb + offset,), 255, dtype=torch.uint8, device="cuda")[offset:]
    g = torch.empty(hss.CDF_NPARAM, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream

    def grad(nbytes):
        return lib.hss_cdf_grad(a.buf.data_ptr(), dk.data_ptr(), dr.data_ptr(), n, n, g.data_ptr(), loss.data_ptr(),
                                ws.data_ptr(), nbytes, stream)

    assert grad(nb - 1) == hss.ERR_WORKSPACE
    assert grad(nb) == 0
    x = M.feature(keys, M.LOG, np.log2(2.0), np.log2(float(1 << 63)))
    gref, lref = M.grad(a.theta.cpu().numpy().astype(np.float64), x, ranks.astype(np.float64) / n)
    # sums of at most 20001 float32 terms: relative error far below 1e-3 of the largest entry
    assert np.allclose(g.cpu().numpy(), gref, rtol=1e-3, atol=1e-4 * np.abs(gref).max())
    assert float(loss.item()) == pytest.approx(lref, rel=1e-4)
    # Adam's step is lr (m / c1) / (sqrt(v / c2) + 1e-8), lr in the first step: its sign where the gradient
    # is clear of its rounding
    assert lib.hss_cdf_train(a.buf.data_ptr(), dk.data_ptr(), dr.data_ptr(), n, n, 1, 0.01, loss.data_ptr(),
                             ws.data_ptr(), nb, stream) == 0
    b.train(dk, dr, n, 1, 0.01)
    clear = torch.from_numpy(np.abs(gref) > 1e-3 * np.abs(gref).max()).cuda()
    assert a.step == b.step == 1 and torch.allclose(a.theta[clear], b.theta[clear], rtol=0, atol=1e-4)
