"""Inputs whose order is related to their keys: a segment's keys lie between
few probes, which the walking histogram must leave to the other forms.  Same
result as the oracle's, and no slower than with either of those forms forced."""
import numpy as np
import pytest

import oracle
from paper_1803_01237_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KINDS = ["sorted", "reversed", "blocks64", "runs64", "blocks8", "half", "tail"]


def _order(kind, keys):
    """keys (shuffled, int64) in an order of the given kind."""
    n, srt = keys.numel(), torch.sort(keys)[0]
    if kind == "sorted":
        return srt
    if kind == "reversed":
        return srt.flip(0).contiguous()
    if kind.startswith("blocks"):  # each block shuffled
        b = srt.view(int(kind[6:]), -1)
        g = torch.Generator(device="cuda").manual_seed(1)
        return b[:, torch.randperm(b.shape[1], device="cuda", generator=g)].reshape(-1).contiguous()
    if kind.startswith("runs"):
        return torch.sort(keys.view(int(kind[4:]), -1), dim=1)[0].reshape(-1).contiguous()
    if kind == "half":
        return torch.cat([keys[: n // 2], torch.sort(keys[n // 2:])[0]])
    if kind == "tail":  # a constant tail of a hundredth
        return torch.cat([keys[: n - n // 100], keys.new_full((n // 100,), 5)])
    raise ValueError(kind)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("flags", [16, 32])  # rounds driven from the host, and on the device
def test_result(kind, flags):
    from paper_1803_01237_gb300 import hss

    N, p, s = 1 << 22, 1900, 1.5 if flags == 32 else 5.0  # 1.5: a capacity of one on-chip sort
    k = _order(kind, torch.from_numpy(inputs.uniform(N, 2).view(np.int64)).cuda())
    res, _ = hss.partition(k, p, 0.05, 3, oversample=s, key_type="i64", flags=flags)
    ref = oracle.hss(k.cpu().numpy(), p, 0.05, 3, oversample=s, sort=False)
    assert res.rounds == ref.rounds
    assert res.sample_size == [int(x) for x in ref.sample_size]
    assert np.array_equal(res.offsets.cpu().numpy().astype(np.uint64), ref.offsets)
    assert np.array_equal(res.splitter_tags()[0].view(np.uint64), ref.splitter_key.view(np.uint64))


@pytest.mark.parametrize("kind", KINDS)
def test_rounds_no_slower_than_a_forced_form(kind):
    from paper_1803_01237_gb300 import hss

    g = torch.Generator(device="cuda").manual_seed(7)
    k = _order(kind, torch.randint(-(1 << 62), 1 << 62, (1 << 24,), device="cuda", generator=g) * 2)

    def ms(flags):
        best = float("inf")
        for i in range(8):
            res, _ = hss.partition(k, 4096, 0.02, 3, key_type="i64", flags=flags | hss.FLAG_TIMING)
            if i >= 2:
                best = min(best, res.ms_phase["rounds"])
        return best

    chosen, search, staged = ms(0), ms(hss.FLAG_HIST_PROBE), ms(hss.FLAG_HIST_STAGED)
    assert chosen < 1.15 * min(search, staged), (chosen, search, staged)
