"""The walking histogram (rounds of many probes in short segments) against the
CPU oracle: same rounds, samples, splitters and offsets."""
import numpy as np
import pytest

import oracle
from paper_1803_01237_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _keys(kind, N, seed):
    if kind == "equal":
        return np.full(N, 7, dtype=np.uint64)
    if kind == "ends":  # many copies of the smallest and the largest key
        ends = np.array([0, 1, 2**64 - 2, 2**64 - 1], dtype=np.uint64)
        return ends[np.random.default_rng(seed).integers(0, 4, N)]
    if kind == "sorted":  # a segment's keys lie between few probes
        return np.sort(inputs.uniform(N, seed))
    return getattr(inputs, kind)(N, seed)


# Segments of 4 to 2200 keys, a last warp of segments that is not full, and
# (oversample 1.5: a capacity of one on-chip sort) device-driven rounds.
@pytest.mark.parametrize("kind", ["uniform", "zipf", "equal", "ends", "sorted"])
@pytest.mark.parametrize("N,p,oversample", [(20011, 1900, 5.0), (1 << 14, 3400, 1.5), (40009, 4099, 5.0),
                                            ((1 << 22) + 3, 1900, 5.0)])
def test_walk_matches_oracle(kind, N, p, oversample):
    from paper_1803_01237_gb300 import hss

    keys = _keys(kind, N, 5)
    res, _ = hss.partition(torch.from_numpy(keys.view(np.int64)).cuda(), p, 0.05, 11, oversample=oversample,
                           key_type="u64")
    ref = oracle.hss(keys, p, 0.05, 11, oversample=oversample, sort=False)
    assert res.rounds == ref.rounds
    assert res.sample_size == [int(x) for x in ref.sample_size]
    assert res.gamma == [int(x) for x in ref.gamma]
    assert np.array_equal(res.offsets.cpu().numpy().astype(np.uint64), ref.offsets)
    k, s, sp = res.splitter_tags()
    assert np.array_equal(k.view(np.uint64), ref.splitter_key.view(np.uint64))
    assert np.array_equal(s, ref.splitter_seg)
    assert np.array_equal(sp, ref.splitter_spos)
