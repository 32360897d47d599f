"""Batches whose segments are of very different lengths: many short ones and a
few long ones, which the rounds' passes by segment must not leave to one warp."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# Longest segment: at four times 2^15 (by warps), a key more and 2^18 (by CTAs).
@pytest.mark.parametrize("longest", [1 << 17, (1 << 17) + 1, 1 << 18])
def test_uneven_batch_matches_oracle(longest):
    from paper_1803_01237_gb300 import hss

    g = np.random.Generator(np.random.Philox(key=[5, longest]))
    sizes, ps = [700] * 60 + [2 * longest] + [1000 + j for j in range(40)], [7] * 60 + [2] + [5] * 40
    keys = g.integers(0, 1 << 63, size=sum(sizes), dtype=np.uint64)
    r = hss.partition_batch(torch.from_numpy(keys.view(np.int64)).cuda(), sizes, ps, 0.02, 4, key_type="u64")
    off = r.offsets.cpu().numpy().astype(np.uint64)
    a = o = 0
    for j, (n, p) in enumerate(zip(sizes, ps)):
        ref = oracle.hss(keys[a:a + n], p, 0.02, 4 + j, sort=False)
        assert r.job_rounds[j] == ref.rounds
        assert r.job_sample_size[j] == [int(x) for x in ref.sample_size], j
        assert np.array_equal(off[o:o + p + 1], ref.offsets), j
        a += n
        o += p + 1


def test_one_long_job_beside_many_short_ones():
    """The rounds of 4096 short jobs and a job of 2^26 keys on four processors
    take no longer than the two apart (by a warp per segment 1.5 times that)."""
    from paper_1803_01237_gb300 import hss

    gen = torch.Generator(device="cuda").manual_seed(1)
    short, long_ = ([1 << 14] * 4096, [4] * 4096), ([1 << 26], [4])
    keys = torch.randint(-(1 << 62), 1 << 62, (1 << 27,), device="cuda", generator=gen) * 2

    def rounds_ms(sizes, ps):
        best = float("inf")
        for i in range(7):
            r = hss.partition_batch(keys[:sum(sizes)], sizes, ps, 0.05, 3, key_type="i64", flags=hss.FLAG_TIMING)
            if i >= 2:
                best = min(best, r.ms_phase["rounds"])
        return best

    apart = rounds_ms(*short) + rounds_ms(*long_)
    assert rounds_ms(short[0] + long_[0], short[1] + long_[1]) < 1.25 * apart
