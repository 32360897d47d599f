"""The recount of a first level whose keys agree in their top byte (row ids,
timestamps, small integers): a few segments of many tiles, beside segments that
need none, against torch's stable sort; and its cost, which must not depend on
how few segments there are."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _check(k, p, payload, key_type="i64"):
    from paper_1803_01237_gb300 import hss

    n = k.numel()
    pay = torch.arange(n, device="cuda", dtype=torch.int32) if payload else None
    o = hss.local_sort(k, p, payload=pay, key_type=key_type)
    keys, pout = o if payload else (o, None)
    for s in range(p):
        a, b = s * n // p, (s + 1) * n // p
        v, i = torch.sort(k[a:b], stable=True)
        assert torch.equal(keys[a:b], v), (p, s)
        if payload:
            assert torch.equal(pout[a:b].long(), i + a), (p, s)


# One tile and a key, tiles for some CTAs twice (1217 and more), 256 tiles of
# one CTA and the next; bits: the keys' width, their top byte 4, 1 or 0.
@pytest.mark.parametrize("payload", [False, True])
@pytest.mark.parametrize("n,p,bits", [(4097, 1, 40), (3 * 4096 + 5, 1, 9), (1217 * 4096 + 1, 1, 40), (1 << 22, 3, 12),
                                      (2433 * 4096 + 77, 4, 33), ((1 << 24) + 12345, 16, 40)])
def test_narrow_keys(n, p, bits, payload):
    g = torch.Generator(device="cuda").manual_seed(n + p)
    _check(torch.randint(0, 1 << bits, (n,), device="cuda", generator=g), p, payload)


@pytest.mark.parametrize("payload", [False, True])
def test_narrow_segments_beside_wide_ones(payload):
    """Of four segments the first and the last are counted again, by different bytes."""
    g = torch.Generator(device="cuda").manual_seed(9)
    n = 1 << 22
    k = torch.randint(-(1 << 62), 1 << 62, (n,), device="cuda", generator=g) * 2
    k[: n // 4] = torch.randint(0, 1 << 20, (n // 4,), device="cuda", generator=g)
    k[3 * n // 4:] = torch.randint(1 << 52, (1 << 52) + (1 << 35), (n // 4,), device="cuda", generator=g)
    _check(k, 4, payload)


def test_one_segment_is_counted_by_the_whole_chip():
    """2^26 keys in one segment: counting them again reads them once more, a few
    per cent of the sort.  By eight CTAs it takes twice the sort's time."""
    from paper_1803_01237_gb300 import hss

    g = torch.Generator(device="cuda").manual_seed(3)
    n = 1 << 26
    out = torch.empty(n, device="cuda", dtype=torch.int64)
    times = []
    for k in (torch.randint(-(1 << 62), 1 << 62, (n,), device="cuda", generator=g) * 2,
              torch.randint(0, 1 << 40, (n,), device="cuda", generator=g)):
        best = float("inf")
        for i in range(7):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            hss.local_sort(k, 1, key_type="i64", out=out)
            e1.record()
            torch.cuda.synchronize()
            if i >= 2:
                best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[1] < 1.5 * times[0], times
