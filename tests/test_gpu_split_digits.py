"""Sampled splitters with the digits kept between the statistics and the split
pass: ragged last tiles, and the sort in place (where the output cannot hold
them and they are found again)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("payload", [False, True])
@pytest.mark.parametrize("p", [1, 13, 100])
def test_clustered_segments(p, payload, in_place):
    from paper_1803_01237_gb300 import hss

    n = (1 << 22) + 4097 * (p + 1) + 3
    g = torch.Generator(device="cuda").manual_seed(p)
    centre = torch.randint(0, 1 << 62, (9,), device="cuda", generator=g)
    k = centre[torch.randint(0, 9, (n,), device="cuda", generator=g)]
    k = k + (torch.randn(n, device="cuda", generator=g, dtype=torch.float64) * 3e7).long()
    pay = torch.arange(n, device="cuda", dtype=torch.int32) if payload else None
    want, order = [], []
    for s in range(p):
        a, b = s * n // p, (s + 1) * n // p
        v, i = torch.sort(k[a:b], stable=True)
        want.append(v)
        order.append(i + a)
    src, psrc = k.clone(), pay.clone() if payload else None
    out, pout = (src, psrc) if in_place else (torch.empty_like(k), torch.empty_like(pay) if payload else None)
    hss.local_sort(src, p, payload=psrc, key_type="i64", out=out, out_payload=pout)
    assert torch.equal(out, torch.cat(want))
    if payload:
        assert torch.equal(pout.long(), torch.cat(order))
