"""hss_set_tuning: what is asked for is what the sort does.  The tilings change
no result, so they are read off the plan in the workspace and the launches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N, P = 1 << 22, 64  # 2^22 keys: a level that packs fully by itself


@pytest.fixture()
def hss():
    from paper_1803_01237_gb300 import hss as h
    h.reset_tuning()
    yield h
    h.reset_tuning()


def _packs(counts, limit):
    """Packs of consecutive sub-buckets (none above the on-chip size) of at most
    limit keys, those without keys left out."""
    packs = run = 0
    for c in counts:
        if run and run + c > limit:
            packs, run = packs + 1, 0
        run += int(c)
    return packs + (run > 0)


@pytest.mark.parametrize("asked,limit", [(None, 1536), (0, 1536), (1024, 1024), (1023, 1023), (1536, 1536)])
def test_pack_keys(hss, asked, limit):
    rng = np.random.default_rng(5)
    keys = rng.integers(0, 1 << 63, size=N, dtype=np.uint64) * np.uint64(2)
    expect = sum(_packs(np.bincount((seg >> np.uint64(56)).astype(np.int64), minlength=256), limit)
                 for seg in keys.reshape(P, -1))
    dk = torch.from_numpy(keys.view(np.int64)).cuda()
    out = torch.empty_like(dk)
    ws = torch.full((hss.workspace_bytes("local_sort", N, P, "u64", False),), 255, dtype=torch.uint8, device="cuda")
    if asked is not None:
        hss.set_tuning(pack_keys=asked)
        assert hss.get_tuning()["pack_keys"] == (asked or 1024)
    rc = hss.load().hss_local_sort(dk.data_ptr(), None, hss.KEY_TYPES["u64"], N, P, out.data_ptr(), None, ws.data_ptr(),
                                   ws.numel(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rc == 0
    # the last level's counts: segments of the first class, and none of the other classes, large ones or tiles
    w = ws[: ws.numel() // 4 * 4].view(torch.int32).cpu().numpy()
    at = np.flatnonzero(w[:-4] == expect)
    assert any((w[i + 1:i + 5] == 0).all() for i in at)


@pytest.mark.parametrize("asked", [None, 0, 1])
@pytest.mark.parametrize("p", [P, 512])
def test_first_split(hss, asked, p):
    """A sample is one launch: of every local sort (1), of none (0), and where
    nothing was asked for, of segments of 2^15 keys and more."""
    keys = torch.randint(-(1 << 62), 1 << 62, (N,), device="cuda") * 2

    def launches():
        before = hss.launch_count()
        hss.local_sort(keys, p)
        torch.cuda.synchronize()
        return hss.launch_count() - before

    hss.set_tuning(first_split=0)
    plain = launches()
    hss.set_tuning(first_split=1)
    sampled = launches()
    assert sampled == plain + 1
    if asked is None:
        hss.reset_tuning()
    else:
        hss.set_tuning(first_split=asked)
    assert hss.get_tuning()["first_split"] == (asked or 0)
    by_size = sampled if N // p >= 1 << 15 else plain
    assert launches() == (by_size if asked is None else sampled if asked else plain)
