"""The on-chip sort at the edges of its classes, windows and groups, against
numpy's stable sort: sizes around the class limits and the window of eight,
segment starts that are not 16- or 32-byte aligned, crowded and duplicated
keys (the refined groups, the run sort of keys the 32-bit words do not tell
apart, groups of one value) and both key types."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 7, 8, 9, 31, 33, 1023, 1024, 1025, 1033, 1535, 1536, 1537, 2047, 4089, 4095, 4096, 4097, 14335, 14336,
         14337]


def _keys(kind, n, g):
    r = g.integers(0, 1 << 63, size=n, dtype=np.uint64) * np.uint64(2) + g.integers(0, 2, size=n, dtype=np.uint64)
    if kind == "uniform":
        return r
    if kind == "narrow":  # all high words equal
        return (np.uint64(0x123456789) << np.uint64(28)) + (r >> np.uint64(45))
    if kind == "clusters":  # a few narrow clusters: one group holds most of the segment
        return (r >> np.uint64(40)) + (g.integers(0, 3, size=n).astype(np.uint64) << np.uint64(61))
    if kind == "orders":  # every binary order of magnitude
        return r >> g.integers(0, 64, size=n).astype(np.uint64)
    if kind == "close":  # distinct keys that agree in their upper 40 bits, among spread ones
        return np.where(g.random(n) < 0.3, (r & np.uint64(0x7)) + np.uint64(1 << 62), r)
    if kind == "few":  # groups of one value
        return g.integers(0, 5, size=n).astype(np.uint64) << np.uint64(40)
    if kind == "pairs":  # every key about twice
        return r[g.integers(0, max(1, n // 2), size=n)]
    if kind == "ends":  # the smallest and largest values of both key types
        return np.array([0, 1, (1 << 63) - 1, 1 << 63, (1 << 64) - 2, (1 << 64) - 1], dtype=np.uint64)[
            g.integers(0, 6, size=n)]
    if kind == "border":  # small values of both signs: narrow around a border of the high words
        return (r.view(np.int64) >> g.integers(30, 64, size=n)).view(np.uint64) + (r & np.uint64(1) << np.uint64(32))
    if kind == "ladder":  # 60 close keys under outliers at every order of magnitude: each count peels off one
        return np.where(np.arange(n) % 97 < 60, r & np.uint64(0xffff),
                        np.uint64(1) << (np.uint64(16) + r % np.uint64(48)))
    raise ValueError(kind)


@pytest.mark.parametrize("payload", [False, True])
@pytest.mark.parametrize("kind", ["uniform", "narrow", "clusters", "orders", "close", "few", "pairs", "ends", "ladder", "border"])
def test_on_chip_sort_edges(kind, payload):
    import torch

    from paper_1803_01237_gb300 import hss

    g = np.random.Generator(np.random.Philox(key=[17, sum(map(ord, kind))]))
    for n in SIZES:
        # 1 segment, and (for the larger sizes) 3 segments of n keys in a larger call
        for p, shift in ((1, 0), (1, 1), (3, 3), (40, 2)):
            if p == 40 and n > 4097:
                continue
            N = n * p
            for key_type in ("u64", "i64"):
                raw = _keys(kind, N + shift, g)
                kv = raw.view(np.int64) if key_type == "i64" else raw
                dk = torch.from_numpy(raw.view(np.int64)).cuda()[shift:]
                pay = np.arange(N + shift, dtype=np.int32)
                dp = torch.from_numpy(pay).cuda()[shift:] if payload else None
                out = torch.empty(N + 3, dtype=torch.int64, device="cuda")[shift:shift + N]
                o = hss.local_sort(dk, p, payload=dp, key_type=key_type, out=out)
                off = [(s * N) // p for s in range(p + 1)]
                want = np.concatenate([shift + off[s] + np.argsort(kv[shift + off[s]:shift + off[s + 1]], kind="stable")
                                       for s in range(p)])
                assert np.array_equal(out.cpu().numpy(), raw.view(np.int64)[want]), (kind, n, p, shift, key_type)
                if payload:
                    assert np.array_equal(o[1].cpu().numpy(), pay[want]), (kind, n, p, shift, key_type)


@pytest.mark.parametrize("payload", [False, True])
@pytest.mark.parametrize("kind", ["uniform", "clusters", "orders", "nested", "runs"])
def test_first_split_of_clustered_segments(kind, payload):
    """Segments large enough to be sampled, at both ends of the range that
    takes sampled splitters and ragged in between: clustered keys (split on
    splitters), keys whose crowding is duplicates (the byte split stays) and
    uniform ones."""
    import torch

    from paper_1803_01237_gb300 import hss

    N = (1 << 22) + 3
    g = np.random.Generator(np.random.Philox(key=[23, sum(map(ord, kind))]))
    r = g.integers(0, 1 << 63, size=N, dtype=np.uint64) * np.uint64(2) + g.integers(0, 2, size=N, dtype=np.uint64)
    if kind == "clusters":
        means = g.integers(0, 1 << 63, size=32, dtype=np.uint64) * np.uint64(2)
        r = means[g.integers(0, 32, size=N)] + np.rint(g.standard_normal(N) * 2.0**40).astype(np.int64).view(np.uint64)
    elif kind == "orders":
        r = r >> g.integers(0, 64, size=N).astype(np.uint64)
    elif kind == "nested":  # clusters far narrower than a splitter resolves, and one value with a third of the keys
        r = np.where(g.random(N) < 0.33, np.uint64(77), (r >> np.uint64(44)) + (r % np.uint64(9) << np.uint64(60)))
    elif kind == "runs":  # long runs of equal keys next to each other in the input
        r = np.repeat(r[: N // 50 + 1] >> np.uint64(50), 50)[:N]
    pay = np.arange(N, dtype=np.int32)
    for p in (8, 9, 127, 128):
        for key_type in ("u64", "i64"):
            kv = r.view(np.int64) if key_type == "i64" else r
            o = hss.local_sort(torch.from_numpy(r.view(np.int64)).cuda(), p, key_type=key_type,
                               payload=torch.from_numpy(pay).cuda() if payload else None)
            off = [(s * N) // p for s in range(p + 1)]
            want = np.concatenate([off[s] + np.argsort(kv[off[s]:off[s + 1]], kind="stable") for s in range(p)])
            assert np.array_equal((o[0] if payload else o).cpu().numpy(), r.view(np.int64)[want]), (kind, p, key_type)
            if payload:
                assert np.array_equal(o[1].cpu().numpy(), pay[want]), (kind, p, key_type)
