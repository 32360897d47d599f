"""Branches that the other tests' sizes do not reach: workspaces off a 16-byte
boundary, the walking histogram for signed keys and for proposed cuts, and the
sampled first split of host arrays and of batches."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1803_01237_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _same(res, ref):
    assert res.rounds == ref.rounds
    assert res.sample_size == [int(x) for x in ref.sample_size]
    assert res.gamma == [int(x) for x in ref.gamma]
    assert np.array_equal(res.offsets.cpu().numpy().astype(np.uint64), ref.offsets)
    k, s, sp = res.splitter_tags()
    assert np.array_equal(k.view(np.uint64), ref.splitter_key.view(np.uint64))
    assert np.array_equal(s, ref.splitter_seg)
    assert np.array_equal(sp, ref.splitter_spos)


@pytest.fixture(scope="module", autouse=True)
def _profiler_started():
    """The first profile of a process may start too late to see a kernel."""
    _kernels(lambda: torch.zeros(1, device="cuda"))


def _kernels(call):
    """The kernels that a call launched, by name, and its result."""
    from torch.profiler import ProfilerActivity, profile

    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        res = call()
        torch.cuda.synchronize()
    return {e.key for e in prof.key_averages()}, res


def _ran(kernel, names):
    return not names or any(kernel in n for n in names)  # no names: the process is profiled by something else


# Marks taken by a warp per segment, and by a CTA.
@pytest.mark.parametrize("p", [64, 8])
@pytest.mark.parametrize("offset", [8, 16])
def test_workspace_off_16_bytes(p, offset):
    from paper_1803_01237_gb300 import hss

    lib, N, eps, seed = hss.load(), (1 << 20) + 13, 0.02, 6
    keys = inputs.gauss_mix(N, seed)
    dk = _dev(keys)
    prm = hss._params(p, eps, seed, 5.0, 0, hss.FLAG_HOST_ROUNDS)
    nb = int(lib.hss_workspace_bytes(hss.OP["partition"], N, ctypes.byref(prm), p, hss.KEY_TYPES["u64"], 0))
    ws = torch.full((nb + offset,), 255, dtype=torch.uint8, device="cuda")[offset:]
    spl = torch.empty((p - 1, 2), dtype=torch.int64, device="cuda")
    off = torch.empty(p + 1, dtype=torch.int64, device="cuda")
    st = hss.Stats()
    rc = lib.hss_partition(dk.data_ptr(), hss.KEY_TYPES["u64"], N, ctypes.byref(prm), spl.data_ptr(), off.data_ptr(),
                           ws.data_ptr(), nb, ctypes.byref(st), torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    _same(hss._result(None, None, spl, off, st), oracle.hss(keys, p, eps, seed, sort=False))


def test_batch_workspace_off_16_bytes():
    from paper_1803_01237_gb300 import hss

    sizes, ps = [40000, 7, 100001, 1 << 16], [5, 2, 16, 4]
    keys = inputs.zipf(sum(sizes), 3)
    ws = torch.full(((1 << 26) + 8,), 255, dtype=torch.uint8, device="cuda")[8:]
    r = hss.partition_batch(_dev(keys), sizes, ps, 0.05, 9, key_type="u64", ws=ws)
    off = r.offsets.cpu().numpy().astype(np.uint64)
    a = o = 0
    for j, (n, p) in enumerate(zip(sizes, ps)):
        ref = oracle.hss(keys[a:a + n], p, 0.05, 9 + j, sort=False)
        assert r.job_sample_size[j] == [int(x) for x in ref.sample_size] and np.array_equal(off[o:o + p + 1], ref.offsets)
        a, o = a + n, o + p + 1


@pytest.mark.parametrize("kind", ["uniform", "equal", "signs"])
def test_walk_of_signed_keys(kind):
    from paper_1803_01237_gb300 import hss

    N, p = 40009, 4099
    keys = inputs.uniform(N, 5).view(np.int64)
    if kind == "equal":
        keys = np.full(N, -7, dtype=np.int64)
    if kind == "signs":  # both ends and both sides of zero, many times each
        keys = np.array([-2**63, -1, 0, 1, 2**63 - 1], dtype=np.int64)[np.random.default_rng(2).integers(0, 5, N)]
    dk = _dev(keys)
    names, (res, _) = _kernels(lambda: hss.partition(dk, p, 0.05, 11, key_type="i64", flags=hss.FLAG_HOST_ROUNDS))
    assert _ran("k_histogram_walk", names)
    _same(res, oracle.hss(keys, p, 0.05, 11, sort=False))


@pytest.mark.parametrize("key_type", ["u64", "i64"])
@pytest.mark.parametrize("kind", ["quantiles", "ends"])
def test_walk_of_proposed_cuts(kind, key_type):
    """2^24 positions of proposed cuts, non-member cuts all: quantiles that leave
    no round to do; unsorted, repeated, the smallest and largest key among them."""
    from paper_1803_01237_gb300 import hss

    N, p, eps = 40009, 4099, 1.9 if kind == "quantiles" else 0.05
    keys = inputs.zipf(N, 3) if kind == "ends" else inputs.uniform(N, 5)
    if kind == "ends":
        keys[:40], keys[40:80] = np.uint64(0), np.uint64(2**64 - 1)
    if key_type == "i64":
        keys = keys.view(np.int64)
    prop = np.sort(keys)[(np.arange(1, p + 1) * N) // (p + 1)]
    if kind == "ends":
        g = np.random.default_rng(4)
        prop = np.concatenate([prop[::2], prop[::4], prop[::4]])[:p]
        prop[g.integers(0, p, 600)] = np.uint64(0).astype(keys.dtype)
        prop[g.integers(0, p, 600)] = np.iinfo(keys.dtype).max
        prop[g.integers(0, p, 600)] = np.iinfo(keys.dtype).min
        g.shuffle(prop)
    assert prop.size * p >= 1 << 24
    dk, dp = _dev(keys), _dev(prop)
    names, (res, _) = _kernels(lambda: hss.partition_with_proposal(dk, p, eps, 11, dp, key_type=key_type,
                                                                   flags=hss.FLAG_HOST_ROUNDS))
    assert _ran("k_histogram_walk", names)
    assert res.rounds == 0 or kind == "ends"
    _same(res, oracle.hss(keys, p, eps, 11, sort=False, proposal=prop))


def _clustered(n, g):
    centre = torch.randint(0, 1 << 62, (11,), device="cuda", generator=g)
    k = centre[torch.randint(0, 11, (n,), device="cuda", generator=g)]
    return k + (torch.randn(n, device="cuda", generator=g, dtype=torch.float64) * 1e9).long()


def _stable(k):
    v, i = torch.sort(k, stable=True)
    return v.cpu().numpy(), i.cpu().numpy().astype(np.int32)


def test_clustered_host_arrays_in_chunks():
    """Two chunks of processors, each sampled and split with kept digits."""
    from paper_1803_01237_gb300 import hss

    n, p = (1 << 25) + 12345, 100
    k = _clustered(n, torch.Generator(device="cuda").manual_seed(1))
    keys, pay = k.cpu().numpy(), np.arange(n, dtype=np.int32)
    want, order = _stable(k)
    names, (out, outp, _, off, _) = _kernels(lambda: hss.sort_host(keys, p, 0.05, 2, payload=pay, key_type="i64"))
    assert _ran("k_seg_sample", names)
    assert np.array_equal(out, want) and np.array_equal(outp, order)
    assert off[0] == 0 and off[-1] == n


@pytest.mark.parametrize("payload", [False, True])
def test_clustered_batch(payload):
    from paper_1803_01237_gb300 import hss

    sizes, ps = [1 << 20, 700001, 3, 1 << 21, 1234567, 4096], [8, 5, 1, 16, 9, 1]
    k = _clustered(sum(sizes), torch.Generator(device="cuda").manual_seed(2))
    pay = torch.arange(sum(sizes), device="cuda", dtype=torch.int32) if payload else None
    names, r = _kernels(lambda: hss.sort_batch(k, sizes, ps, 0.05, 4, payload=pay, key_type="i64"))
    assert _ran("k_seg_sample", names)
    a = 0
    for n in sizes:
        want, order = _stable(k[a:a + n])
        assert np.array_equal(r.keys[a:a + n].cpu().numpy(), want)
        if payload:
            assert np.array_equal(r.payload[a:a + n].cpu().numpy(), order + a)
        a += n
