"""Pushes and intents at the edges of the one-block sort's sizes (and the grid sort's first ones) against the oracle,
bit for bit with dyadic values: without a plan, with one, with a plan whose keys differ, and keys out of range."""
import numpy as np
import pytest
import torch

from oracle import ParameterManagerOracle
from tests.test_gpu_store import dev
from tests.seqgen import dyadic_init

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 300, 70_000, 3_000_000])   # 1, 2 and 3 passes
@pytest.mark.parametrize("n", [1, 33, 1023, 1024, 1025, 4096, 4097, 8192, 8193])
def test_sizes(gpu_lib, K, n):
    D = 4
    rng = np.random.default_rng(n + K)
    init = dyadic_init(K, D, 1)
    pm = gpu_lib.ParameterManager(K, D, 2, replica_capacity=4 * n + 16, init_values=torch.from_numpy(init).cuda())
    ref = ParameterManagerOracle(K, D, 2, init)
    keys = np.minimum(rng.integers(0, K, size=n), rng.integers(0, K, size=n))

    def push(w, k):
        d = (rng.integers(-64, 65, size=(len(k), D)) * 2.0 ** -10).astype(np.float32)
        pm.push(w, dev(k), torch.from_numpy(d).cuda())
        ref.push(w, k, d)

    for w in range(2):
        for api, k in ((pm, dev(keys)), (ref, keys)):
            api.intent(w, k, 1 + w, 3)       # a window at the next advance, one further on
            api.intent(w, k[: n // 2], 0, 1)       # active now
    push(0, keys)                            # no plan of n keys holds clock 0
    for api in (pm, ref):
        api.advance_clock(0)
        api.advance_clock(1)
        api.advance_clock(1)
    push(0, keys)                            # the plan's keys
    push(1, keys)
    if n > 1 and K > 1:
        push(1, np.roll(keys, 1))            # the plan's length, other keys
    pm.push_noalloc(0, dev(keys), torch.full((n, D), 0.25, device="cuda"))
    ref.push(0, keys, np.full((n, D), 0.25, np.float32))
    pm.wait()
    touched = np.unique(keys)
    for w in range(2):
        assert np.array_equal(pm.replica_keys(w), touched)
        out = pm.pull(w, dev(touched))
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), ref.pull(w, touched))
    for api in (pm, ref):
        api.sync()
    pm.wait()
    assert np.array_equal(pm.read_main(touched), ref.main[touched])
    st = pm.stats()
    assert st["planned_pushes"] == (3 if n > 1 and K > 1 else 2)
    assert st["plan_misses"] == (1 if n > 1 and K > 1 and not np.array_equal(np.roll(keys, 1), keys) else 0)
    pm.close()


@pytest.mark.parametrize("n", [40, 4096, 8192, 9000])
def test_keys_out_of_range(gpu_lib, n):
    K, D = 1000, 4
    pm = gpu_lib.ParameterManager(K, D, 1)
    keys = np.arange(n) % K
    keys[[3, n - 1]] = [K, 0xFFFFFFFF]
    for call in (lambda: pm.intent(0, dev(keys), 1, 2), lambda: pm.push(0, dev(keys), torch.ones(n, D, device="cuda"))):
        call()
        with pytest.raises(gpu_lib.AdaPMError) as e:
            pm.wait()
        assert e.value.status == gpu_lib.ERANGE
    good = keys[keys < K]
    want = np.bincount(good, minlength=K)[:, None] * np.ones(D)
    assert np.array_equal(pm.read_main(np.arange(K)), want)
    pm.advance_clock(0)
    assert np.array_equal(pm.replica_keys(0), np.unique(good))
    pm.close()


# 32,768 keys: the last size whose plan scans in its scatter (its blocks' digit counts fit one pass), 32,769 the next
@pytest.mark.parametrize("n,ahead", [(100, 1), (4097, 1), (4097, 2), (32_768, 2), (32_769, 2)])
def test_device_keys_may_change_behind_an_intent(gpu_lib, n, ahead):
    """An intent reads device keys in stream order, whichever stream sorts or lists them."""
    K, D = 70_000, 4
    rng = np.random.default_rng(n + ahead)
    stream = torch.cuda.Stream()
    pm = gpu_lib.ParameterManager(K, D, 1, stream=stream)
    keys = rng.integers(0, K, size=n)
    with torch.cuda.stream(stream):
        d = torch.from_numpy(keys.astype(np.int32)).cuda()
        for _ in range(20):                # (many, so that the side streams lag)
            pm.intent(0, d, ahead, ahead + 1)
        d.fill_(5)
    for _ in range(ahead):
        pm.advance_clock(0)
    stream.synchronize()
    pm.wait()
    assert np.array_equal(pm.replica_keys(0), np.unique(keys))
    assert pm.refcounts(0, np.unique(keys)).tolist() == [20] * len(np.unique(keys))
    with torch.cuda.stream(stream):
        pm.push(0, dev(keys), torch.ones(n, D, device="cuda"))
    pm.wait()
    pm.sync()
    pm.wait()
    assert np.array_equal(pm.read_main(np.arange(K)), np.bincount(keys, minlength=K)[:, None] * np.ones(D))
    st = pm.stats()
    assert (st["planned_pushes"], st["plan_misses"]) == (1, 0)
    pm.close()
