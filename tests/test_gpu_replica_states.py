"""Replicas as aliases of their main rows, against the CPU oracle, bit for bit (dyadic values).

Every worker but the last holds a replica of every key, so each write of a main row has every other holder's
alias to detach; the calls take a replica through each of its states (alias, pending, own value, folded) and out
of it by a sync or an eviction.  The sizes fill the kernels' lists: more holders than one round of lookups, more
(key, holder) pairs than a warp or a push block lists at once, more listed slots than a warp merges at once.
"""
import numpy as np
import pytest
import torch

from oracle import ParameterManagerOracle
from tests.test_gpu_store import compare_full_state, dev
from tests.seqgen import dyadic_init

pytestmark = pytest.mark.gpu

CASES = [
    # K, D, W (the last worker holds nothing)
    (3, 4, 2),
    (70, 36, 5),
    (700, 64, 9),      # 2,048 pairs and more per push block
    (300, 8, 32),      # 30 other holders per evicted replica
    (150, 132, 32),
    (90, 300, 4),
    (40, 1024, 3),
]


@pytest.mark.parametrize("refresh,staging", [(False, False), (True, False), (False, True)])
@pytest.mark.parametrize("K,D,W", CASES)
def test_every_state_and_way_out(gpu_lib, K, D, W, refresh, staging):
    init = dyadic_init(K, D, K + D)
    pm = gpu_lib.ParameterManager(K, D, W, init_values=torch.from_numpy(init).cuda(), delta_refresh=refresh,
                                  pull_staging=staging)
    ref = ParameterManagerOracle(K, D, W, init, delta_refresh=refresh)
    rng = np.random.default_rng(7)
    every = np.arange(K)

    def push(w, keys):
        d = (rng.integers(-64, 65, size=(len(keys), D)) * 2.0 ** -10).astype(np.float32)
        pm.push(w, dev(keys), torch.from_numpy(d).cuda())
        ref.push(w, keys, d)

    def both(call, *a):
        getattr(pm, call)(*a)
        getattr(ref, call)(*a)

    def intent(w, keys, a, b):
        pm.intent(w, dev(keys), a, b)
        ref.intent(w, keys, a, b)

    def check():
        for w in range(W):
            out = pm.pull(w, dev(every))
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), ref.pull(w, every)), w
        compare_full_state(pm, ref, K, W)

    for w in range(W - 1):
        intent(w, every, 0, 2)
        intent(w, every[::2], 3, 4)
    check()
    push(W - 1, rng.permutation(every))                      # main written under every alias
    check()
    both("sync")
    check()
    push(0, np.concatenate([every, every[::3]]))             # first push
    push(0, rng.permutation(every)[: K // 2])                # second push of some
    check()
    push(W - 1, every)                                       # main written under pending aliases
    for w in range(W - 1):
        push(w, rng.permutation(every)[: (2 * K) // 3])      # pushes on replicas with and without own values
    check()
    both("sync")                                             # every holder pending
    check()
    for w in range(W - 1):
        push(w, every[w % 3::3])
    for _ in range(2):
        for w in range(W - 1):
            both("advance_clock", w)                         # evictions with other holders left, one after another
            check() if W <= 9 else None
    check()
    for w in range(W - 1):
        both("advance_clock", w)                             # some keys come back
    push(0, every)
    both("sync")
    both("sync")
    check()
    pm.close()
