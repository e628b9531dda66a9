"""What a caller has enqueued behind a push whose sort gave up leaves the store alone, as the header promises: an
advance that would have destroyed and created replicas, and a sync.  (The wait that gives up is bounded, about a
second; no GPU fault is involved.)"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("relocate,early", [(False, False), (False, True), (True, False)])
def test_advance_and_sync_after_a_failed_sort(gpu_lib, relocate, early):
    A, K, D, W = gpu_lib, 300, 8, 2
    init = torch.rand(K, D, device="cuda")
    pm = A.ParameterManager(K, D, W, init_values=init, relocate=relocate, early_events=early)
    old, new = torch.arange(0, 200, device="cuda"), torch.arange(150, 300, device="cuda")
    for w in range(W):
        pm.intent(w, old, 0, 1)
        pm.intent(w, new, 1, 2)
        pm.push(w, old, torch.rand(200, D, device="cuda"))   # pending updates
    pm.wait()
    state = [pm.read_main(np.arange(K))] + [x for w in range(W) for x in pm.replica_rows(w, np.arange(K))]
    pm.debug_fail_next_barrier()
    pm.push(1, new, torch.ones(150, D, device="cuda"))
    pm.advance_clock(1)
    pm.sync()
    pm.advance_clock(0)
    pm.sync()
    after = [pm.read_main(np.arange(K))] + [x for w in range(W) for x in pm.replica_rows(w, np.arange(K))]
    for i, (a, b) in enumerate(zip(state, after)):
        assert np.array_equal(a, b), f"array {i}"
    with pytest.raises(A.AdaPMError) as e:
        pm.wait()
    assert e.value.status == A.ETIMEOUT
    pm.close()
