"""adapm_debug_fail_next_barrier applies to the next eager push of its context, whatever sort its size would take,
and to no recorded one.  The wait that gives up is bounded (about a second); no GPU fault is involved."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("n", [500, 20_000])
def test_recorded_push_is_not_the_one_that_fails(gpu_lib, n, noalloc):
    A, K, D = gpu_lib, 1000, 8
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        keys = torch.arange(n, device="cuda", dtype=torch.int32) % K
        deltas = torch.ones(n, D, device="cuda")
        pm = A.ParameterManager(K, D, 1)
        push = pm.push_noalloc if noalloc else pm.push
        push(0, keys, deltas)
        pm.wait()
        once = pm.read_main(np.arange(K))
        pm.debug_fail_next_barrier()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            push(0, keys, deltas)
        g.replay()
        pm.wait()
        assert np.array_equal(pm.read_main(np.arange(K)), 2 * once)
        push(0, keys, deltas)
        assert np.array_equal(pm.read_main(np.arange(K)), 2 * once)
        with pytest.raises(A.AdaPMError) as e:
            pm.wait()
        assert e.value.status == A.ETIMEOUT
        del g
        pm.close()
