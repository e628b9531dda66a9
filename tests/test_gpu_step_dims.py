"""Row widths that the training steps cannot split into float4 parts are refused before anything runs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,dim,ok", [
    ("mf", 2, False), ("mf", 6, False), ("mf", 10, False), ("mf", 4, True), ("mf", 12, True),
    ("complex", 4, False), ("complex", 6, False), ("complex", 12, False), ("complex", 8, True), ("complex", 24, True)])
def test_adagrad_rows_split_into_vectors(gpu_lib, kind, dim, ok):
    K, n = 40, 5
    init = np.random.default_rng(dim).uniform(0.1, 0.5, size=(K, 2 * dim)).astype(np.float32)
    pm = gpu_lib.ParameterManager(K, 2 * dim, 1, init_values=torch.from_numpy(init).cuda())
    a, b, c, ng = (torch.arange(i * n, (i + 1) * n, device="cuda", dtype=torch.int32) for i in range(4))

    def step():
        if kind == "mf":
            pm.mf_step(0, a, b, torch.ones(n, device="cuda"), dim, True, 0.05)
        else:
            pm.complex_step(0, a, b, c, ng, 1, dim, 0.05)

    if ok:
        step()
    else:
        with pytest.raises(gpu_lib.AdaPMError) as e:
            step()
        assert e.value.status == gpu_lib.EINVAL and "multiple" in str(e.value)
    pm.wait()
    changed = (pm.read_main(np.arange(K)) != init).any(axis=1)
    used = 2 * n if kind == "mf" else 4 * n
    assert changed[:used].all() == ok and not changed[used:].any() and (ok or not changed.any())
    pm.close()


def test_plain_sgd_takes_every_row_width(gpu_lib):
    pm = gpu_lib.ParameterManager(10, 12, 1, init_values=torch.full((10, 12), 0.5, device="cuda"))
    k = torch.zeros(1, device="cuda", dtype=torch.int32)
    pm.mf_step(0, k, k + 1, torch.ones(1, device="cuda"), 12, False, 0.05)
    pm.wait()
    assert (pm.read_main([0, 1]) != 0.5).all() and (pm.read_main([2]) == 0.5).all()   # 1 - 12 x 0.25 is not 0
    pm.close()
