"""Training steps at the edges of their batches of 32 rows, ring depths and row widths, per element against the
oracle (the checks and derived bounds of test_gpu_steps), and on replicas that have a push pending."""
import numpy as np
import pytest
import torch

from oracle import ParameterManagerOracle, steps
from tests import test_gpu_steps as base
from tests.test_gpu_store import dev

pytestmark = pytest.mark.gpu


# rows per centre: 2 x window x (1 + negatives)
@pytest.mark.parametrize("dim,window,negatives,batch", [
    (4, 1, 0, 6000), (64, 1, 7, 30), (128, 1, 15, 20), (132, 1, 16, 20), (256, 2, 7, 12), (260, 1, 31, 10),
    (384, 1, 32, 8), (388, 2, 3, 10), (1024, 1, 24, 6)])
def test_sgns_batch_edges(gpu_lib, dim, window, negatives, batch):
    base.test_sgns_one_step_per_element(gpu_lib, dim, window, negatives, batch)


@pytest.mark.parametrize("half_dim,negatives,batch", [
    (4, 1, 20), (4, 3, 6000), (12, 15, 30), (16, 30, 30), (64, 31, 20), (128, 32, 16), (132, 63, 10), (256, 64, 8)])
def test_complex_batch_edges(gpu_lib, half_dim, negatives, batch):
    base.test_complex_one_step_per_element(gpu_lib, half_dim, negatives, batch)


@pytest.mark.parametrize("kind", ["mf", "complex", "sgns"])
def test_step_on_replicas_with_a_pending_push(gpu_lib, kind):
    rng = np.random.default_rng(3)
    K, n, k = 60, 25, 9
    dim = {"mf": 12, "complex": 16, "sgns": 20}[kind]
    D = dim if kind == "sgns" else 2 * dim
    init = (rng.normal(0, 0.2, size=(K, D))).astype(np.float32)
    if D > dim:
        init[:, dim:] = np.abs(init[:, dim:]) + 0.1
    pm = gpu_lib.ParameterManager(K, D, 2, init_values=torch.from_numpy(init).cuda())
    ref = ParameterManagerOracle(K, D, 2, init)
    every = np.arange(K)
    for api, conv in ((pm, dev), (ref, np.asarray)):
        for w in range(2):
            api.intent(w, conv(every), 0, 2)
    for w, keys in ((0, every[::2]), (1, every[::3]), (0, every[::5])):   # some of them twice
        d = np.abs(rng.normal(0, 0.05, size=(keys.size, D))).astype(np.float32)
        pm.push(w, dev(keys), torch.from_numpy(d).cuda())
        ref.push(w, keys, d)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    a, b, c = (rng.integers(0, K // 2, size=n) for _ in range(3))
    ng = rng.integers(0, K // 2, size=(n, k))
    for w in range(2):
        if kind == "mf":
            v = rng.normal(size=n).astype(np.float32)
            pm.mf_step(w, dev(a), dev(b), torch.from_numpy(v).cuda(), dim, True, 0.05, loss_out=loss)
            want = steps.mf_step(ref, w, a, b, v, dim, 0.05, True)
        elif kind == "complex":
            pm.complex_step(w, dev(a), dev(b), dev(c), dev(ng.reshape(-1)), k, dim, 0.05, loss_out=loss)
            want = steps.complex_step(ref, w, a, b, c, ng, dim, 0.05)
        else:
            pm.sgns_step(w, dev(a), dev(np.stack([b, c], 1).reshape(-1)), dev(np.stack([ng, ng], 1).reshape(-1)), 2,
                         k, K // 2, dim, 0.05, loss_out=loss)
            want = steps.sgns_step(ref, w, a, np.stack([b, c], 1), np.stack([ng, ng], 1), K // 2, 0.05)
        pm.wait()
        assert abs(float(loss.item()) - want) <= 1e-4 * abs(want)
    pm.sync()
    ref.sync()
    # up to ~100 updates of at most lr = 0.05 per element, each within a few 2^-24 of itself and of its sums
    assert np.max(np.abs(pm.read_main(every) - ref.main)) <= 100 * 16 * 2.0 ** -24
    pm.close()
