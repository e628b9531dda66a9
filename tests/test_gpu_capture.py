"""Calls recorded in a CUDA graph: every launch of the graph does what the same eager calls do, bit for bit, on the
state it finds; calls that a launch cannot repeat are refused; a graph that is never launched leaves no trace."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _state(pm, K, W):
    k = np.arange(K)
    return [pm.read_main(k)] + [x for w in range(W) for x in pm.replica_rows(w, k)]


def _same(a, b, K, W, what):
    for i, (x, y) in enumerate(zip(_state(a, K, W), _state(b, K, W))):
        assert np.array_equal(x, y), f"{what}: array {i}"


# one block's sort, and on either side of its limit; several sub-tiles and spans
@pytest.mark.parametrize("n", [1000, 8192, 8193, 60_000])
@pytest.mark.parametrize("noalloc,relocate,refresh", [(False, False, False), (True, False, True), (False, True, False)])
def test_graph_launches_repeat_pull_push_sync(gpu_lib, n, noalloc, relocate, refresh):
    K, D, W = 5000, 12, 2
    rng = np.random.default_rng(n)
    init = torch.from_numpy(rng.normal(0, 0.1, size=(K, D)).astype(np.float32)).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        keys = torch.randint(0, K, (n,), device="cuda", dtype=torch.int32)
        deltas = torch.randn(n, D, device="cuda")
        outs = [torch.empty(n, D, device="cuda") for _ in range(2)]
        pair = [gpu_lib.ParameterManager(K, D, W, init_values=init, relocate=relocate, delta_refresh=refresh)
                for _ in range(2)]
        for pm in pair:
            pm.intent(0, keys, 0, 9)                                   # with a push plan of the same keys
            pm.intent(1, torch.arange(0, K, 3, device="cuda"), 0, 9)
            pm.intent(0, keys, 1, 3)                                   # early events are due

        def calls(pm, out):
            pm.pull(0, keys, out=out)
            (pm.push_noalloc if noalloc else pm.push)(0, keys, deltas)
            pm.pull(1, keys, out=out)
            pm.sync()

        for pm, out in zip(pair, outs):
            calls(pm, out)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            calls(pair[0], outs[0])
        for launch in range(3):
            g.replay()
            calls(pair[1], outs[1])
            for pm in pair:
                pm.wait()
            assert torch.equal(outs[0], outs[1]), f"launch {launch}: pulled rows"
            _same(pair[0], pair[1], K, W, f"launch {launch}")
            for pm in pair:                                            # eager work between the launches
                pm.push(1, keys, deltas)
            keys.copy_(torch.randint(0, K, (n,), device="cuda", dtype=torch.int32))
            deltas.mul_(0.5)
        for pm in pair:
            pm.advance_clock(0)
            pm.wait()
        _same(pair[0], pair[1], K, W, "after an advance")
        del g
        for pm in pair:
            pm.close()


@pytest.mark.parametrize("kind,n", [("mf", 300), ("mf", 6000), ("complex", 900), ("sgns", 400)])
def test_graph_launches_repeat_training_steps(gpu_lib, kind, n):
    K, dim, W, k = 2000, 16, 2, 10
    D = dim if kind == "sgns" else 2 * dim
    init = torch.rand(K, D, device="cuda").add_(0.1)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b, c = (torch.randint(0, K // 2, (n,), device="cuda", dtype=torch.int32) for _ in range(3))
        ng = torch.randint(0, K // 2, (n * 2 * k,), device="cuda", dtype=torch.int32)
        v = torch.randn(n, device="cuda")
        pair = [gpu_lib.ParameterManager(K, D, W, init_values=init) for _ in range(2)]
        loss = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2)]

        def step(i):
            if kind == "mf":
                pair[i].mf_step(0, a, b, v, dim, True, 0.05, loss_out=loss[i])
            elif kind == "complex":
                pair[i].complex_step(0, a, b, c, ng[:n * k], k, dim, 0.05, loss_out=loss[i])
            else:
                pair[i].sgns_step(0, a, torch_ctx, ng, 2, k, K // 2, dim, 0.05, loss_out=loss[i])

        torch_ctx = torch.stack([b, c], 1).reshape(-1)
        for i in range(2):
            pair[i].intent(0, torch.cat([a, b]), 0, 5)
            step(i)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            step(0)
        for launch in range(2):
            g.replay()
            step(1)
            for pm in pair:
                pm.wait()
            assert loss[0].item() == loss[1].item() and loss[0].item() != 0.0
            _same(pair[0], pair[1], K, W, f"launch {launch}")
        del g
        for pm in pair:
            pm.close()


def test_calls_that_move_clocks_and_intents_are_refused(gpu_lib):
    A, K, D = gpu_lib, 3000, 8
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        keys = torch.randint(0, K, (20_000,), device="cuda", dtype=torch.int32)
        deltas = torch.ones(20_000, D, device="cuda")
        pm = A.ParameterManager(K, D, 2)
        timed = A.ParameterManager(K, D, 1, action_timing="adaptive")
        pm.intent(0, keys[:100], 1, 2)
        pm.push(0, keys, deltas)
        pm.wait()
        before = pm.read_main(np.arange(K))
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for call in (lambda: pm.intent(0, keys, 1, 3), lambda: pm.intent(1, keys[:5], 0, 3),
                         lambda: pm.advance_clock(0), lambda: timed.sync()):
                with pytest.raises(A.AdaPMError) as e:
                    call()
                assert e.value.status == A.EINVAL and "graph" in str(e.value)
            pm.push(0, keys, deltas)
        del g                                                          # recorded, never launched
        assert pm.clock(0) == 0 and np.array_equal(pm.read_main(np.arange(K)), before)
        pm.push(0, keys, deltas)                                       # grid barriers still count from where they were
        pm.wait()
        assert np.array_equal(pm.read_main(np.arange(K)), 2 * before)
        pm.advance_clock(0)
        pm.wait()
        assert pm.clock(0) == 1 and np.array_equal(pm.replica_keys(0), np.unique(keys[:100].cpu().numpy()))
        pm.close()
        timed.close()


def test_pinned_host_inputs_are_read_at_each_launch(gpu_lib):
    K, D, n = 500, 8, 700
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        keys = torch.randint(0, K, (n,), dtype=torch.int32).pin_memory()
        deltas = torch.ones(n, D).pin_memory()
        pm = gpu_lib.ParameterManager(K, D, 1)
        pm.push(0, keys, deltas)
        pm.wait()
        want = np.bincount(keys.numpy(), minlength=K).astype(np.float32)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            pm.push(0, keys, deltas)
        for launch in range(2):
            keys.copy_(torch.randint(0, K, (n,), dtype=torch.int32))
            deltas.fill_(2.0 + launch)
            g.replay()
            pm.wait()
            want += (2.0 + launch) * np.bincount(keys.numpy(), minlength=K)
            assert np.array_equal(pm.read_main(np.arange(K)), np.repeat(want[:, None], D, axis=1))
        del g
        pm.close()
