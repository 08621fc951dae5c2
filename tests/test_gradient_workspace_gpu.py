"""The batch gradient's kept workspace: nothing of one call shows in the next, and the memory is given back."""
import gc
import os
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
sys.path.insert(0, os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden"))
import make_surrogate_gradient as M  # noqa: E402

MB = 1 << 20


@pytest.fixture(scope="module")
def ck():
    import torch
    from paper_1209_6038_gb300 import build, cloak
    build.build()
    cloak.load()
    torch.cuda.init()
    return cloak


def network(ck, params):
    c = ck.Cloak(ck.RADIAL)
    ck.cloak_surrogate_params(c.h, params)
    return c


def step(ck, c, stage, n, seed, lr=0.0, stream=None):
    import torch
    rng = np.random.default_rng([seed, n])
    x, t = M.batch(stage, n)
    x, t = x[rng.permutation(n)], t[rng.permutation(n)] * np.float32(1 + seed)
    x, t = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        return ck.cloak_surrogate_step(c.h, x, t, stage=stage, lr=lr).copy()


def test_calls_on_one_handle_match_fresh_handles(ck):
    """Stages, data, sizes and streams in turn; every gradient bit for bit that of a handle of its own, whose workspace
    was made for it (the last handle's end gives the kept ones back)."""
    import torch
    calls = [(1, 2560, 0, 0.0), (2, 2560, 1, 0.0), (1, 2560, 2, 0.0), (2, 2560, 3, 1e-3), (1, 2560, 4, 1e-3),
             (1, 256, 5, 0.0), (2, 384, 6, 0.0), (1, 2560, 7, 0.0), (2, 256, 8, 0.0), (1, 256, 5, 0.0)]
    params, kept, states = M.params(), [], []
    streams = [None, torch.cuda.Stream(), torch.cuda.Stream()]
    c = network(ck, params)
    for i, (stage, n, seed, lr) in enumerate(calls):
        states.append(ck.cloak_surrogate_params(c.h).copy())
        kept.append(step(ck, c, stage, n, seed, lr, streams[i % 3]))
    c.close()
    for (stage, n, seed, _), g, p in zip(calls, kept, states):
        gc.collect()
        c = network(ck, p)
        fresh = step(ck, c, stage, n, seed)
        c.close()
        if stage == 2:  # only the output layer's gradient is formed where the step also updates
            assert np.array_equal(g[-1285:], fresh[-1285:])
        else:
            assert np.array_equal(g, fresh)
    assert not np.array_equal(states[3], states[5])


def free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("by", ["training", "the last handle"])
def test_kept_memory_is_given_back(ck, by):
    """A batch of 65536 rows keeps some 450 MB; 64 MB stand for what the driver holds back for its own use."""
    import torch
    gc.collect()
    c, other = network(ck, M.params()), network(ck, M.params())
    step(ck, c, 1, 256, 0)
    torch.cuda.empty_cache()
    before = free(torch)
    step(ck, c, 1, 65536, 0)
    torch.cuda.empty_cache()
    assert before - free(torch) > 300 * MB  # kept for the next batch of this size
    if by == "training":
        ck.cloak_surrogate_train(other.h, 19456, 0, 1)
        torch.cuda.empty_cache()
        assert before - free(torch) < 64 * MB
    c.close()
    other.close()
    assert before - free(torch) < 64 * MB


def test_kept_memory_is_bounded(ck):
    """Several sizes and networks: 1 GiB at most stays, a workspace above that is not kept."""
    import torch
    gc.collect()
    cs = [network(ck, M.params()) for _ in range(3)]
    step(ck, cs[0], 1, 256, 0)
    torch.cuda.empty_cache()
    before = free(torch)
    for c, n in zip(cs, (65536, 65536 + 128, 65536 + 256)):
        step(ck, c, 1, n, 0)
    step(ck, cs[0], 1, 196608, 0)
    torch.cuda.empty_cache()
    assert before - free(torch) < 1024 * MB + 64 * MB
    for c in cs:
        c.close()


def test_threads_with_handles_of_their_own(ck):
    """Four threads, each with its handle and stream, take and hand back workspaces of the same sizes at once."""
    import threading
    import torch
    plan = [(1, 2560, 0), (1, 256, 1), (2, 2560, 2), (1, 2560, 3), (1, 256, 4), (1, 2560, 5)]
    ref = []
    for stage, n, seed in plan:
        c = network(ck, M.params())
        ref.append(step(ck, c, stage, n, seed))
        c.close()
    wrong = []

    def work(k):
        c, s = network(ck, M.params()), torch.cuda.Stream()
        for i in [(j + k) % len(plan) for j in range(3 * len(plan))]:
            stage, n, seed = plan[i]
            if not np.array_equal(step(ck, c, stage, n, seed, 0.0, s), ref[i]):
                wrong.append((k, i))
        c.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
