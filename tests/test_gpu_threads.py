"""Two host threads, each with a context and a stream of its own, calling the same
entry points with sizes that need different amounts of shared memory: every call
launches and gives the result of a single thread."""
import threading

import numpy as np
import pytest

import workloads
from gpu_util import context, load_population, need_gpu, spec_of

pytestmark = pytest.mark.gpu


def rollout_calls(ctx, big):
    from paper_2106_07551_gb300 import alloc_traj
    import torch
    # as many combinations as SMs, two or three units each: two or three groups a CTA
    w = workloads.spread(n_agents=3, n_envs=152 * 128, pop=4, envs_per_pair=128, episode_len=1, seed=1)
    load_population(ctx, w)
    spec, n_eps = spec_of(w), 3 if big else 2
    traj = alloc_traj(spec, n_eps)
    pairs = torch.from_numpy(w.pair_ids).cuda()

    def call():
        ctx.rollout(spec, pairs, n_eps, 5, traj)
        return traj["reward"]
    return call


def solver_calls(ctx, big, lp):
    import torch
    m = 30 if big else 3
    P = torch.from_numpy(np.random.default_rng(m).normal(size=(1, m, m))).cuda()
    x, y = (torch.zeros((1, m), dtype=torch.float64, device="cuda") for _ in range(2))
    b = torch.zeros((1, 2), dtype=torch.float64, device="cuda")

    def call():
        if lp:
            ctx.meta_lp_nash(P, x, y, b)
        else:
            ctx.meta_fictitious_play(P, 20, x, y, b)
        return x
    return call


def exploit_calls(ctx, big):
    w = workloads.leduc(pop=1, seed=3)
    dims = (17, 128 if big else 70, 128, 3)
    for p in w.policies:
        p.dims, p.params = dims, workloads.random_mlp(np.random.default_rng(p.seat), dims)
    load_population(ctx, w)
    return lambda: np.array(ctx.exploitability([0], [1.0], [1], [1.0]))


CALLS = {"rollout": rollout_calls, "fictitious_play": lambda c, b: solver_calls(c, b, False),
         "lp": lambda c, b: solver_calls(c, b, True), "exploitability": exploit_calls}


@pytest.mark.parametrize("kind", list(CALLS))
def test_threads_with_different_sizes(kind):
    torch = need_gpu()
    context().close()
    from paper_2106_07551_gb300 import Context
    start, errors, results = threading.Barrier(2), [], [None, None]

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream), Context(0, stream) as ctx:
                call = CALLS[kind](ctx, i == 1)
                torch.cuda.synchronize()
                first = call()
                ctx.sync()
                first = first.clone() if torch.is_tensor(first) else first
                start.wait(60)
                for _ in range(3000):
                    out = call()
                ctx.sync()
                results[i] = bool((out == first).all())
        except Exception as e:                           # noqa: BLE001 (reported by the main thread)
            errors.append(e)
            start.abort()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert results == [True, True]
