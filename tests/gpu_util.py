"""Helpers shared by the GPU parity tests (no method arithmetic here)."""
import numpy as np
import pytest

import workloads


def need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def context():
    torch = need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_07551_gb300 import Context
    return Context(0, torch.cuda.current_stream(0))


def spec_of(w: workloads.Workload, flags: int = 0, n_envs: int | None = None, local_ratio=None):
    from paper_2106_07551_gb300 import make_spec
    return make_spec(w.env_kind, w.n_agents, w.obs_dim, w.n_actions, w.n_landmarks,
                     w.episode_len, w.n_envs if n_envs is None else n_envs, flags, local_ratio)


def load_population(ctx, w: workloads.Workload):
    from paper_2106_07551_gb300 import policy_desc
    descs = [policy_desc(p.kind, p.dtype, p.seat, p.dims, p.params) for p in w.policies]
    ids = ctx.pop_load(spec_of(w), descs)
    assert list(ids) == list(range(len(w.policies)))
    return ids


def logits_close(gpu, ref, rtol):
    """|g - o| <= rtol * max(|o|, rms(o over the row)) for every entry."""
    gpu = np.asarray(gpu, np.float64)
    ref = np.asarray(ref, np.float64)
    rms = np.sqrt(np.mean(ref ** 2, axis=-1, keepdims=True))
    scale = np.maximum(np.abs(ref), rms)
    bad = np.abs(gpu - ref) > rtol * scale + 1e-30
    return int(bad.sum()), float((np.abs(gpu - ref) / np.maximum(scale, 1e-30)).max(initial=0.0))


def plant_odd_weights(policies):
    """Infinities, a NaN and finite weights that round to a bf16 infinity, one kind per
    policy (the eighth of each eight stays as it is)."""
    for n, p in enumerate(policies):
        i, h1, h2, o = p.dims
        w1, b1, w2, b2, w3, _ = np.split(p.params, np.cumsum([h1 * i, h1, h2 * h1, h2, o * h2]))   # views
        huge = np.float32(3.4e38)           # bf16 rounds from 3.3962e38 up to infinity
        for a, at, v in [[(w1, 3 * i, np.inf)], [(w2, 5 * h1 + 9, -np.inf), (w2, 6 * h1 + 2, np.inf)],
                         [(w1, 7 * i + 2, np.nan)], [(w1, 2 * i, huge)], [(b1, 11, np.inf)], [(w3, h2 + 4, np.inf)],
                         [(b2, 3, huge)], []][n % 8]:
            a[at] = v


def logits_same_class(gpu, ref, params, dims, x):
    """Logits of one policy on the rows x: the same entries are NaN, +inf and -inf, and
    the finite ones agree to the rounding of an fp32 forward in any order, (in + h1 + h2
    + 3) 2^-24 of the same forward in absolute values (a ReLU enlarges no difference; a
    finite entry has its non-finite weights behind closed ReLUs: zero there)."""
    gpu, ref = np.asarray(gpu, np.float64), np.asarray(ref, np.float64)
    np.testing.assert_array_equal(np.isnan(gpu), np.isnan(ref))
    np.testing.assert_array_equal(np.where(np.isinf(gpu), gpu, 0), np.where(np.isinf(ref), ref, 0))
    i, h1, h2, o = dims
    p = np.abs(np.where(np.isfinite(params), params, 0).astype(np.float64))
    w1, b1, w2, b2, w3, b3 = np.split(p, np.cumsum([h1 * i, h1, h2 * h1, h2, o * h2]))
    size = np.abs(np.asarray(x, np.float64)) @ w1.reshape(h1, i).T + b1
    size = (size @ w2.reshape(h2, h1).T + b2) @ w3.reshape(o, h2).T + b3
    ok = np.isfinite(ref)
    assert np.all(np.abs(gpu[ok] - ref[ok]) <= (i + h1 + h2 + 3) * 2.0 ** -24 * size[ok])


def four_se_rule(mean, se, exact):
    """At most 3 entries beyond 4 standard errors and none beyond 5."""
    z = np.abs(np.asarray(mean) - np.asarray(exact)) / np.maximum(np.asarray(se), 1e-12)
    return int((z > 4).sum()), float(z.max(initial=0.0))
