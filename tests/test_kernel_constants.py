"""Host-side checks of numeric facts the kernels rely on (no GPU needed)."""
import os
import re

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_collision_threshold_is_exact():
    """The spread kernels test |p_i - p_j| < 0.3 on the squared distance: with
    the correctly rounded fp32 square root, fl(sqrt(s)) < 0.3f  <=>  s < T.
    T must be the smallest fp32 value whose rounded root reaches 0.3f."""
    src = open(os.path.join(ROOT, "paper_2106_07551_gb300", "csrc", "spread_env.cuh")).read()
    lit = re.search(r"kCollideSq\s*=\s*(0x[0-9a-fA-Fp.+-]+)f;", src).group(1)
    T = np.float32(float.fromhex(lit))
    c = np.float32(0.3)
    assert np.sqrt(T) >= c
    assert np.sqrt(np.nextafter(T, np.float32(0))) < c
    bits = int(np.float32(T).view(np.uint32))
    s = np.arange(bits - 1_000_000, bits + 1_000_000, dtype=np.int64).astype(np.uint32).view(np.float32)
    np.testing.assert_array_equal(np.sqrt(s) < c, s < T)


def test_min_of_rounded_roots_is_root_of_min():
    """fl(sqrt(.)) is monotone, so min_a fl(sqrt(x_a)) == fl(sqrt(min_a x_a))
    (the kernels take one root per landmark)."""
    rng = np.random.default_rng(0)
    x = (rng.random((200_000, 8)) * 8).astype(np.float32)
    np.testing.assert_array_equal(np.sqrt(x).min(axis=1), np.sqrt(x.min(axis=1)))


def test_remote_shared_memory_waits_for_its_cta():
    """A CTA's shared memory may be accessed by its cluster's other CTAs only once it
    runs: every kernel that stores to or loads from a peer arrives at and waits for a
    cluster barrier first. The barriers follow code in which lanes diverge, so none
    is the .aligned form."""
    csrc = os.path.join(ROOT, "paper_2106_07551_gb300", "csrc")
    kernels = 0
    for name in sorted(os.listdir(csrc)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        assert not re.search(r"barrier\.cluster\.[a-z.]*aligned", src), name
        # one-line helpers that arrive or wait, by name
        call = {w: [f"barrier.cluster.{w}"] + [f + "()" for f in
                re.findall(r"void (\w+)\(\) \{ asm volatile\(\"barrier\.cluster\." + w, src)] for w in ("arrive", "wait")}
        for body in re.split(r"(?=__global__)", src)[1:]:
            remote = re.search(r"(?:st|ld)\.shared::cluster", body)
            if not remote:
                continue
            kernels += 1
            before = body[:remote.start()]
            arrive = min((before.find(c) for c in call["arrive"] if c in before), default=-1)
            assert arrive >= 0, f"{name}: no cluster barrier before the first remote access"
            assert any(c in before[arrive:] for c in call["wait"]), f"{name}: no wait before the first remote access"
    assert kernels == 2                  # Kuhn's clusters and the linear program's


def test_action_buffers_alternate_across_units():
    """Groups that share a unit exchange actions through two buffers with one barrier a
    step, so successive exchanges must take different buffers also where one unit (of an
    odd number of steps) ends and the next begins: the buffer comes from a variable that
    is declared before the loop over items and flipped after each exchange."""
    src = open(os.path.join(ROOT, "paper_2106_07551_gb300", "csrc", "spread_rollout.cu")).read()
    body = src[src.index("spread_rollout_x3_kernel("):]
    uses = re.findall(r"\bacts\[([^\]]*)\]\[", body)
    uses.remove("2")                                     # the declaration
    assert len(uses) == 2 and len(set(uses)) == 1
    var = uses[0]
    assert re.fullmatch(r"\w+", var), var
    items = body.index("item < plan.items")
    assert re.search(r"\b%s = 0;" % var, body[:items])
    assert re.search(r"\b%s \^= 1u;" % var, body[body.rindex("acts["):])
