"""Contexts on streams of their own share the GPU: three cloths' rollouts replayed as graphs, none
of which fills the chip, take together less than three in turn would (as every launch takes only
the CTAs its tree has tasks for), and give each cloth's own bits.  A context that takes every
SM for its waiting CTAs makes the three nearly as slow as in turn (0.88 of it on 45 x 45
nodes; with the CTAs a tree has use for it is 0.35)."""
import time

import pytest

import scenes
from tests._helpers import cuda, make_cloth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [45, 61])
def test_three_rollouts_at_once(n):
    import torch
    scs = [scenes.draped_cloth(n=n, seed=s, n_steps=2) for s in range(3)]
    jobs = []
    for sc in scs:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            cl = make_cloth(sc, global_solver=1)
            cl.set_graphs(True)
            jobs.append((stream, cl, cuda(sc.x0), cuda(sc.v0)))

    def run(which):
        out = []
        for stream, cl, x0, v0 in which:
            with torch.cuda.stream(stream):
                out.append(cl.rollout(x0, v0, 2))
        return out

    def seconds(which):
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(3):
                run(which)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / 3)
        return best

    alone = []
    for j in jobs:
        alone += run([j])
        torch.cuda.synchronize()
    alone = [[t.clone() for t in r] for r in alone]
    one = [seconds([j]) for j in jobs]
    three = seconds(jobs)
    together = run(jobs)
    torch.cuda.synchronize()
    for a, b in zip(alone, together):
        assert all(torch.equal(p, q) for p, q in zip(a, b))
    for _, cl, _, _ in jobs:
        cl.close()
    assert three < 0.6 * sum(one), (three, one)
