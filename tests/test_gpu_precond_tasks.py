"""The adjoint's preconditioner solves with their factor entries loaded ahead of the waits
(contexts of few tasks) and without (many), for fronts that are one task and fronts split
by rows: the gradients are bitwise those of one launch per tree level."""
import numpy as np
import pytest

import scenes
from tests._helpers import cuda, make_batch, make_cloth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 8, 17, 33, 61, 120])
def test_tree_tasks_are_bitwise_the_levels(n, monkeypatch):
    import torch
    sc = scenes.draped_cloth(n=n, seed=n, n_steps=1)
    gv = 0.3 * np.random.default_rng(n).standard_normal((sc.m, 3))
    grads = []
    for level in (False, True):
        if level:
            monkeypatch.setenv("DC_LEVEL_SOLVES", "1")
        cl = make_cloth(sc, global_solver=1)
        cl.rollout(cuda(sc.x0), cuda(sc.v0), 1)
        grads.append(cl.backward(cuda(sc.loss_w), cuda(gv)))
        cl.stats()                   # raises if a dependency wait gave up
        cl.close()
    for a, b in zip(*grads):
        assert torch.equal(a, b) and torch.isfinite(a).all()


def test_many_fronts_are_bitwise_the_levels(monkeypatch):
    import torch
    base = [scenes.batch_instance(s, n_steps=1) for s in range(12)]
    scs = base * 10
    cat = lambda name: cuda(np.concatenate([getattr(sc, name) for sc in scs]))
    grads = []
    for level in (False, True):
        if level:
            monkeypatch.setenv("DC_LEVEL_SOLVES", "1")
        b = make_batch(scs, global_solver=1)
        b.rollout(cat("x0"), cat("v0"), 1)
        grads.append(b.backward(cat("loss_w"), allow_nonconverged=True))
        b.stats()
        b.close()
    for a, c in zip(*grads):
        assert torch.equal(a, c)
