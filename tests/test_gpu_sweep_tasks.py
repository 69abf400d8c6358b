"""The global solve through the tree-scheduled sweeps at the sizes where their tasks
change: cloths whose fronts are all small, with a few row-split fronts, with long row sums
(K > 128), and a batch with enough small fronts for the
grouped kernel; against the oracle's banded Cholesky, and every instance of the batch
bitwise the cloth alone.

Tolerance: the two factorisations differ by about cond(P) eps; 2e-11 as for the GPU
factor of P."""
import numpy as np
import pytest

import scenes
from tests._helpers import cuda, make_batch, make_cloth, oracle_model, rel_inf

pytestmark = pytest.mark.gpu


def _want(sc, rhs):
    M = oracle_model(sc)
    out = np.zeros_like(rhs)
    out[M.free] = M.solve_P(rhs[M.free])
    return out


@pytest.mark.parametrize("n", [3, 8, 17, 33, 66, 90])
@pytest.mark.parametrize("factor_on_gpu", [0, 1])
def test_one_cloth(n, factor_on_gpu):
    sc = scenes.draped_cloth(n=n, seed=n, n_steps=1)
    rhs = np.random.default_rng(n).standard_normal((sc.m, 3))
    cl = make_cloth(sc, global_solver=1, factor_on_gpu=factor_on_gpu)
    got = cl.global_solve(cuda(rhs)).cpu().numpy()
    cl.stats()                      # raises if a dependency wait gave up
    cl.close()
    assert rel_inf(got, _want(sc, rhs)) < 2e-11


def test_grouped_batch_is_bitwise_the_cloths_alone():
    import torch
    scs = [scenes.batch_instance(s, n_steps=1) for s in range(24)]
    rhs = [np.random.default_rng(s).standard_normal((sc.m, 3)) for s, sc in enumerate(scs)]
    b = make_batch(scs, global_solver=1)
    got = b.split(b.global_solve(cuda(np.concatenate(rhs))))
    x = b.rollout(cuda(np.concatenate([sc.x0 for sc in scs])), cuda(np.concatenate([sc.v0 for sc in scs])), 1)[0]
    x = b.split(x)
    b.stats()
    for i in (0, 7, 15, 23):
        cl = make_cloth(scs[i], global_solver=1)
        assert torch.equal(cl.global_solve(cuda(rhs[i])), got[i])
        assert torch.equal(cl.rollout(cuda(scs[i].x0), cuda(scs[i].v0), 1)[0], x[i])
        cl.close()
    b.close()
    assert rel_inf(got[0].cpu().numpy(), _want(scs[0], rhs[0])) < 2e-11


def test_many_small_fronts_are_bitwise_the_cloths_alone():
    """Above 32 small fronts per SM: groups of four on CTAs of 128 threads."""
    import torch
    base = [scenes.batch_instance(s, n_steps=1) for s in range(12)]
    scs = base * 12
    rhs = [np.random.default_rng(s).standard_normal((sc.m, 3)) for s, sc in enumerate(base)]
    b = make_batch(scs, global_solver=1)
    got = b.split(b.global_solve(cuda(np.concatenate(rhs * 12))))
    x = b.rollout(cuda(np.concatenate([sc.x0 for sc in scs])), cuda(np.concatenate([sc.v0 for sc in scs])), 1)[0]
    x = b.split(x)
    b.stats()
    for i, sc in enumerate(base):
        cl = make_cloth(sc, global_solver=1)
        want = cl.global_solve(cuda(rhs[i]))
        wx = cl.rollout(cuda(sc.x0), cuda(sc.v0), 1)[0]
        cl.close()
        for k in (0, 5, 11):
            assert torch.equal(got[12 * k + i], want) and torch.equal(x[12 * k + i], wx)
    b.close()
