"""The assembly of the adjoint's fronts for flat rest shapes (bending adds w I) and curved
ones (the projection's derivative too), with fewer and more pairs than a sorting window
(2048): the Krylov solve takes exactly the iterations it took with the assembly that formed
every term in list order (the preconditioner is the same bits), and the gradients are the
oracle's to GRAD_TOL."""
import dataclasses

import numpy as np
import pytest

import scenes
from oracle import cloth as oc
from tests._helpers import GRAD_TOL, cuda, make_cloth, oracle_model, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,curved,iters", [(2, False, 6), (2, True, 6), (3, False, 7), (3, True, 7),
                                            (11, False, 18), (11, True, 19), (20, False, 27), (20, True, 27)])
def test_assembly(n, curved, iters):
    sc = scenes.small_scene(n, seed=n, contact="both", drop=True, n_steps=2)
    if curved:
        rest = sc.rest_pos.copy()
        rest[:, 2] += 0.3 * rest[:, 0] ** 2 - 0.2 * rest[:, 0] * rest[:, 1]
        sc = dataclasses.replace(sc, rest_pos=rest)
    cl = make_cloth(sc)
    M = oracle_model(sc)
    _, _, recs = oc.rollout(M, sc.x0, sc.v0, 2)
    gv = 0.3 * np.random.default_rng(n).standard_normal((sc.m, 3))
    want = oc.rollout_gradient(M, recs, sc.loss_w, gv, None)
    cl.rollout(cuda(sc.x0), cuda(sc.v0), 2)
    got = cl.backward(cuda(sc.loss_w), cuda(gv))
    st = cl.stats()
    cl.close()
    assert rel_l2(got[0].cpu().numpy(), want[0]) <= GRAD_TOL
    assert st["adj_iters"] == iters and st["adj_fallbacks"] == 0
