"""The element and node kernels' three-lane and one-thread forms: a batch below both lines,
one above the triangle line (8000) and one above the node line (20000) give a cloth the
same bits in two steps and in their gradients (the batches' largest cloth is the same: an
instance's Krylov sums are split by it), the states are those of the cloth alone, and the
step is the oracle's (STATE_TOL, the repository's per-step bound).  Curved rest shapes take
the bending projection, "mass" its velocity part, 2 x 2 and 3 x 3 cloths partly filled
warps."""
import dataclasses

import numpy as np
import pytest

import scenes
from tests._helpers import STATE_TOL, cuda, make_batch, make_cloth, oracle_model, rel_inf

pytestmark = pytest.mark.gpu


def _scene(n, curved):
    sc = scenes.small_scene(n, seed=n, contact="both", drop=True, n_steps=2)
    if curved:
        rest = sc.rest_pos.copy()
        rest[:, 2] += 0.3 * rest[:, 0] ** 2 - 0.2 * rest[:, 0] * rest[:, 1]
        sc = dataclasses.replace(sc, rest_pos=rest)
    return dataclasses.replace(sc, params=dataclasses.replace(sc.params, k_stretch=0.01, k_bend=1e-8))


@pytest.mark.parametrize("n", [2, 3, 11])
@pytest.mark.parametrize("curved,mode", [(False, "rowsum"), (True, "rowsum"), (True, "mass")])
def test_forms_agree(n, curved, mode):
    import torch
    from oracle import cloth as oc
    sc = _scene(n, curved)
    rng = np.random.default_rng(n)
    w = rng.standard_normal((sc.m, 3))
    cl = make_cloth(sc, contact_compliance=mode, global_solver=1)
    want = cl.rollout(cuda(sc.x0), cuda(sc.v0), 2, traj=True)
    x1 = oc.rollout(oracle_model(sc, contact_compliance=mode), sc.x0, sc.v0, 1)[0][1]
    assert rel_inf(want[2][1].cpu().numpy(), x1) <= STATE_TOL
    cl.close()
    pad = dataclasses.replace(scenes.draped_cloth(n=60, seed=1, n_steps=2), obstacles=sc.obstacles, params=sc.params)
    grads = []
    for n_pads in (1, 2, 6):             # 6962 triangles, 3600 nodes a pad
        b = make_batch([sc] + [pad] * n_pads + [sc], contact_compliance=mode, global_solver=1)
        cat = lambda a, p: cuda(np.concatenate([a] + [p] * n_pads + [a]))
        got = b.rollout(cat(sc.x0, pad.x0), cat(sc.v0, pad.v0), 2)
        for g, r in zip(got, want[:2]):
            assert torch.equal(b.split(g)[0], r) and torch.equal(b.split(g)[-1], r)
        if mode != "mass":
            dx0, dv0, dth = b.backward(cat(w, pad.loss_w), cat(w, 0 * pad.x0))
            grads.append([b.split(dx0)[-1], b.split(dv0)[-1], dth[-1]])
        b.close()
    for g in grads[1:]:
        assert all(torch.equal(p, q) for p, q in zip(g, grads[0]))
