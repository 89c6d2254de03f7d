"""The step kernel's variants agree: a uniform batch in its compile-time (or small-block) variant,
the same environments in the variant of large blocks, and the same behind a lone drone in an uneven
batch, where they start at odd places of their tile and the downwash reads its sources in single
loads. Heights are spread, so that no wake is near-singular. The variants sum the wakes in other
orders; each sum rounds by about N 2^-24 of the largest wakes, far below the substep tolerance of the
oracle comparison that the first variant is held to as well."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_08039_gb300 as mdg
from paper_2606_08039_gb300 import workloads as wl
from helpers import assert_horizon_close, oracle_arrays, oracle_step, spread_heights, tolerance_response

pytestmark = pytest.mark.gpu
P = oracle.cf2x()


def _run(cuda, dpe, sw, rk4, rollout, block=None):
    c = mdg.Constants.cf2x()
    c.integrator = mdg.INTEGRATOR_RK4 if rk4 else mdg.INTEGRATOR_EULER
    h = mdg.Handle(dpe, np.full(len(dpe), 7, np.uint32), c)
    if block:
        h.set_block_size(block)
    state = mdg.pack_state(*sw, device=cuda)
    act = torch.as_tensor(wl.waypoints(301, h.n), device=cuda)
    kin, idx, rel = h.new_obs(cuda)
    if rollout:
        h.rollout(state, act, mdg.ACT_PID, 2, 1, mdg.OBS_LAST, kin, idx, rel)
    else:
        h.step_obs(state, act, mdg.ACT_PID, 2, kin, idx, rel)
    assert h.status()[0] == mdg.OK
    return state, kin, idx, rel, act


@pytest.mark.parametrize("rk4", [False, True])
@pytest.mark.parametrize("drones", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 16, 17, 32, 33, 64, 65])
def test_variants_agree(cuda, drones, rk4):
    envs = 1 + 130 // drones
    swarm = spread_heights(wl.full_aero(302, n_envs=envs, drones=drones), dz=0.3 if drones <= 16 else 0.1)
    sw = (swarm.p, swarm.q, swarm.v, swarm.w)
    dpe = swarm.drones_per_env
    runs = [_run(cuda, dpe, sw, rk4, r, b) for r in (False, True) for b in (None, 512)]
    state, kin, idx, rel, act = runs[0]
    for other in runs[1:]:
        assert torch.equal(idx, other[2])
        for a, b in zip((state, kin, rel), (other[0], other[1], other[3])):
            torch.testing.assert_close(a, b, rtol=1e-5, atol=1e-5)
    # behind a lone drone, far away, with the same actions
    uneven = np.concatenate([[1], dpe]).astype(np.int32)
    sw1 = [np.concatenate([a[:1], a]) for a in sw]
    sw1[0][0] = (0.0, 0.0, 0.4)
    h = mdg.Handle(uneven, np.full(len(uneven), 7, np.uint32),
                   None if not rk4 else _rk4_constants())
    for rollout in (False, True):
        s1 = mdg.pack_state(*sw1, device=cuda)
        k1, i1, r1 = h.new_obs(cuda)
        act1 = torch.cat([act[:1], act])
        if rollout:
            h.rollout(s1, act1, mdg.ACT_PID, 2, 1, mdg.OBS_LAST, k1, i1, r1)
        else:
            h.step_obs(s1, act1, mdg.ACT_PID, 2, k1, i1, r1)
        torch.testing.assert_close(s1[:, 1:], state, rtol=1e-5, atol=1e-5)
        assert torch.equal(torch.where(i1[1:] >= 0, i1[1:] - 1, i1[1:]), idx)
    # the oracle
    if not rk4:
        x0 = swarm.x13()
        z = np.zeros((swarm.n, 6)), np.zeros((swarm.n, 4))
        layout = (dpe, np.full(envs, 7))
        wp, types = act.cpu().numpy().astype(np.float64), np.full(envs, mdg.ACT_PID)
        xo = oracle_step(P, layout, x0, *z, wp, types, 2)[0]
        assert_horizon_close(oracle_arrays(state)[0], xo, tolerance_response(P, layout, x0, *z, wp, types, 2), 2,
                             what=f"{drones} drones")


@pytest.mark.parametrize("rk4", [False, True])
@pytest.mark.parametrize("sizes", [[10] * 7, [12] * 9, [14] * 5, [18] * 4, [30] * 3, [6, 10, 16, 1, 1, 2, 8, 12, 32, 14, 18]])
def test_runtime_pairs_agree_with_single_sources(cuda, sizes, rk4):
    """Even sizes without a variant of their own, at even places inside the warps of small blocks, read the
    downwash sources in pairs; the same environments in blocks of 512 read them one by one."""
    dpe = np.array(sizes, np.int32)
    place = 0
    for n in sizes:  # as whole environments fill blocks of 32 drones
        place = 0 if place + n > 32 else place
        assert n == 1 or (place % 2 == 0 and n % 2 == 0)
        place += n
    n = int(dpe.sum())
    p = np.zeros((n, 3), np.float32)
    k = np.concatenate([np.arange(m) for m in sizes])
    p[:, 0], p[:, 1], p[:, 2] = 0.3 * (k % 4), 0.3 * (k // 4), 0.4 + 0.2 * k  # every drone on a height of its own
    _, q, v, w = wl.random_states(303, n)
    sw = (p, q, 0.1 * v, 0.1 * w)
    runs = [_run(cuda, dpe, sw, rk4, r, b) for b in (32, 512) for r in (False, True)]
    for other in runs[1:]:
        assert torch.equal(runs[0][2], other[2])
        for a, b in zip((runs[0][0], runs[0][1], runs[0][3]), (other[0], other[1], other[3])):
            torch.testing.assert_close(a, b, rtol=1e-5, atol=1e-5)


def _rk4_constants():
    c = mdg.Constants.cf2x()
    c.integrator = mdg.INTEGRATOR_RK4
    return c
