"""The ABC flow's carried steps, one and two nodes per thread: a node's states do not depend on how many
nodes share its thread, warp or launch shape, nor on checkpoints stored on the way, for every refresh
period and for step counts that end inside a period or before the waiting increments join the state."""
import math

import numpy as np
import pytest

import oracle as O
from paper_2408_02758_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FLOW = I.FlowSpec.abc(1.7, 1.4, 0.97)
BIG = 152 * 128 + 40  # more than one warp per SM sub-partition: two nodes per thread


@pytest.fixture(scope="module")
def F():
    from paper_2408_02758_gb300 import ftle

    return ftle


@pytest.fixture(scope="module")
def nodes():
    return (np.random.default_rng(6).random((3, BIG)) * 2 * math.pi).astype(np.float32)


def advect(F, x, steps, ckpt=0, **opt):
    import torch

    n = x.shape[1]
    dm = F.DeviceMesh(torch.from_numpy(np.ascontiguousarray(x)).cuda(),
                      torch.zeros(n + 1, dtype=torch.int32, device="cuda"),
                      torch.zeros(0, dtype=torch.int32, device="cuda"))
    phi = F.flowmap_empty(3, n, "fp32c")
    ck = F.checkpoints_empty(3, n, steps, ckpt, "fp32c") if ckpt else None
    F.ftle_advect(dm, FLOW, 0.0, steps * 0.01, 0.01, "fp32c", phi, ck, ckpt, options=F.make_options(**opt))
    return F.flowmap_pairs(phi, 3, n).cpu().numpy(), None if ck is None else ck.view(-1, 3, n, 2).cpu().numpy()


@pytest.mark.parametrize("refresh", [2, 4, 8, 32])
@pytest.mark.parametrize("steps", [1, 3, 4, 7, 8, 9, 45])
def test_states_do_not_depend_on_the_mesh(F, nodes, steps, refresh):
    whole, _ = advect(F, nodes, steps, abc_refresh=refresh)
    for n in (1, 31, 32, 33, 63, 64, 65, 1000):
        assert np.array_equal(advect(F, nodes[:, :n], steps, abc_refresh=refresh)[0], whole[:, :n])
    for opt in ({"advect_block": 32}, {"advect_block": 256, "advect_blocks_per_sm": 1}):
        assert np.array_equal(advect(F, nodes, steps, abc_refresh=refresh, **opt)[0], whole)
    # each step's increment (at most h U, U the largest pair sum) is off by a few roundings, at most
    # 2^-21 of it; an error grows along the flow by at most exp(L T), L = U
    U, T = 1.7 + 1.4, steps * 0.01
    ref = O.advect(FLOW.kind, FLOW.params, nodes[:, :500].astype(np.float64), T, 0.01)
    assert np.abs(whole[:, :500].astype(np.float64).sum(-1) - ref).max() <= T * U * 2.0**-21 * math.exp(U * T)


@pytest.mark.parametrize("ckpt", [1, 3, 8, 37])
def test_checkpoints_leave_the_steps_alone(F, nodes, ckpt):
    two, c2 = advect(F, nodes, 45, ckpt=ckpt)
    one, c1 = advect(F, nodes[:, :77], 45, ckpt=ckpt)
    assert np.array_equal(two, advect(F, nodes, 45)[0])
    assert np.array_equal(two[:, :77], one) and np.array_equal(c2[:, :, :77], c1)
    for s in range(45 // ckpt + 1):  # a checkpoint is the flowmap of that many steps
        if s:
            assert np.array_equal(c1[s], advect(F, nodes[:, :77], s * ckpt)[0])
