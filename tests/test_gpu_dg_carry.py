"""The double gyre's carried steps, one and two nodes per thread: a node's states do not depend on how
many nodes share its thread, warp or launch shape (tile edges, ragged ends, nodes outside the domain
between safe ones, checkpoints, horizons beyond one coefficient table), and they agree with the oracle."""
import math

import numpy as np
import pytest

import oracle as O
from paper_2408_02758_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FLOW = I.FlowSpec.double_gyre(0.1, 0.3, 0.7)
BIG = 152 * 128 + 40  # more than one warp per SM sub-partition: two nodes per thread


@pytest.fixture(scope="module")
def F():
    from paper_2408_02758_gb300 import ftle

    return ftle


@pytest.fixture(scope="module")
def nodes():
    x = np.random.default_rng(5).random((2, BIG)) * np.array([[2.0], [1.0]])
    x[:, ::7] += np.array([[0.3], [0.2]])  # some leave the domain
    x[0, :4], x[1, :4] = [0, 2, 0.5, 1.5], [0.5, 0.5, 0, 1]
    return x.astype(np.float32)


def advect(F, x, steps, dt=0.01, ckpt=0, **opt):
    import torch

    n = x.shape[1]
    dm = F.DeviceMesh(torch.from_numpy(np.ascontiguousarray(x)).cuda(),
                      torch.zeros(n + 1, dtype=torch.int32, device="cuda"),
                      torch.zeros(0, dtype=torch.int32, device="cuda"))
    phi = F.flowmap_empty(2, n, "fp32c")
    ck = F.checkpoints_empty(2, n, steps, ckpt, "fp32c") if ckpt else None
    F.ftle_advect(dm, FLOW, 0.0, steps * dt, dt, "fp32c", phi, ck, ckpt, options=F.make_options(**opt) if opt else None)
    segs = phi[-7 * 2 * n * 2:].cpu().numpy() if n % 16 == 0 else None  # unpadded slots
    return F.flowmap_pairs(phi, 2, n).cpu().numpy(), None if ck is None else ck.view(-1, 2, n, 2).cpu().numpy(), segs


@pytest.mark.parametrize("steps", [1, 7, 8, 15, 16, 17, 40, 2049])
def test_states_do_not_depend_on_the_mesh(F, nodes, steps):
    whole, _, _ = advect(F, nodes, steps)
    for n in (1, 31, 32, 33, 63, 64, 65, 1000):
        assert np.array_equal(advect(F, nodes[:, :n], steps)[0], whole[:, :n])
    for opt in ({"advect_block": 32}, {"advect_block": 256, "advect_blocks_per_sm": 1}):
        assert np.array_equal(advect(F, nodes, steps, **opt)[0], whole)


@pytest.mark.parametrize("ckpt", [1, 5, 16, 50])
def test_checkpoints_with_one_and_two_nodes_per_thread(F, nodes, ckpt):
    two, c2, s2 = advect(F, nodes[:, : BIG // 16 * 16], 120, ckpt=ckpt)
    one, c1, s1 = advect(F, nodes[:, :4096], 120, ckpt=ckpt)
    assert np.array_equal(two[:, :4096], one) and np.array_equal(c2[:, :, :4096], c1)
    n2 = two.shape[1]
    assert np.array_equal(s2.reshape(7, 2, n2, 2)[:, :, :4096], s1.reshape(7, 2, 4096, 2))
    # slot s holds the state after s * ckpt steps, closer than a float's rounding
    s = 120 // ckpt
    ref = O.advect(FLOW.kind, FLOW.params, nodes[:, :4096].astype(np.float64), s * ckpt * 0.01, 0.01)
    # each step's increment (at most 0.01 pi A 1.8) is off by a few roundings, at most 2^-21 of it; an
    # error grows along the flow by at most exp(L T) with L = pi^2 A (1 + 2 eps) (|x - 1| <= 1.3 here)
    tol = s * ckpt * 0.01 * 1.8 * math.pi * 0.1 * 2.0**-21 * math.exp(math.pi**2 * 0.1 * 1.8 * 1.2) + 1e-12
    assert np.abs(c1[s].astype(np.float64).sum(-1) - ref).max() <= tol
