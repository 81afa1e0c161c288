"""Plain float double gyre, one and two nodes per thread: the flowmap does not depend on how many nodes
share a thread or on the launch shape, its checkpoints are flowmaps of fewer steps, and the field equals
the batch's, which advances one node per thread by the same float operations."""
import numpy as np
import pytest

from paper_2408_02758_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FLOW = I.FlowSpec.double_gyre(0.1, 0.3, 0.7)
BIG = 152 * 128 + 40


def advect(F, x, steps, ckpt=0, **opt):
    import torch

    n = x.shape[1]
    dm = F.DeviceMesh(torch.from_numpy(np.ascontiguousarray(x)).cuda(),
                      torch.zeros(n + 1, dtype=torch.int32, device="cuda"),
                      torch.zeros(0, dtype=torch.int32, device="cuda"))
    phi = F.flowmap_empty(2, n, "fp32")
    ck = F.checkpoints_empty(2, n, steps, ckpt, "fp32") if ckpt else None
    F.ftle_advect(dm, FLOW, 0.0, steps * 0.01, 0.01, "fp32", phi, ck, ckpt, options=F.make_options(**opt))
    return phi.cpu().numpy(), None if ck is None else ck.view(-1, 2, n).cpu().numpy()


@pytest.fixture(scope="module")
def F():
    from paper_2408_02758_gb300 import ftle

    return ftle


@pytest.mark.parametrize("steps", [1, 30, 2049])
def test_flowmap_does_not_depend_on_the_mesh(F, steps):
    x = (np.random.default_rng(7).random((2, BIG)) * np.array([[2.4], [1.3]]) - 0.2).astype(np.float32)
    whole, ck = advect(F, x, steps, ckpt=13)
    for n in (1, 31, 32, 33, 63, 64, 65, 1000):
        assert np.array_equal(advect(F, x[:, :n], steps)[0], whole[:, :n])
    for opt in ({"advect_block": 32}, {"advect_block": 256, "advect_blocks_per_sm": 1}):
        assert np.array_equal(advect(F, x, steps, **opt)[0], whole)
    if steps >= 13:
        assert np.array_equal(ck[1], advect(F, x, 13)[0])


@pytest.mark.parametrize("shape", [(40, 21), (221, 111)])
def test_field_equals_the_batch(F, shape):
    import torch

    m = I.make_mesh(shape, (0, 0), (2, 1), I.TRI, 0.3, 5)
    dm = F.DeviceMesh.from_mesh(m)
    single = F.compute(dm, FLOW, 3.0, 0.01, "fp32")
    out = torch.empty_like(single)
    ws = F.workspace_empty(F.ftle_batch_workspace_bytes([dm], "fp32"))
    F.ftle_batch([dm], [FLOW], [3.0], 0.01, "fp32", [out], ws)
    assert torch.equal(torch.nan_to_num(single), torch.nan_to_num(out))
