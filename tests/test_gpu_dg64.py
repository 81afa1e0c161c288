"""Double-precision double gyre on the FP32 pipes: chunk edges of the coefficient table, ragged node
counts, nodes outside the domain or next to a wall (integrated in double), checkpoints, both
coordinate types, and arguments that leave the whole mesh to the double kernel."""
import math

import numpy as np
import pytest

import oracle as O
from paper_2408_02758_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2408_02758_gb300 import ftle

    return ftle


def points(n, seed):
    """Domain nodes, walls and corners, then a few nodes outside the domain and next to the walls."""
    x = np.random.default_rng(seed).random((2, n)) * np.array([[2.0], [1.0]])
    special = np.array([[0, 0], [2, 1], [0, 0.3], [2, 0.7], [0.4, 0], [1.6, 1], [-0.1, 0.5], [0.5, 1.2], [2.25, -0.5],
                        [1e-200, 0.25], [0.25, 1e-12], [2.0**-30, 2.0**-30]]).T
    k = min(n, special.shape[1])
    x[:, n - k:] = special[:, :k]
    return np.ascontiguousarray(x)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 300, 5003])
@pytest.mark.parametrize("steps", [1, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("sign", [1, -1])
def test_flowmap_against_oracle(F, n, steps, sign):
    import torch

    dt, T = 2.0 / 1024, sign * steps * 2.0 / 1024
    p = (0.1, 0.25, 2 * math.pi / 10)
    x = points(n, n + steps)
    if n % 2:
        x = x.astype(np.float32).astype(np.float64)
    c = torch.from_numpy(x).cuda()
    if n % 2:
        c = c.float()
    dm = F.DeviceMesh(c, torch.zeros(n + 1, dtype=torch.int32, device="cuda"),
                      torch.zeros(0, dtype=torch.int32, device="cuda"))
    ck = F.checkpoints_empty(2, n, steps, 256, "fp64") if steps >= 256 else None
    phi = F.flowmap_empty(2, n, "fp64")
    F.ftle_advect(dm, I.FlowSpec.double_gyre(*p), 0.0, T, dt, "fp64", phi, ck, 256)
    # a step rounds the state by at most 2.3e-16 here and in the oracle (its increments' roundings
    # are far below); an error grows along the flow by at most exp(L |T|)
    def tol(t):
        return 4.6e-16 * (t / dt + 1) * math.exp(math.pi**2 * p[0] * (1 + 2 * p[1]) * t)

    got, ref = phi.cpu().numpy(), O.advect(I.DOUBLE_GYRE, p, x, T, dt)
    inside = (np.abs(x - np.array([[1.0], [0.5]])) <= np.array([[1.0], [0.5]])).all(0)
    assert np.abs(got - ref)[:, inside].max(initial=0) <= tol(abs(T))
    assert np.allclose(got, ref, rtol=1e-9, atol=0)  # outside, and tiny coordinates keep their digits
    if ck is not None:
        for s in range(steps // 256 + 1):
            r = O.advect(I.DOUBLE_GYRE, p, x, sign * s * 256 * dt, dt) if s else x
            assert np.abs(ck[s].view(2, n).cpu().numpy() - r)[:, inside].max(initial=0) <= tol(s * 256 * dt)


@pytest.mark.parametrize("p,dt,T", [((0.0, 0.25, 1.0), 0.01, 1.0), ((0.1, 1.5, 1.0), 0.01, 1.0),
                                    ((2.0, 0.25, 1.0), 0.1, 1.0), ((0.1, 0.5, 1.0), 0.05, 40.0)])
def test_other_arguments_run_in_double(F, p, dt, T):
    import torch

    x = np.random.default_rng(3).random((2, 257)) * np.array([[2.0], [1.0]])
    dm = F.DeviceMesh(torch.from_numpy(x).cuda(), torch.zeros(258, dtype=torch.int32, device="cuda"),
                      torch.zeros(0, dtype=torch.int32, device="cuda"))
    phi = F.flowmap_empty(2, 257, "fp64")
    F.ftle_advect(dm, I.FlowSpec.double_gyre(*p), 0.0, T, dt, "fp64", phi)
    assert np.allclose(phi.cpu().numpy(), O.advect(I.DOUBLE_GYRE, p, x, T, dt), rtol=0, atol=1e-6)
