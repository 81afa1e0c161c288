"""3D CSR rows without gradient records (plain float flowmaps, double coordinates): the staged kernel, the
default, equals the plain-load kernel bit for bit on whole and ragged tiles, on a row longer than a
stage, and with col_idx off a 16-byte boundary (left to the plain kernel)."""
import numpy as np
import pytest

from paper_2408_02758_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def mesh(case, dtype):
    shape = {"whole": (16, 16, 16), "ragged": (17, 13, 11), "one": (2, 2, 2)}.get(case, (24, 20, 18))
    m = I.make_mesh(shape, (0, 0, 0), (2, 1, 1), I.KUHN, 0.3, 5, coord_dtype=dtype)
    if case != "hub":
        return m
    n = m.n_nodes
    rows = [m.col_idx[m.row_ptr[i]: m.row_ptr[i + 1]] for i in range(n)]
    rows[0] = np.arange(1, n, dtype=np.int32)
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    return I.mesh_from_arrays(m.coords, rp, np.concatenate(rows))


@pytest.mark.parametrize("case", ["whole", "ragged", "one", "hub", "offset"])
@pytest.mark.parametrize("dtype,prec", [(np.float32, "fp32"), (np.float64, "fp32"), (np.float64, "fp32c")])
def test_staged_equals_direct(case, dtype, prec):
    import torch

    from paper_2408_02758_gb300 import ftle as F

    m = mesh(case, dtype)
    dm = F.DeviceMesh.from_mesh(m)
    if case == "offset":
        ci = torch.empty(m.nnz + 1, dtype=torch.int32, device="cuda")
        ci[1:] = dm.col_idx
        dm = F.DeviceMesh(dm.coords, dm.row_ptr, ci[1:])
    phi = F.flowmap_empty(3, m.n_nodes, prec)
    F.ftle_advect(dm, I.FlowSpec.abc(), 0.0, 1.0, 0.01, prec, phi)
    got = []
    for staging in (0, 1):
        out = torch.full((m.n_nodes,), 9.0, device="cuda")
        lam = torch.full((m.n_nodes,), 9.0, dtype=torch.float64, device="cuda")
        ws = F.workspace_empty(F.ftle_workspace_bytes(m.n_nodes))
        F.ftle_gradient_eig(dm, phi, prec, 1.0, out, lam, ws, options=F.make_options(grad_staging=staging))
        cnt = F.ftle_read_counters(ws)
        assert cnt["n_wait_timeouts"] == 0
        got.append((out.cpu().numpy(), lam.cpu().numpy(), cnt["n_flagged"]))
    assert got[0][2] == got[1][2]
    assert np.array_equal(got[0][0], got[1][0], equal_nan=True) and np.array_equal(got[0][1], got[1][1], equal_nan=True)
