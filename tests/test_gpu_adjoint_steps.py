"""The adjoint of the double gyre's steps on both of its routes -- nodes whose every stage angle is small
enough to turn stage one's sines and cosines, and steps too long for that, evaluated in full -- and on
both block sizes (segments of up to 50 steps, and longer ones), against the oracle's forward-mode derivative.
Tolerance: that of the short integrations in test_gpu_adjoint (1e-4 of a component, at least 1e-3 of
the largest), the float steps being no more than there."""
import numpy as np
import pytest

import oracle as O
from paper_2408_02758_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32c", "fp32"])
@pytest.mark.parametrize("T,dt,ckpt", [(5.0, 0.02, 50), (5.0, 0.02, 51), (-3.0, 0.02, 64), (5.0, 1.0, 3), (4.0, 0.8, 60)])
def test_adjoint_routes(T, dt, ckpt, prec):
    import torch

    from paper_2408_02758_gb300 import ftle
    from paper_2408_02758_gb300.autograd import ftle_field

    mesh = I.make_mesh((67, 31), (0.0, 0.0), (2.0, 1.0), I.TRI, 0.3, 11)  # 2077 nodes: a ragged last block
    p0 = I.FlowSpec.double_gyre().params[:3].copy()
    x0 = mesh.coords.astype(np.float64)
    wts = ((x0[0] >= 0.5) & (x0[0] <= 1.5)).astype(np.float64)
    wts /= wts.sum()
    params = torch.tensor(p0, dtype=torch.float64, requires_grad=True)
    field = ftle_field(params, ftle.DeviceMesh.from_mesh(mesh), T, dt, prec, ckpt)
    (field.double().cpu() * torch.from_numpy(wts)).sum().backward()
    got = params.grad.numpy()
    want, _ = O.param_grad(x0, mesh.row_ptr, mesh.col_idx, p0, T, dt, wts)
    # plain float flowmaps: rounding 6e-8 a step over spacings of 1/33, 250 steps
    tol = 1e-4 if prec == "fp32c" else 2e-3
    rel = np.abs(got - want) / np.maximum(np.abs(want), 1e-3 * np.abs(want).max())
    assert np.all(rel < tol), (got, want, rel)
