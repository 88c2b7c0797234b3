"""The exact adjoint's column scatter (quad accumulators, vector reductions) where
its tiles can go wrong: ragged detectors, partial angle ranges, 16-bit storage
and accumulation over ranges, against the FP64 oracle at 1e-4 relative L2 (the
repository's tolerance for FP32 operators; 1e-2 where the result is stored in
16 bits)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,nu,nv,na,a0,count", [((41, 37, 30), 401, 33, 29, 0, 29),
                                                 ((33, 65, 34), 613, 27, 23, 3, 17),
                                                 ((3, 40, 1), 677, 129, 3, 0, 3)])
@pytest.mark.parametrize("dtype,tol", [(torch.float32, 1e-4), (torch.bfloat16, 1e-2)])
def test_adjoint_columns(tigre, n, nu, nv, na, a0, count, dtype, tol):
    assert nu * nv * count >= 250000
    geo = synth.geometry(n, (1.0, 0.9, 1.1), (nu, nv), (70.0 / nu, 48.0 / nv), dso=300.0, dsd=450.0,
                         off_origin=(0.4, -0.6, 0.3), off_det=(1.1, -0.4))
    ang = np.random.default_rng(nv).uniform(-4.0, 9.0, na)
    y = np.random.default_rng(nu).random((count, nv, nu)).astype(np.float32)
    with tigre.Geometry(geo, ang) as G:
        yt = torch.from_numpy(y).cuda().to(dtype)
        n0 = tigre.tigre_launch_count()
        x = G.backward(yt, angle_begin=a0, weight="adjoint")
        assert tigre.tigre_launch_count() - n0 == 2  # the scatter and the sum of cells
    ref = oracle.adjoint(geo, ang[a0:a0 + count], yt.float().cpu().numpy())
    assert rel(x.float().cpu().numpy(), ref) < tol
