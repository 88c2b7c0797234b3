"""The FDK row filter at the edges of its block shapes (8 rows up to 2048
columns, 4 up to 8192, one beyond; even and odd row lengths down to one pixel;
rows that are no multiple of the block's) through the whole FDK call, against
the FP64 oracle at 1e-4 relative L2."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [1, 2, 7, 8, 33, 258, 509, 2048, 2049, 8192, 8193])
@pytest.mark.parametrize("nv", [3, 9])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
def test_fdk_filter_shapes(tigre, nu, nv, dtype):
    geo = synth.geometry((24, 22, 10), 1.0, (nu, nv), (45.0 / nu, 15.0 / nv), dso=200.0, dsd=300.0,
                         off_det=(0.3, -0.2))
    ang = synth.angles(5, first=0.3)
    y = np.random.default_rng(nu).random((5, nv, min(nu, 509))).astype(np.float32)
    if nu > 509:  # long rows: 509 random knots, as a column coordinate is only good to nu 2^-23 px
        at = np.linspace(0.0, 508.0, nu)
        y = np.stack([[np.interp(at, np.arange(509), r) for r in img] for img in y]).astype(np.float32)
    with tigre.Geometry(geo, ang) as G:
        yt = torch.from_numpy(y).cuda().to(dtype)
        x = G.fdk(yt, dtype=torch.float32).cpu().numpy()
    ref = oracle.fdk(geo, ang, yt.float().cpu().numpy())
    assert np.linalg.norm(x - ref) / np.linalg.norm(ref) < 1e-4
