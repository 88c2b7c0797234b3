"""Projections of angle ranges of volumes wider than one x-y brick: whatever
kernel a range takes (one or two angles are too few for the column projector),
it is the full projection's slice bit for bit, as for narrow volumes."""
import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = {  # (volume, detector, angles)
    "wide in x, full range by columns": ((520, 300, 90), (600, 100), 12),
    "wide in y, full range by columns": ((260, 530, 85), (640, 96), 14),
    "wide, full range by bricks": ((520, 300, 20), (600, 12), 12),
}


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_ranges_equal_the_full_projection(tigre, name, dtype):
    n, det, na = SHAPES[name]
    geo = synth.geometry(n, 0.5, det, (460.0 / det[0], 0.8 * n[2] / det[1]), dso=800.0, dsd=1200.0,
                         off_origin=(0.4, -0.6, 0.3), off_det=(0.4, -0.3))
    ang = np.random.default_rng(na).uniform(0.0, 2.0 * np.pi, na)
    with tigre.Geometry(geo, ang) as G:
        v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=na)).cuda().to(dtype)
        full = G.forward(v, dtype=torch.float32)
        assert torch.isfinite(full).all()
        for a0, count in ((0, 1), (5, 2), (3, 7), (na - 1, 1)):
            part = G.forward(v, dtype=torch.float32, angle_begin=a0, angle_count=count)
            assert torch.equal(part, full[a0:a0 + count]), (a0, count)
