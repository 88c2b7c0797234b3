"""The column projector (warps of detector rows, quads with z fastest) against
the scalar kernel, bit for bit, where its tiles can go wrong: detector rows and
columns that are no multiple of a warp's, short angle groups, partial ranges,
rays that enter and leave through the top and bottom faces, and rays that only
graze the volume."""
import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


def geometry(nu, nv, n=(41, 37, 30), pitch=None, dso=300.0):
    dv = 30.0 * 1.6 / nv if pitch is None else pitch
    return synth.geometry(n, (1.0, 0.9, 1.1), (nu, nv), (70.0 / nu, dv), dso=dso, dsd=1.5 * dso,
                          off_origin=(0.4, -0.6, 0.3), off_det=(1.1, -0.4))


CASES = {
    # (detector columns, rows, angles, range): at least 250,000 rays each
    "rows 16": (1501, 16, 12, (0, None)),
    "rows 18, odd columns": (1999, 18, 7, (0, None)),
    "rows 27, a range": (1203, 27, 23, (3, 11)),
    "rows 129, three angles": (677, 129, 3, (0, None)),
    "one row over a tile": (401, 33, 29, (0, None)),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_columns_equal_the_scalar_kernel(tigre, name, dtype):
    nu, nv, na, (a0, count) = CASES[name]
    geo = geometry(nu, nv)
    ang = np.random.default_rng(nv).uniform(-4.0, 9.0, na)
    count = na if count is None else count
    assert nu * nv * count >= 250000
    with tigre.Geometry(geo, ang) as G:
        v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=nu)).cuda().to(dtype)
        out = {}
        for path in (tigre.FWD_L1, tigre.FWD_AUTO):
            tigre.tigre_geometry_set_forward_path(G.handle, path)
            n0 = tigre.tigre_launch_count()
            out[path] = G.forward(v, dtype=torch.float32, angle_begin=a0, angle_count=count)
            launches = tigre.tigre_launch_count() - n0
        assert launches == 2  # one set of quads and one march: the column projector
    assert torch.isfinite(out[tigre.FWD_AUTO]).all()
    assert torch.equal(out[tigre.FWD_L1], out[tigre.FWD_AUTO])


@pytest.mark.parametrize("n", [(41, 37, 2), (3, 64, 30), (1, 1, 40)])
def test_columns_on_thin_volumes(tigre, n):
    """Volumes of one to three voxels along an axis, seen under a wide detector
    (most rays miss, some cross a corner with one sample)."""
    geo = geometry(901, 96, n=n, pitch=0.5)
    with tigre.Geometry(geo, synth.angles(5, first=0.1)) as G:
        v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=1)).cuda()
        out = {}
        for path in (tigre.FWD_L1, tigre.FWD_AUTO):
            tigre.tigre_geometry_set_forward_path(G.handle, path)
            out[path] = G.forward(v)
    assert torch.equal(out[tigre.FWD_L1], out[tigre.FWD_AUTO])
