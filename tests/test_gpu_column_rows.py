"""The column projector's two warp shapes (8 or 16 detector rows) on planes of at
least 640^2 voxels: ragged rows and columns, partial angle ranges, few rows, and a
batch, against the quad kernel on the same volume, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


def geometry(n, nu, nv):
    """Detector rows about one plane apart at the axis, the detector a little
    larger than the volume's shadow."""
    return synth.geometry(n, 0.4, (nu, nv), (560.0 / nu, 0.4 * 1.45 * n[2] / nv), dso=800.0, dsd=1200.0,
                          off_origin=(0.3, -0.5, 0.2), off_det=(0.4, -0.3))


CASES = {  # (volume, columns, rows, angles, range)
    "16 rows, one tile": ((656, 648, 12), 701, 16, 230, (0, 230)),
    "16-row warps, ragged": ((644, 660, 250), 333, 261, 13, (0, 13)),
    "16-row warps, a range": ((652, 640, 250), 301, 258, 23, (5, 13)),
    "8-row warps, ragged": ((648, 644, 110), 459, 111, 60, (0, 60)),
    "8-row warps, a range": ((640, 641, 200), 401, 202, 40, (7, 33)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_rows_equal_the_quad_kernel(tigre, name):
    n, nu, nv, na, (a0, count) = CASES[name]
    ang = np.random.default_rng(nv).uniform(-4.0, 9.0, na)
    with tigre.Geometry(geometry(n, nu, nv), ang) as G:
        v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=nu)).cuda()
        out, launches = {}, {}
        for path in (tigre.FWD_QUAD, tigre.FWD_AUTO):
            tigre.tigre_geometry_set_forward_path(G.handle, path)
            n0 = tigre.tigre_launch_count()
            out[path] = G.forward(v, angle_begin=a0, angle_count=count)
            launches[path] = tigre.tigre_launch_count() - n0
    assert launches == {tigre.FWD_QUAD: 3, tigre.FWD_AUTO: 2}  # two sets of quads; one
    assert torch.isfinite(out[tigre.FWD_AUTO]).all()
    assert torch.equal(out[tigre.FWD_QUAD], out[tigre.FWD_AUTO])


def test_more_than_2_28_quads(tigre):
    """Byte offsets beyond 32 bits (704 x 696 x 646 padded voxels), ragged tiles."""
    geo, ang = geometry((700, 692, 642), 203, 349), synth.angles(11, first=0.3)
    with tigre.Geometry(geo, ang) as G:
        v = torch.rand(tuple(G.vol_shape), device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(5))
        n0 = tigre.tigre_launch_count()
        out = G.forward(v)
        assert tigre.tigre_launch_count() - n0 == 2  # columns
        tigre.tigre_geometry_set_forward_path(G.handle, tigre.FWD_QUAD)
        assert torch.isfinite(out).all() and torch.equal(out, G.forward(v))


@pytest.mark.parametrize("graph", [False, True])
def test_batched_16_row_warps(tigre, graph):
    """Members of a batch (two iterations of CGLS) equal their problems alone."""
    geo, ang = geometry((640, 644, 250), 333, 259), synth.angles(13, first=0.2)
    with tigre.Geometry(geo, ang) as G:
        bs = [torch.from_numpy(np.random.default_rng(i).random((13, 259, 333)).astype(np.float32)).cuda()
              for i in range(2)]
        ref = []
        for b in bs:
            x = torch.zeros(G.vol_shape, device="cuda")
            h = tigre.tigre_cgls(G.handle, b, x, 2, x0_zero=True)
            ref.append((x, h))
        xs = [torch.zeros(G.vol_shape, device="cuda") for _ in bs]
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        st = tigre.tigre_cgls_batch_begin(G.handle, bs, xs, n_iter_hint=2, stream=s, graph=graph,
                                          x0_zero=True)
        tigre.tigre_cgls_batch_iterate(st, 2)
        hs = [tigre.tigre_cgls_batch_history(st, i, 2) for i in range(2)]
        tigre.tigre_cgls_batch_end(st)
        torch.cuda.synchronize()
    for (x, h), xb, hb in zip(ref, xs, hs):
        assert torch.equal(x, xb)
        assert np.array_equal(h, hb)


ROUTES = {  # (volume, columns, rows, row pitch or None, angles): launches of a projection
    "a small object under a tall detector": (((29, 194, 37), 416, 764, 1.8, 12), 3),
    "a shadow of 20 rows over four tiles": (((200, 210, 20), 300, 400, 1.0, 150), 3),
    "few rows at few angles": (((512, 520, 24), 512, 24, None, 24), 3),
    "few rows at many angles": (((512, 520, 24), 512, 24, None, 200), 2),
    "few rows of a tall volume": (((400, 410, 200), 256, 40, 0.4, 26), 2),
    "tall detector, few angles": (((300, 310, 90), 301, 97, None, 14), 2),
}


@pytest.mark.parametrize("name", list(ROUTES))
def test_calls_too_small_for_columns_take_quads(tigre, name):
    """Where few rays cross the volume, or few rows at few angles do, the quad
    kernel (two sets of quads and a march: three launches) is the faster one; the
    results are the same bits."""
    (n, nu, nv, dv, na), launches = ROUTES[name]
    geo = geometry(n, nu, nv)
    if dv:
        geo["d_det"] = (560.0 / nu * n[1] / 640.0, dv * 0.4 * 1.5)
    with tigre.Geometry(geo, synth.angles(na, first=0.1)) as G:
        v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=nu)).cuda().to(torch.bfloat16)
        n0 = tigre.tigre_launch_count()
        out = G.forward(v)
        assert tigre.tigre_launch_count() - n0 == launches
        tigre.tigre_geometry_set_forward_path(G.handle, tigre.FWD_QUAD)
        assert torch.equal(out, G.forward(v))
