"""Every launch shape of the voxel-driven backprojector (4, 8 or 16 voxels per
thread, chosen by the blocks of 16 voxels) in each of its forms: plain sums, the
SART update with its normaliser, whose short cut runs where every cell lies on
the detector, and batches.  Against the FP64 oracle on sampled voxels at 1e-4
relative L2, the repository's tolerance for FP32 operators."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-4

SHAPES = {  # (volume, detector): blocks of 16 voxels per thread
    "16 voxels, 306 blocks": ((161, 130, 43), (90, 57)),
    "16 voxels, 456 blocks": ((97, 150, 83), (70, 61)),
    "8 voxels, 476 blocks": ((97, 130, 101), (70, 61)),
    "8 voxels, 612 blocks": ((161, 130, 91), (90, 77)),
    "16 voxels, 3264 blocks": ((513, 250, 81), (127, 61)),
}


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def blocks(n):
    return ((n[0] + 31) // 32) * ((n[1] + 7) // 8) * ((n[2] + 15) // 16)


def geometry(n, det, margin):
    """A volume of 1 mm voxels; margin < 1: its shadow exceeds the detector."""
    half = 0.5 * max(n[0], n[1])
    du = margin * synth.detector_pixel(det[0], half)
    dv = margin * synth.detector_pixel(det[1], 0.5 * n[2], dso=1000.0 - half)
    return synth.geometry(n, 1.0, det, (du, dv), off_origin=(0.4, -0.3, 0.2), off_det=(0.7, -0.4))


def sample(n):
    vox = synth.random_voxels(*n, 2000, seed=3)
    vox[:4] = [(0, 0, 0), (n[0] - 1, n[1] - 1, n[2] - 1), (0, n[1] - 1, n[2] - 1), (n[0] - 1, 0, 0)]
    return vox


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("weight,mode", [("matched", oracle.BP_MATCHED), ("fdk", oracle.BP_FDK)])
def test_backward(tigre, shape, weight, mode):
    n, det = SHAPES[shape]
    assert str(blocks(n)) in shape
    geo, ang, vox = geometry(n, det, 1.0), synth.angles(7, first=0.2), sample(n)
    y = np.random.default_rng(n[0]).random((7, det[1], det[0])).astype(np.float32)
    with tigre.Geometry(geo, ang) as G:
        got = G.backward(torch.from_numpy(y).cuda(), weight=weight).cpu().numpy()
    got = got[vox[:, 2], vox[:, 1], vox[:, 0]]
    assert rel(got, oracle.backward_voxels(geo, ang, y, vox, mode)) < TOL


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("margin", [0.7, 1.2])
def test_sart_update(tigre, shape, margin):
    """One SIRT iteration from zero: x = A_w^T (W b) / A_w^T 1 with W = 1 / (A 1).
    b is zero on rays that only graze the volume, whose W amplifies the FP32
    set-up of the ray."""
    n, det = SHAPES[shape]
    geo, ang, vox = geometry(n, det, margin), synth.angles(6, first=0.1), sample(n)
    a1 = oracle.forward(geo, ang, np.ones((n[2], n[1], n[0]), np.float32))
    b = np.random.default_rng(9).random(a1.shape) * (a1 > 0.1 * a1.max())
    r = np.where(a1 > 0.0, b / np.where(a1 > 0.0, a1, 1.0), 0.0)
    num = oracle.backward_voxels(geo, ang, r, vox, oracle.BP_MATCHED)
    den = oracle.backward_voxels(geo, ang, np.ones_like(r), vox, oracle.BP_MATCHED)
    with tigre.Geometry(geo, ang) as G:
        x = torch.zeros(G.vol_shape, device="cuda")
        tigre.tigre_sirt(G.handle, torch.from_numpy(b.astype(np.float32)).cuda(), x, 1)
    got = x.cpu().numpy()[vox[:, 2], vox[:, 1], vox[:, 0]]
    seen = den > 1e-12  # SIRT leaves voxels that no ray sees as they are
    assert rel(got, np.where(seen, num / np.where(seen, den, 1.0), 0.0)) < TOL


@pytest.mark.parametrize("shape", list(SHAPES)[:4])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_batch_equals_alone(tigre, shape, dtype):
    n, det = SHAPES[shape]
    with tigre.Geometry(geometry(n, det, 1.1), synth.angles(9, first=0.2)) as G:
        bs = [torch.from_numpy(np.random.default_rng(i).random(tuple(G.proj_shape)).astype(np.float32))
              .cuda().to(dtype) for i in range(3)]
        ref = []
        for b in bs:
            x = torch.zeros(G.vol_shape, device="cuda", dtype=dtype)
            ref.append((tigre.tigre_cgls(G.handle, b, x, 3, x0_zero=True), x))
        xs = [torch.zeros(G.vol_shape, device="cuda", dtype=dtype) for _ in bs]
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        st = tigre.tigre_cgls_batch_begin(G.handle, bs, xs, n_iter_hint=3, stream=s, x0_zero=True)
        tigre.tigre_cgls_batch_iterate(st, 3)
        hs = [tigre.tigre_cgls_batch_history(st, i, 3) for i in range(3)]
        tigre.tigre_cgls_batch_end(st)
        torch.cuda.synchronize()
    for (h, x), hb, xb in zip(ref, hs, xs):
        assert torch.equal(x, xb)
        assert np.array_equal(h, hb)
