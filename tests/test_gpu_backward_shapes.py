"""The voxel-driven backprojector at the edges of its launch shapes (4, 8 or 16
voxels per thread, chosen by the number of blocks): ragged columns and a ragged
last chunk of planes, against the FP64 oracle on sampled voxels, and the SART
update (whose normaliser takes a short cut inside the detector) against the
oracle's step.  Tolerance 1e-4 relative L2, the repository's for FP32
operators."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-4


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def geometry(n, det, margin=1.0):
    """A volume of 1 mm voxels; margin < 1: its shadow exceeds the detector."""
    half = 0.5 * max(n[0], n[1])
    du = margin * synth.detector_pixel(det[0], half)
    dv = margin * synth.detector_pixel(det[1], 0.5 * n[2], dso=1000.0 - half)
    return synth.geometry(n, 1.0, det, (du, dv), off_origin=(0.4, -0.3, 0.2), off_det=(0.7, -0.4))


SHAPES = {  # (volume, detector): blocks of 16 voxels per thread
    "4 voxels": ((33, 70, 61), (50, 41)),          # 2 x 9 x 4
    "8 voxels": ((161, 130, 43), (90, 57)),        # 6 x 17 x 3
    "16 voxels": ((513, 250, 81), (127, 61)),      # 17 x 32 x 6
}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("weight,mode", [("matched", oracle.BP_MATCHED), ("fdk", oracle.BP_FDK)])
@pytest.mark.parametrize("margin", [1.0, 0.6])
def test_backward_shapes(tigre, shape, weight, mode, margin):
    n, det = SHAPES[shape]
    geo, ang = geometry(n, det, margin), synth.angles(7, first=0.2)
    y = np.random.default_rng(n[0]).random((7, det[1], det[0])).astype(np.float32)
    vox = synth.random_voxels(*n, 2000, seed=3)
    vox[:4] = [(0, 0, 0), (n[0] - 1, n[1] - 1, n[2] - 1), (0, n[1] - 1, n[2] - 1), (n[0] - 1, 0, 0)]
    with tigre.Geometry(geo, ang) as G:
        b = G.backward(torch.from_numpy(y).cuda(), weight=weight).cpu().numpy()
    got = b[vox[:, 2], vox[:, 1], vox[:, 0]]
    assert rel(got, oracle.backward_voxels(geo, ang, y, vox, mode)) < TOL


@pytest.mark.parametrize("n,det", [((40, 37, 33), (31, 25)), ((129, 130, 41), (70, 33))])
def test_sart_update_shapes(tigre, n, det):
    """The shadow exceeds the detector, so no ray only grazes the volume (SART's
    row weights would amplify the FP32 set-up of such rays)."""
    geo, ang = geometry(n, det, 0.7), synth.angles(6, first=0.1)
    b = np.random.default_rng(9).random((6, det[1], det[0])).astype(np.float32)
    x_ref, h_ref = oracle.sirt(geo, ang, b.astype(np.float64), 2)
    with tigre.Geometry(geo, ang) as G:
        x = torch.zeros(G.vol_shape, device="cuda")
        h = tigre.tigre_sirt(G.handle, torch.from_numpy(b).cuda(), x, 2)
    assert rel(h, h_ref) < TOL
    assert rel(x.cpu().numpy(), x_ref) < TOL
