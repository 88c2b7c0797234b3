"""A captured graph of one adjoint call stays valid when the handle later serves
a call of the other scatter (few rays: scalar accumulators; many: quads), whose
workspace must not replace the one that the graph holds."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


def test_graph_of_few_angles_survives_a_call_of_many(tigre):
    geo = synth.geometry((41, 37, 30), (1.0, 0.9, 1.1), (401, 33), (70.0 / 401, 48.0 / 33),
                         dso=300.0, dsd=450.0, off_origin=(0.4, -0.6, 0.3))
    ang = np.random.default_rng(1).uniform(-4.0, 9.0, 29)
    y = np.random.default_rng(2).random((29, 33, 401)).astype(np.float32)
    few, many = slice(3, 8), slice(0, 29)  # 66,000 and 384,000 rays
    ref = {s: oracle.adjoint(geo, ang[s], y[s]) for s in (few, many)}

    def rel(x, s):
        return float(np.linalg.norm(x.cpu().numpy() - ref[s]) / np.linalg.norm(ref[s]))

    with tigre.Geometry(geo, ang) as G:
        yt = torch.from_numpy(y).cuda()
        yf = yt[few].contiguous()
        x = G.backward(yf, angle_begin=3, weight="adjoint")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            G.backward(yf, out=x, angle_begin=3, weight="adjoint")
        full = G.backward(yt, weight="adjoint")
        held = [torch.full((1 << 22,), 7.0, device="cuda") for _ in range(4)]
        x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert rel(x, few) < 1e-4 and rel(full, many) < 1e-4
        assert all(bool((h == 7.0).all()) for h in held)
        assert rel(G.backward(yt, weight="adjoint"), many) < 1e-4
