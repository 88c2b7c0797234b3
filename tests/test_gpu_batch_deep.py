"""A batch of many deep, narrow volumes: the backprojector's small chunks of 62
members of 4780 planes (1195 each) are more than one grid's z extent of 65535.
Each member equals its problem alone."""
import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


def test_many_deep_members(tigre):
    geo = synth.geometry((8, 6, 4780), 1.0, (12, 16), (1.6, 450.0), dso=20000.0, dsd=30000.0)
    members = 62
    with tigre.Geometry(geo, synth.angles(3, first=0.2)) as G:
        gen = torch.Generator(device="cuda").manual_seed(3)
        bs = [torch.rand(tuple(G.proj_shape), device="cuda", generator=gen) for _ in range(members)]
        xs = [torch.zeros(G.vol_shape, device="cuda") for _ in bs]
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        st = tigre.tigre_cgls_batch_begin(G.handle, bs, xs, n_iter_hint=2, stream=s, x0_zero=True)
        tigre.tigre_cgls_batch_iterate(st, 2)
        hs = [tigre.tigre_cgls_batch_history(st, i, 2) for i in range(members)]
        tigre.tigre_cgls_batch_end(st)
        torch.cuda.synchronize()
        for i in (0, 1, 53, 54, 55, 61):
            x = torch.zeros(G.vol_shape, device="cuda")
            h = tigre.tigre_cgls(G.handle, bs[i], x, 2, x0_zero=True)
            assert torch.equal(x, xs[i]), i
            assert np.array_equal(h, hs[i]), i
