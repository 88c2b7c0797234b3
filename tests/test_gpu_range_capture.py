"""A first projection of an angle range needs nothing prepared but the workspaces:
it can be captured in a CUDA graph on a handle whose workspaces exist, and ranges
of sorted angles allocate nothing."""
import gc

import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu

NA = 24
ANGLES = {"sorted": synth.angles(NA, first=0.1), "descending": synth.angles(NA, first=0.1)[::-1].copy(),
          "unsorted": np.random.default_rng(5).permutation(synth.angles(NA, first=0.1))}


def geometry():
    return synth.geometry((96, 90, 88), 1.0, (300, 101), (0.72, 1.35), dso=400.0, dsd=600.0,
                          off_det=(0.3, -0.2))


@pytest.mark.parametrize("order", list(ANGLES))
def test_first_call_of_a_range_inside_a_capture(tigre, order):
    with tigre.Geometry(geometry(), ANGLES[order]) as G:
        v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=3)).cuda()
        full = G.forward(v)  # the workspaces
        out = torch.zeros((11,) + tuple(G.proj_shape[1:]), device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            G.forward(v, out=out, angle_begin=5, angle_count=11)
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, full[5:16])
        # after a call outside a capture (an unsorted range then has its table)
        assert torch.equal(G.forward(v, angle_begin=5, angle_count=11), full[5:16])


@pytest.mark.parametrize("order", ["sorted", "descending"])
def test_sorted_ranges_allocate_nothing(tigre, order):
    gc.collect()  # handles left to the garbage collector by earlier tests
    count = [0]

    def alloc(nbytes, stream):
        count[0] += 1
        return torch.cuda.caching_allocator_alloc(nbytes, device=torch.cuda.current_device(),
                                                  stream=stream)

    tigre.tigre_set_allocator(alloc, lambda p, s: torch.cuda.caching_allocator_delete(p))
    try:
        with tigre.Geometry(geometry(), ANGLES[order]) as G:
            v = torch.from_numpy(synth.random_volume(G.vol_shape, seed=4)).cuda()
            full = G.forward(v)
            before = count[0]
            for a0, n in ((0, 9), (5, 11), (13, 11), (1, 23), (2, 12)):
                assert torch.equal(G.forward(v, angle_begin=a0, angle_count=n), full[a0:a0 + n])
            assert count[0] == before
    finally:
        torch.cuda.synchronize()
        tigre.tigre_set_allocator(None, None)
