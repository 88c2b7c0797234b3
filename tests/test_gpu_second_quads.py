"""Ranges for which the quad kernel is the faster one need a second set of quads.
Where it does not fit, or is missing inside a stream capture, the column kernel
takes the call: the same bits."""
import gc

import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu

def handle(tigre, na=100):
    """100 (50) angles of 60 rows take columns and one set of quads, the first 20 of
    them do not, and read both sets; 100 angles are paired, 50 are not."""
    geo = synth.geometry((200, 190, 60), 0.5, (240, 60), (0.85, 0.72), dso=400.0, dsd=600.0)
    return tigre.Geometry(geo, synth.angles(na, first=0.1))


def volume(G):
    return torch.from_numpy(synth.random_volume(G.vol_shape, seed=8)).cuda()


@pytest.mark.parametrize("na", [50, 100])
def test_capture_without_the_second_set(tigre, na):
    with handle(tigre, na) as G:
        v = volume(G)
        n0 = tigre.tigre_launch_count()
        full = G.forward(v)
        assert tigre.tigre_launch_count() - n0 == 2  # columns
        out = torch.zeros((20,) + tuple(G.proj_shape[1:]), device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            G.forward(v, out=out, angle_begin=0, angle_count=20)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, full[:20])
        n0 = tigre.tigre_launch_count()
        assert torch.equal(G.forward(v, angle_begin=0, angle_count=20), full[:20])
        assert tigre.tigre_launch_count() - n0 == 3  # two sets and the quad kernel
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, full[:20])


def test_memory_for_one_set_only(tigre):
    gc.collect()  # handles left to the garbage collector by earlier tests
    quads = 16 * 204 * 194 * 64
    live, limit = {}, [1]

    def alloc(nbytes, stream):
        if nbytes >= quads and sum(n >= quads for n in live.values()) >= limit[0]:
            return 0
        p = torch.cuda.caching_allocator_alloc(nbytes, device=torch.cuda.current_device(),
                                               stream=stream)
        live[p] = nbytes
        return p

    def free(ptr, stream):
        live.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    tigre.tigre_set_allocator(alloc, free)
    try:
        with handle(tigre) as G:
            v = volume(G)
            counts, parts = [], []
            for limit[0] in (1, 1, 2):
                n0 = tigre.tigre_launch_count()
                parts.append(G.forward(v, angle_begin=0, angle_count=20))
                counts.append(tigre.tigre_launch_count() - n0)
            full = G.forward(v)
        assert counts == [2, 2, 3]
        assert all(torch.equal(p, full[:20]) for p in parts)
        assert not live
    finally:
        torch.cuda.synchronize()
        tigre.tigre_set_allocator(None, None)
