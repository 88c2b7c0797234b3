"""FDK from two host threads, each with its own handle and stream and its own
row length: both lengths run the same filter instance, whose shared-memory limit
belongs to the process, so a call on short rows must not lower it under a
launch on long ones."""
import threading

import numpy as np
import pytest
import torch

from paper_1905_03748_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [(2048, 1400), (8192, 2800), (12400, 16000)])
def test_two_threads_with_different_row_lengths(tigre, lengths):
    calls, errors, out = 300, [], {}

    def work(nu, G, y, x, stream):
        try:
            for _ in range(calls):
                tigre.tigre_fdk(G.handle, y, x, stream=stream.cuda_stream)
            stream.synchronize()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    jobs = []
    for nu in lengths:
        geo = synth.geometry((12, 10, 4), 1.0, (nu, 2), (25.0 / nu, 4.0), dso=200.0, dsd=300.0)
        G = tigre.Geometry(geo, synth.angles(2))
        y = torch.from_numpy(np.random.default_rng(nu).random((2, 2, nu)).astype(np.float32)).cuda()
        out[nu] = (G.fdk(y), torch.empty(G.vol_shape, device="cuda"))
        jobs.append((nu, G, y, out[nu][1], torch.cuda.Stream()))
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for _, G, *_ in jobs:
        G.close()
    assert not errors, errors
    for nu in lengths:
        assert torch.equal(*out[nu])
