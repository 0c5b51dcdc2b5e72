"""What the long-range stage keeps between calls: a call does not depend on the
calls and the graph replays before it."""
import numpy as np
import pytest

import synth
from oracle import pm as opm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    return torch, hacc


def _box(torch, n, L, seed):
    pos = synth.blob_mixture(n, L, seed=seed)
    return pos, torch.from_numpy(pos).cuda()


def test_replays_of_another_side_leave_a_call_alone(env):
    # one grid size, two box sides: a call after the other side's replay gives the bits it gave before, and the
    # replay those of its own side
    torch, hacc = env
    ng, sides = 32, (32.0, 20.0)
    pos = [_box(torch, 5000, L, k) for k, L in enumerate(sides)]
    box = [hacc.Box(L=L, ng=ng) for L in sides]
    stream = torch.cuda.Stream()
    ctx = hacc.Context()
    try:
        with torch.cuda.stream(stream):
            alone = [ctx.pm_force(box[k], hacc.PM(), pos[k][1], stream=stream).clone() for k in (0, 1)]
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                out = ctx.pm_force(box[0], hacc.PM(), pos[0][1], stream=stream)
            for _ in range(2):
                second = ctx.pm_force(box[1], hacc.PM(), pos[1][1], stream=stream).clone()
                graph.replay()
                replayed = out.clone()
                after = ctx.pm_force(box[1], hacc.PM(), pos[1][1], stream=stream).clone()
                stream.synchronize()
                assert torch.equal(second, alone[1]) and torch.equal(after, alone[1])
                assert torch.equal(replayed, alone[0])
    finally:
        ctx.close()
    for k, L in enumerate(sides):
        ref = opm.pm_accel(pos[k][0][:, :3].astype(np.float64), pos[k][0][:, 3].astype(np.float64), L, ng)
        rms = np.sqrt((ref ** 2).sum(1).mean())
        assert np.abs(alone[k].cpu().numpy()[:, :3] - ref).max() / rms <= 1e-4
