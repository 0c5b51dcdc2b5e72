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


@pytest.mark.parametrize("exponent", [-30, 31, 36, 38])
def test_force_scales_with_the_unit_of_length(env, exponent):
    # the same box in units 2^-exponent as long (grid spacings of 8e-10 to 2e11): the acceleration is
    # m / length^2, and every step of the solve scales by a power of two.  Densities below 2^-126, which a
    # transform may take for zero, are at most 2^-12 of the mean at the largest spacing: the bar of every force
    # comparison covers them.
    torch, hacc = env
    ng, L = 24, 20.0
    _, p = _box(torch, 4000, L, 7)
    q = p.clone()
    q[:, :3] *= 2.0 ** exponent
    ctx = hacc.Context()
    try:
        a = ctx.pm_force(hacc.Box(L=L, ng=ng), hacc.PM(), p).double()
        b = ctx.pm_force(hacc.Box(L=L * 2.0 ** exponent, ng=ng), hacc.PM(), q).double() * 4.0 ** exponent
    finally:
        ctx.close()
    rms = (a ** 2).sum(1).mean().sqrt()
    assert float((b - a).abs().max() / rms) <= 1e-4


@pytest.mark.parametrize("ng", [256, 258])
def test_grids_at_the_bound_of_the_batched_transforms(env, ng):
    torch, hacc = env
    L = 64.0
    pos, p = _box(torch, 3000, L, ng)
    ctx = hacc.Context()
    try:
        a = ctx.pm_force(hacc.Box(L=L, ng=ng), hacc.PM(), p).cpu().numpy()
    finally:
        ctx.close()
    ref = opm.pm_accel(pos[:, :3].astype(np.float64), pos[:, 3].astype(np.float64), L, ng)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    assert np.abs(a[:, :3] - ref).max() / rms <= 1e-4


def test_large_grids_keep_the_work_area_of_one_transform(env):
    # 514 = 2 x 257: transforms of such sides need a work area, about their own data each.  What the context
    # holds is its grids (28 bytes a point and 32 a mode) and at most one transform's data for either direction,
    # with a quarter to spare; three components at once would take half as much again as that in the inverse alone
    torch, hacc = env
    ng, L = 514, 128.0
    _, p = _box(torch, 3000, L, 5)
    mode_bytes = 8 * ng * ng * (ng // 2 + 1)
    ctx = hacc.Context()
    try:
        ctx.pm_force(hacc.Box(L=L, ng=16), hacc.PM(), p)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        ctx.pm_force(hacc.Box(L=L, ng=ng), hacc.PM(), p, acc=torch.empty_like(p))
        torch.cuda.synchronize()
        held = free - torch.cuda.mem_get_info()[0]
    finally:
        ctx.close()
    assert held <= 28 * ng ** 3 + 4 * mode_bytes + 2.5 * mode_bytes
