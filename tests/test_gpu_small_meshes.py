"""Meshes in which a cell's neighbours reach past the middle of the box: the
separation of a pair carries the rounding of one subtraction there too."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

FORCE_TOL = 1e-4   # the bar of every force comparison
# (cells per cutoff, box side): 3 and 4 cells of a cutoff; 5, 6, 7 and 8 of half of one
MESHES = [(1, 9.5), (1, 10.0), (1, 12.25), (1, 13.0), (2, 8.0), (2, 10.0), (2, 11.25), (2, 12.75)]


def _mesh_cells(hacc, R, L, rc):
    return hacc.mesh_cells(L, rc) if R == 1 else hacc.mesh_cells(L, np.float32(rc) / 2)


@pytest.mark.parametrize("R,L", MESHES)
@pytest.mark.parametrize("cap", [-1, 64])
def test_pairs_are_antisymmetric_to_the_last_bit(split_params, R, L, cap):
    # with the separation rounded once, the terms of i and of j differ in sign alone, wherever the pair lies
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    rc = np.float32(split_params["r_cut"])
    assert _mesh_cells(hacc, R, L, rc) == {(1, 9.5): 3, (1, 10.0): 3, (1, 12.25): 3, (1, 13.0): 4, (2, 8.0): 5,
                                           (2, 10.0): 6, (2, 11.25): 7, (2, 12.75): 8}[R, L]
    rng = np.random.default_rng(int(100 * L) + R)
    m = 200
    d = rng.normal(size=(m, 3))
    d *= (rng.uniform(0.02, 0.99, m) * rc / np.sqrt((d ** 2).sum(1)))[:, None]
    a = rng.uniform(0.0, L, (m, 3))
    low = rng.random((m, 3)) < 0.5   # next to the middle, on the side where x - L is inexact
    a[low] = rng.uniform(0.3 * L, 0.5 * L, low.sum())
    pos = np.ones((m, 2, 4), np.float32)
    pos[:, 0, :3] = a
    pos[:, 1, :3] = np.remainder(a + np.where(low, np.abs(d), d), L)
    pos[pos == np.float32(L)] = 0.0
    rows = torch.from_numpy(pos).cuda()
    ctx = hacc.Context()
    try:
        ctx.set_stencil(R)
        ctx.set_item_cap(cap)
        acc = torch.stack([ctx.sr_force(hacc.Box(L=L), split_params, rows[k]) for k in range(m)]).cpu().numpy()
    finally:
        ctx.close()
    f = acc[:, :, :3]
    assert (f[:, 0] != 0).any(1).all()
    bad = (f[:, 0] != -f[:, 1]).any(1)
    assert not bad.any(), (int(bad.sum()), pos[bad][0], f[bad][0])


@pytest.mark.parametrize("R,L", MESHES)
@pytest.mark.parametrize("cap", [-1, 0, 64])
def test_small_meshes_against_the_oracle(split_params, R, L, cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    sp = dict(split_params)
    sp["r_cut"], sp["eps"] = float(np.float32(sp["r_cut"])), float(np.float32(sp["eps"]))
    rng = np.random.default_rng(int(100 * L) + R)
    n = 3000
    pos = np.ones((n, 4), np.float32)
    pos[:, :3] = rng.uniform(0.0, L, (n, 3))
    pos[pos == np.float32(L)] = 0.0
    vel = np.zeros_like(pos)
    ref, within = (oracle.force_mesh if L >= 9.5 else oracle.force_brute)(pos, L, sp)
    _, _, pe = oracle.diagnostics(pos[:, :3].astype(np.float64), vel[:, :3].astype(np.float64),
                                  pos[:, 3].astype(np.float64), L, sp)
    ctx = hacc.Context()
    try:
        ctx.set_stencil(R)
        ctx.set_item_cap(cap)
        box, p = hacc.Box(L=L), torch.from_numpy(pos).cuda()
        a = ctx.sr_force(box, split_params, p).cpu().numpy()
        cand, got = ctx.pair_counts(box, split_params, p)
        out = ctx.diagnostics(box, split_params, p, torch.from_numpy(vel).cuda()).cpu().numpy()
        P, V = torch.from_numpy(pos).cuda(), torch.from_numpy(vel).cuda()
        h = 2.0 ** -12
        if R == 1:   # a tick of zero velocities is a kick by the forces of the same sums
            flags = hacc.TICK_FIRST | hacc.TICK_LAST
            ctx.batch_tick(split_params, [hacc.BatchBox(L=L, offset=0, n=n, dt=h, flags=flags)], P, V)
        ctx.sync()
    finally:
        ctx.close()
    rms = np.sqrt((ref ** 2).sum(1).mean())
    assert np.abs(a[:, :3] - ref).max() / rms <= FORCE_TOL
    assert abs(got - within) <= max(2, within // 200000) and got <= cand
    assert out[4] == pytest.approx(pe, rel=1e-4)
    if R == 1:
        assert np.array_equal(V.cpu().numpy()[:, :3], np.float32(h) * a[:, :3])
