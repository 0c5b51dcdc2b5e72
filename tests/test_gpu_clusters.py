"""GPU parity of the pair kernel at the edges of its clusters and items: cells
holding one particle fewer, as many and one more than a cluster (8), a half
warp, a warp and an item (64) hold, in meshes so small that every cell lies at
a periodic face, against the FP64 oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# 27-cell sums of FP32 pair terms: the bar of every force comparison
FORCE_TOL = 1e-4
COUNTS = (1, 7, 8, 9, 15, 16, 17, 31, 33, 63, 64, 65, 71, 129, 200, 520)


@pytest.mark.parametrize("nc", [3, 4, 5])
@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("cap", [-1, 0, 16, 160])
def test_cell_counts_around_cluster_and_item_sizes(split_params, nc, masses, cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    sp = dict(split_params)
    sp["r_cut"] = float(np.float32(sp["r_cut"]))
    sp["eps"] = float(np.float32(sp["eps"]))
    L = float(np.float32(nc * 3.2))
    rng = np.random.default_rng(10 * nc + masses)
    w = L / nc
    rows = []
    for c in range(nc ** 3):
        cell = np.array([c % nc, (c // nc) % nc, c // nc ** 2])
        n = COUNTS[c % len(COUNTS)] if c < 2 * len(COUNTS) else int(rng.integers(0, 24))
        rows.append((cell + rng.uniform(0.001, 0.999, (n, 3))) * w)
    x = np.concatenate(rows)
    pos = np.ones((len(x), 4), np.float32)
    pos[:, :3] = x
    if masses:
        pos[:, 3] = rng.uniform(0.25, 4.0, len(x))
    pos = pos[rng.permutation(len(pos))]
    ref, within = oracle.force_mesh(pos, L, sp)
    ctx = hacc.Context()
    try:
        ctx.set_item_cap(cap)
        p = torch.from_numpy(pos).cuda()
        box = hacc.Box(L=L, nc=nc)
        a = ctx.sr_force(box, sp, p).cpu().numpy()
        cand, got = ctx.pair_counts(box, sp, p)
    finally:
        ctx.close()
    rms = np.sqrt((ref ** 2).sum(1).mean())
    assert np.abs(a[:, :3] - ref).max() / rms <= FORCE_TOL
    assert abs(got - within) <= max(2, within // 200000) and got <= cand


@pytest.mark.parametrize("nc", [3, 40])
def test_wide_cells_are_ordered(split_params, nc):
    # cells at the bounds of the ordering's paths for cells above 256 particles, alone in their block of cells
    # and crowded together (more keys than a block stages), in a mesh of few and of many cells
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    rc = np.float32(split_params["r_cut"])
    L = float(np.float32(nc * 3.2))
    rng = np.random.default_rng(nc)
    rows = []
    for c, n in {0: 256, 1: 257, 2: 512, 3: 513, 4: 2047, 5: 2048, 6: 2049, 9: 300, nc ** 3 - 1: 900}.items():
        cell = np.array([c % nc, (c // nc) % nc, c // nc ** 2])
        rows.append((cell + rng.uniform(0.001, 0.999, (n, 3))) * (L / nc))
    x = np.concatenate(rows)
    pos = np.ones((len(x), 4), np.float32)
    pos[:, :3] = x
    pos = pos[rng.permutation(len(pos))]
    ctx = hacc.Context()
    try:
        p = torch.from_numpy(pos.copy()).cuda()
        cell, start, perm = (t.cpu().numpy() for t in ctx.bin(hacc.Box(L=L, nc=nc), rc, p))
    finally:
        ctx.close()
    _, cell_o, ok = oracle.wrap_cell(pos, L, nc)
    _, start_o, perm_o = oracle.bin_cells(cell_o, nc)
    assert ok and np.array_equal(cell, cell_o) and np.array_equal(start, start_o) and np.array_equal(perm, perm_o)
