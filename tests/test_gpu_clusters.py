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


@pytest.mark.parametrize("n", [200, 8192, 8193, 12288, 12289, 65536, 65537, 90001])
def test_shared_items_sum_as_in_a_batch(split_params, n):
    # sizes at the bounds of the item caps and of the sharing of items by a block: a box's forces are those of
    # the oracle, its trajectory in a batch is bit for bit the same alone and next to another box, and one
    # sub-cycle is that of the box in a call of its own (later ones order equal sub-cells differently: by the
    # row of the pool, and by the place in the previous sub-cycle)
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    import synth
    sp = dict(split_params)
    sp["r_cut"], sp["eps"] = float(np.float32(sp["r_cut"])), float(np.float32(sp["eps"]))
    L = float(np.float32(max(10.0, n ** (1 / 3))))
    pos = synth.blob_mixture_scaled(n, L, seed=n) if n > 512 else synth.blob_mixture(n, L, seed=n)
    rng = np.random.default_rng(n)
    vel = np.zeros_like(pos)
    vel[:, :3] = rng.normal(0.0, 0.1, (n, 3))
    ctx = hacc.Context()
    try:
        p = torch.from_numpy(pos).cuda()
        a = ctx.sr_force(hacc.Box(L=L), sp, p).cpu().numpy()
        runs = []
        for m in (0, 300, 70000):   # the batch's other box: none, one that is shared, one that is not
            q = np.concatenate([pos, pos[:1].repeat(m, 0)])
            q[n:, :3] = rng.uniform(0.0, 40.0, (m, 3))
            P = torch.from_numpy(q).cuda()
            V = torch.from_numpy(np.concatenate([vel, np.zeros((m, 4), np.float32)])).cuda()
            boxes = [hacc.BatchBox(L=L, offset=0, n=n, dt=0.02)]
            if m:
                boxes.append(hacc.BatchBox(L=41.0, offset=n, n=m, dt=0.02))
            ctx.batch_subcycle(sp, boxes, P, V, n_sub=2)
            runs.append((P[:n].clone(), V[:n].clone()))
        one = [torch.from_numpy(x).cuda() for x in (pos, vel, pos, vel)]
        ctx.batch_subcycle(sp, [hacc.BatchBox(L=L, offset=0, n=n, dt=0.02)], one[0], one[1], n_sub=1)
        ctx.subcycle(hacc.Box(L=L), sp, one[2], one[3], 0.02, 1)
        ctx.sync()
    finally:
        ctx.close()
    for P, V in runs[1:]:
        assert torch.equal(P, runs[0][0]) and torch.equal(V, runs[0][1])
    assert torch.equal(one[0], one[2]) and torch.equal(one[1], one[3])
    ref, _ = oracle.force_mesh(pos, L, sp)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    assert np.abs(a[:, :3] - ref).max() / rms <= FORCE_TOL
