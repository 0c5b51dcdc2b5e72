"""Cells hundreds of thousands of cutoffs wide: pairs just inside the cutoff, across a
cell's face, are kept by the selection of a cluster's neighbours."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("side", [2.0 ** 18, 2.0 ** 21, 2.0 ** 22])
def test_pairs_at_the_cutoff_in_cells_far_wider_than_it(split_params, axis, side):
    import torch
    from scipy.spatial import cKDTree
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    sp = dict(split_params, r_cut=float(np.float32(3.0005)))   # pairs at 3: 0.99983 of it
    rng = np.random.default_rng(axis + int(side))
    face = int(side / 3)   # integers, exact in FP32: the last before the face of cell 1
    m, n = 800, 9000
    x = np.floor(rng.uniform(0.0, side, (n, 3)))   # 330 particles a cell: clusters of a sub-cell or two each
    base = np.floor(rng.uniform(0.0, side, (m, 3)))
    base[:, axis] = face
    mate = base.copy()
    mate[:, axis] = face + 3
    x = np.concatenate([x, base, mate])
    pos = np.ones((len(x), 4), np.float32)
    pos[:, :3] = x
    pos = pos[rng.permutation(len(pos))]
    tree = cKDTree(pos[:, :3].astype(np.float64), boxsize=side)
    want = 2 * len(tree.query_pairs(sp["r_cut"]))
    ctx = hacc.Context()
    try:
        p = torch.from_numpy(pos).cuda()
        box = hacc.Box(L=side, nc=3)
        ctx.set_item_cap(64)
        a = ctx.sr_force(box, sp, p).clone()
        cand, within = ctx.pair_counts(box, sp, p)
        ctx.set_item_cap(-1)
        b = ctx.sr_force(box, sp, p).clone()
        assert ctx.pair_counts(box, sp, p) == (cand, within)
    finally:
        ctx.close()
    assert want >= 2 * m and within == want
    # nearly every particle has one partner or none: the force is that pair's, in any order
    alone = np.array([len(q) for q in tree.query_ball_point(pos[:, :3].astype(np.float64), sp["r_cut"])]) == 2
    a, b = a.cpu().numpy(), b.cpu().numpy()
    assert alone.sum() > m and (a[alone, axis] != 0).any() and np.array_equal(a[alone], b[alone])
