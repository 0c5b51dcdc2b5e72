"""Sub-cycles and full steps of a box with a massive halo: cells of thousands of
particles side by side, which the in-cell ordering treats apart."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

NC, L = 12, float(np.float32(12 * 3.2))


def halo_box(counts, n, seed):
    """n particles: counts[c] in cell c, the rest uniform; every mass is another FP32 value."""
    rng = np.random.default_rng(seed)
    rows = []
    for c, k in counts.items():
        cell = np.array([c % NC, (c // NC) % NC, c // NC ** 2])
        rows.append((cell + rng.uniform(0.02, 0.98, (k, 3))) * (L / NC))
    left = n - sum(counts.values())
    rows.append(rng.uniform(0.0, L, (left, 3)))
    pos = np.ones((n, 4), np.float32)
    pos[:, :3] = np.concatenate(rows)
    pos[:, 3] = 0.5 + np.arange(n) / np.float32(1 << 20)
    pos[:, 3] = rng.permutation(pos[:, 3])
    assert len(np.unique(pos[:, 3])) == n
    pos = pos[rng.permutation(n)]
    vel = np.zeros_like(pos)
    vel[:, :3] = rng.normal(0.0, 0.1, (n, 3))
    return pos, vel


# (a cell of up to about 4000 particles, one that a ranking by runs of rows cannot take): neighbours in x, far
# apart in one block of cells, and in the other order; on both sides of the largest call whose blocks sort every cell
@pytest.mark.parametrize("counts,n", [({0: 3000, 1: 20000}, 100001), ({0: 12000, 7: 2049, 3: 2048}, 65537),
                                      ({8: 2300, 9: 9000, 10: 2300}, 80000),
                                      ({0: 2049, 1: 12000, 2: 2048, 3: 2500}, 65536)])
@pytest.mark.parametrize("call", ["subcycle", "step"])
def test_neighbouring_dense_cells_keep_their_rows(split_params, counts, n, call):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    # softened so that a sub-cycle is short against every close encounter
    sp = dict(split_params, eps=float(np.float32(0.04)))
    sp["r_cut"] = float(np.float32(sp["r_cut"]))
    pos, vel = halo_box(counts, n, seed=n)
    dt = 3e-4
    ctx = hacc.Context()
    try:
        p, v = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(vel.copy()).cuda()
        box = hacc.Box(L=L, nc=NC)
        if call == "subcycle":
            xo, vo = oracle.subcycle(pos, vel, L, sp, dt, 3)
            ctx.subcycle(box, sp, p, v, dt, 3)
        else:
            xo, vo = oracle.step(pos, vel, L, sp, dt, 3)
            ctx.step(box, sp, hacc.PM(), p, v, dt, 3)
        ctx.sync()
        p, v = p.cpu().numpy(), v.cpu().numpy()
    finally:
        ctx.close()
    # every row is its own particle's still, and where the oracle has it
    assert np.array_equal(p[:, 3], pos[:, 3])
    d = p[:, :3].astype(np.float64) - xo
    d -= L * np.round(d / L)
    assert np.abs(d).max() < 2e-5 * L
    assert np.abs(v[:, :3] - vo).max() < 1e-3 * np.sqrt((vo ** 2).sum(1).mean())


# cells above the 2048 keys that a block ranks by buckets: all of a call's particles in one cell, several such cells
# in one block of cells, with smaller ones between them; input in random order and in cell order
@pytest.mark.parametrize("counts,n", [({0: 65536}, 65536), ({0: 65537}, 65537), ({5: 2049}, 2049),
                                      ({0: 2049, 1: 2048, 2: 30000, 3: 1, 4: 2050, NC ** 3 - 1: 9000}, 50000)])
@pytest.mark.parametrize("ordered", [False, True])
def test_big_cells_are_ordered_by_row(split_params, counts, n, ordered):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    pos, _ = halo_box(counts, n, seed=n)
    _, cell_o, ok = oracle.wrap_cell(pos, L, NC)
    assert ok
    if ordered:
        order = np.argsort(cell_o, kind="stable")
        pos, cell_o = pos[order], cell_o[order]
    _, start_o, perm_o = oracle.bin_cells(cell_o, NC)
    ctx = hacc.Context()
    try:
        p = torch.from_numpy(pos.copy()).cuda()
        cell, start, perm = (t.cpu().numpy() for t in ctx.bin(hacc.Box(L=L, nc=NC), np.float32(split_params["r_cut"]), p))
    finally:
        ctx.close()
    assert np.array_equal(cell, cell_o) and np.array_equal(start, start_o) and np.array_equal(perm, perm_o)
