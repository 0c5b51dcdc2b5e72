"""Boxes in which a few cells hold most of the work, cut into smaller items than
the others: forces against the oracle, and trajectories alone and in a batch."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

NC, L = 40, float(np.float32(40 * 3.2))
N = (1 << 20) + 4099   # a size whose cells take items of 64


@pytest.mark.parametrize("counts", [{0: 2049, 41: 2048}, {820: 6000, 821: 2113, NC ** 3 - 1: 2500}])
def test_dense_cells_of_a_large_box(split_params, counts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    sp = dict(split_params)
    sp["r_cut"], sp["eps"] = float(np.float32(sp["r_cut"])), float(np.float32(0.04))
    rng = np.random.default_rng(len(counts))
    rows, sel = [], []
    for c, k in counts.items():
        cell = np.array([c % NC, (c // NC) % NC, c // NC ** 2])
        rows.append((cell + rng.uniform(0.01, 0.99, (k, 3))) * (L / NC))
    x = np.concatenate(rows + [rng.uniform(0.0, L, (N - sum(counts.values()), 3))])
    pos = np.ones((N, 4), np.float32)
    pos[:, :3] = np.minimum(x.astype(np.float32), np.nextafter(np.float32(L), np.float32(0)))
    sel = np.concatenate([np.arange(sum(counts.values())), rng.integers(0, N, 2000)])
    ref, _ = oracle.force_mesh(pos, L, sp, sel=sel)
    ctx = hacc.Context()
    try:
        p = torch.from_numpy(pos).cuda()
        a = ctx.sr_force(hacc.Box(L=L, nc=NC), sp, p).cpu().numpy()
        other = torch.rand(30011, 4, device="cuda") * 40.0
        other[:, 3] = 1.0
        runs = []
        for q in (p, torch.cat([p, other])):
            P, V = q.clone(), torch.zeros_like(q)
            boxes = [hacc.BatchBox(L=L, offset=0, n=N, dt=1e-3, nc=NC)]
            if len(q) > N:
                boxes.append(hacc.BatchBox(L=41.0, offset=N, n=len(q) - N, dt=1e-3))
            ctx.batch_subcycle(sp, boxes, P, V, n_sub=2)
            runs.append((P[:N].clone(), V[:N].clone()))
        ctx.sync()
    finally:
        ctx.close()
    rms = np.sqrt((ref ** 2).sum(1).mean())
    assert np.abs(a[sel, :3] - ref).max() / rms <= 1e-4
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][1], runs[1][1])
