"""The pair potential at the edges of its loops: boxes whose clusters meet every
remainder of a step and of a list, crowded and sparse, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [None, 0.0])
@pytest.mark.parametrize("cap", [-1, 0, 64])
def test_batch_of_boxes_of_every_small_size(split_params, eps, cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    sp = dict(split_params)
    if eps is not None:
        sp["eps"] = eps
    sp["r_cut"], sp["eps"] = float(np.float32(sp["r_cut"])), float(np.float32(sp["eps"]))
    rng = np.random.default_rng(5)
    rows, boxes, off = [], [], 0
    sizes = list(range(1, 150)) + [191, 192, 193, 383, 384, 385, 449, 520, 1100]
    for k, n in enumerate(sizes):
        L = (10.0, 13.0, 16.5)[k % 3]   # 3, 4 and 5 cells a side
        p = np.ones((n, 4), np.float32)
        p[:, :3] = rng.uniform(0.0, L, (n, 3)) if k % 2 else L - 2.5 + rng.uniform(0.0, 2.4, (n, 3))
        p[:, 3] = rng.uniform(0.25, 4.0, n)
        rows.append(p)
        boxes.append((off, n, L))
        off += n
    pos = np.concatenate(rows)
    ctx = hacc.Context()
    try:
        ctx.set_item_cap(cap)
        P = torch.from_numpy(pos).cuda()
        batch = [hacc.BatchBox(L=L, offset=o, n=n, dt=0.0) for o, n, L in boxes]
        got = ctx.batch_diagnostics(sp, batch, P, torch.zeros_like(P)).cpu().numpy()[:, 4]
    finally:
        ctx.close()
    for (o, n, L), pe in zip(boxes, got):
        x = pos[o:o + n].astype(np.float64)
        _, _, ref = oracle.diagnostics(x[:, :3], 0 * x[:, :3], x[:, 3], L, sp)
        # a pair's term is a difference of quantities of up to 3 from some ten FP32 operations (2e-6), its
        # root good to 2^-22 (and close pairs are only that), times two masses of up to 4
        assert abs(pe - ref) <= 2e-6 * 16 * n * (n - 1) / 2 + 1e-6 * abs(ref), (n, L)
