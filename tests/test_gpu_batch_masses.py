"""Batches that mix boxes of equal masses with boxes whose masses differ: each
box bit for bit as it is alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _boxes(rng):
    """(n, L, masses) of each box: shared and whole items, equal masses of one value and of another, masses that
    differ everywhere or in the last particle alone; more boxes than a word has bits."""
    out = [(5003, 17.0, "one"), (70001, 41.0, "one"), (5003, 17.0, "all"), (70001, 41.0, "last"), (9001, 21.0, "2.5")]
    return out + [(100 + 7 * k, 10.0, ("one", "all")[k % 2]) for k in range(38)] + [(5003, 17.0, "last")]


@pytest.mark.parametrize("use_graph", [False, True])
def test_boxes_alone_and_among_other_masses(split_params, use_graph):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1410_2805_gb300 as hacc
    rng = np.random.default_rng(7)
    specs, rows, boxes, off = _boxes(rng), [], [], 0
    for n, L, masses in specs:
        p = np.ones((n, 4), np.float32)
        p[:, :3] = rng.uniform(0.0, L, (n, 3))
        if masses == "all":
            p[:, 3] = rng.uniform(0.25, 4.0, n)
        elif masses == "last":
            p[-1, 3] = 1.5
        elif masses != "one":
            p[:, 3] = float(masses)
        rows.append(p)
        boxes.append((off, n, L))
        off += n
    pos = np.concatenate(rows)
    vel = np.zeros_like(pos)
    vel[:, :3] = rng.normal(0.0, 0.1, (off, 3))
    stream = torch.cuda.Stream()
    ctx = hacc.Context()

    def run(which):
        P, V = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(vel.copy()).cuda()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            ctx.batch_subcycle(split_params, [hacc.BatchBox(L=L, offset=o, n=n, dt=0.002) for o, n, L in which], P, V,
                               n_sub=2, use_graph=use_graph)
        ctx.sync(stream)
        return P, V

    try:
        P, V = run(boxes)
        for b in (0, 1, 2, 3, 4, 5, 6, len(boxes) - 1):
            o, n, _ = boxes[b]
            P1, V1 = run([boxes[b]])
            assert torch.equal(P1[o:o + n], P[o:o + n]) and torch.equal(V1[o:o + n], V[o:o + n]), specs[b]
    finally:
        ctx.close()
