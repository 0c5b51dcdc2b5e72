"""The scratch of a batched pass, which the server's admission and a context's
budget count: no more than a budget that was enough for it has held."""
import pytest

import paper_1410_2805_gb300 as hacc


@pytest.mark.parametrize("n,L,boxes,enough", [(16777216, 256.0, 1, 1399911424), (2097152, 128.0, 1, 174990848),
                                              (8192, 20.0, 1, 684544), (4097, 16.0, 200, 68317504),
                                              (100, 10.0, 33, 309280), (1, 10.0, 700, 780256)])
def test_batch_scratch_fits_where_it_has(n, L, boxes, enough):
    from paper_1410_2805_gb300 import build
    build.build()
    batch = [hacc.BatchBox(L=L, offset=n * b, n=n, dt=0.01) for b in range(boxes)]
    assert 0 < hacc.batch_scratch_bytes(hacc.default_split(), batch) <= enough
