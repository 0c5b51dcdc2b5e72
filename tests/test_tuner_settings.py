"""The autotuners' settings: the default is among them, no two are the same, and
what they keep is that setting in every later call."""
import os
import re

import numpy as np
import pytest

import paper_1410_2805_gb300 as hacc

ITEM_MAX = 64   # larger caps mean this one (hacc_set_item_cap)
HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "hacc.h")


@pytest.mark.parametrize("name,caps,settings", [("HACC_TUNE_CAPS", hacc.TUNE_CAPS, hacc.TUNE_SETTINGS),
                                                ("HACC_BATCH_TUNE_CAPS", hacc.BATCH_TUNE_CAPS,
                                                 hacc.BATCH_TUNE_SETTINGS)])
def test_caps_hold_the_default_and_differ(name, caps, settings):
    assert -1 in caps and ITEM_MAX in caps
    assert len({min(c, ITEM_MAX) for c in caps}) == len(caps)
    assert settings == len(caps) * 2 * hacc.FORCE_VARIANTS
    declared = re.search(r"#define %s \{([^}]*)\}" % name, open(HEADER).read())
    assert declared and tuple(int(c) for c in declared.group(1).split(",")) == caps


@pytest.mark.gpu
@pytest.mark.parametrize("n", [4099, 65536, 65537])
def test_tuned_calls_are_those_of_the_setting(split_params, n):
    # on both sides of the largest box whose items a block shares with the default cap
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth
    L = float(np.float32(n ** (1 / 3)))
    p = torch.from_numpy(synth.blob_mixture_scaled(n, L, seed=n)).cuda()
    box = hacc.Box(L=L)
    ctx, ref = hacc.Context(), hacc.Context()
    try:
        res = ctx.tune(box, split_params, p, reps=2)
        assert res["chosen"] == int(np.argmin(res["times_ms"]))
        ref.set_item_cap(res["item_cap"])
        ref.set_variant(res["variant"])
        ref.set_queue_order(res["heavy_first"])
        a, b = (c.sr_force(box, split_params, p).clone() for c in (ctx, ref))
        assert torch.equal(a, b)
    finally:
        ctx.close()
        ref.close()
