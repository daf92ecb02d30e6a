"""Forward of first layers whose windows are read out of whole input rows, at the edges of its tiles, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import eoq, synth
import gpu_util as G

pytestmark = pytest.mark.gpu

CASES = [
    # (geometry, margin): output widths of one tile of 125 pixels, of two unequal ones, of one pixel; rows that end inside a patch
    (oracle.ConvDesc(1, 9, 250, 8, 64, 7, 7, 2, 3), 5),
    (oracle.ConvDesc(2, 21, 252, 8, 16, 7, 7, 2, 3), 5),
    (oracle.ConvDesc(1, 7, 510, 8, 128, 7, 7, 2, 3), 7),
    (oracle.ConvDesc(3, 38, 6, 8, 48, 5, 5, 2, 0), 4),
    (oracle.ConvDesc(40, 29, 30, 8, 32, 7, 7, 2, 3), 5),
    (oracle.ConvDesc(2, 13, 121, 16, 80, 5, 5, 1, 2), 5),
    (oracle.ConvDesc(1, 11, 122, 16, 112, 8, 8, 1, 3), 6),
]


@pytest.mark.parametrize("d,m", CASES, ids=lambda v: "" if isinstance(v, int) else "n%d_%dx%d_%d_%d_k%d" % (v.n, v.h, v.w, v.c_in, v.c_out, v.kh))
def test_windows_out_of_input_rows(d, m):
    x0, w = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2800, d.w), synth.normal_codes((d.c_out, d.kh, d.kw, d.c_in), 2801, d.c_out, std_codes=9)
    gd = eoq.conv_desc(d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.kw, d.stride, d.pad, m)
    assert "kernel=igemm_input_rows" in eoq.eoq_describe_plan(G.handle(), gd, eoq.EOQ_PASS_FWD)
    xm = G.dev(np.pad(x0, ((0, 0), (0, 0), (m, m), (0, 0))))
    out = (d.n, d.ho, d.wo, d.c_out)
    shortcut = synth.int8_uniform(out, 2802, d.h)
    for b1, gamma, relu, sc in ((0, 128, True, None), (-3, 90, False, shortcut)):
        ref = oracle.layer_forward(d, x0, b1, w, gamma, 2, sc, relu)
        x5, x2, mask = G.zeros(out, torch.int8), G.zeros(out, torch.int16), G.zeros((ref["x5"].size + 7) // 8, torch.uint8)
        keep = sc is not None
        eoq.eoq_conv_fwd(G.handle(), gd, xm, None, b1, G.dev(w), gamma, 2, None if sc is None else G.dev(sc), relu, x5, x2 if keep else None, mask, None,
                         G.workspace(gd, eoq.EOQ_PASS_FWD))
        assert G.status_clear() == 0
        assert np.array_equal(G.host(x5), ref["x5"]) and np.array_equal(G.unpack_mask(mask, out), ref["mask"])
        if keep:
            assert np.array_equal(G.host(x2).astype(np.int32), ref["x2"])
