"""Implicit GEMMs of a handful of tiles (small batches): clusters that share a tile's reduction, and column tiles of every width they
take, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import eoq, synth
import gpu_util as G

pytestmark = pytest.mark.gpu

GEOMETRIES = [
    oracle.ConvDesc(4, 6, 6, 96, 384, 3, 3, 1, 1),     # weights as several column atoms in a cluster
    oracle.ConvDesc(1, 7, 7, 512, 512, 3, 3, 1, 1),    # fewer pixels than half a tile, clusters of eight
    oracle.ConvDesc(1, 14, 14, 256, 256, 3, 3, 1, 1),  # a second row tile of 68 pixels
    oracle.ConvDesc(1, 5, 7, 80, 160, 3, 3, 1, 1),     # column tiles that reach past the last channel
    oracle.ConvDesc(2, 9, 9, 48, 144, 3, 3, 2, 1),     # strided: residue classes with plans of their own
    oracle.ConvDesc(1, 28, 28, 128, 128, 3, 3, 1, 1),  # patch kernel, several column tiles with resident weights
    oracle.ConvDesc(2, 12, 10, 16, 80, 3, 3, 1, 1),
    oracle.ConvDesc(3, 9, 14, 112, 64, 5, 5, 1, 2),    # 25 taps, an odd multiple of 16 channels
    oracle.ConvDesc(2, 8, 8, 1024, 208, 1, 1, 1, 0),
]


@pytest.mark.parametrize("d", GEOMETRIES, ids=lambda d: "n%d_%dx%d_%d_%d_k%ds%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.stride))
@pytest.mark.parametrize("relu", [True, False])
def test_few_tiles(d, relu):
    x0, w = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2700, d.c_in), synth.normal_codes((d.c_out, d.kh, d.kw, d.c_in), 2701, d.c_out, std_codes=6)
    out = (d.n, d.ho, d.wo, d.c_out)
    shortcut, e3 = synth.int8_uniform(out, 2702, d.h), synth.normal_codes(out, 2703, d.w, std_codes=24)
    gd = G.gdesc(d)
    gamma = 118 if relu else 128
    ref = oracle.layer_forward(d, x0, -2, w, gamma, 3, shortcut, relu)
    x5, x2, mask = G.zeros(out, torch.int8), G.zeros(out, torch.int16), G.zeros((ref["x5"].size + 7) // 8, torch.uint8)
    eoq.eoq_conv_fwd(G.handle(), gd, G.dev(x0), None, -2, G.dev(w), gamma, 3, G.dev(shortcut), relu, x5, x2, mask, None, G.workspace(gd, eoq.EOQ_PASS_FWD))
    acc = oracle.conv_dgrad_acc(d, e3, w)
    want, p, _ = oracle.sq_int(acc, -9 - 7)
    e4, e4_exp, total = G.zeros(acc.shape, torch.int8), G.zeros(1, torch.int32), G.zeros(1, torch.int64)
    exp = torch.tensor([-9], dtype=torch.int32, device="cuda:0")
    eoq.eoq_conv_dgrad(G.handle(), gd, G.dev(e3), exp, G.dev(w), e4, e4_exp, total, None, G.workspace(gd, eoq.EOQ_PASS_DGRAD))
    assert G.status_clear() == 0
    assert np.array_equal(G.host(x5), ref["x5"]) and np.array_equal(G.host(x2).astype(np.int32), ref["x2"])
    if relu:
        assert np.array_equal(G.unpack_mask(mask, out), ref["mask"])
    assert np.array_equal(G.host(e4), want) and e4_exp.item() == p and total.item() == int(want.astype(np.int64).sum())


WIDE = [
    oracle.ConvDesc(150, 14, 14, 64, 512, 1, 1, 1, 0),    # narrow tiles for their even shares
    oracle.ConvDesc(100, 14, 14, 64, 528, 1, 1, 1, 0),    # five of 112, the last one of 80
    oracle.ConvDesc(100, 14, 14, 576, 304, 1, 1, 1, 0),   # two of 160, the last one of 144
    oracle.ConvDesc(20, 14, 14, 64, 304, 1, 1, 1, 0),     # few tiles: three of 112, the last one of 80
    oracle.ConvDesc(31, 27, 27, 48, 272, 3, 3, 2, 1),     # three of 96, strided, 16-byte chunks
]


@pytest.mark.parametrize("d", WIDE, ids=lambda d: "n%d_%dx%d_%d_%d_k%ds%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.stride))
@pytest.mark.parametrize("gamma", [118, 128])
def test_forward_column_cuts(d, gamma):
    """More than 128 output channels: equal cuts, and tiles that reach past the last channel."""
    x0, w = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2705, d.c_in), synth.normal_codes((d.c_out, d.kh, d.kw, d.c_in), 2706, d.c_out, std_codes=6)
    out = (d.n, d.ho, d.wo, d.c_out)
    shortcut = synth.int8_uniform(out, 2707, d.h) if gamma != 128 else None
    gd = G.gdesc(d)
    ref = oracle.layer_forward(d, x0, -2, w, gamma, 3, shortcut, True)
    x5, x2, mask = G.zeros(out, torch.int8), G.zeros(out, torch.int16) if gamma != 128 else None, G.zeros((ref["x5"].size + 7) // 8, torch.uint8)
    eoq.eoq_conv_fwd(G.handle(), gd, G.dev(x0), None, -2, G.dev(w), gamma, 3, None if shortcut is None else G.dev(shortcut), True, x5, x2, mask, None,
                     G.workspace(gd, eoq.EOQ_PASS_FWD))
    assert G.status_clear() == 0 and np.array_equal(G.host(x5), ref["x5"]) and np.array_equal(G.unpack_mask(mask, out), ref["mask"])
    assert x2 is None or np.array_equal(G.host(x2).astype(np.int32), ref["x2"])


@pytest.mark.parametrize("b2", [0, 3, -5, 16384, -16384, 16385, -32768, 32767])
@pytest.mark.parametrize("relu", [True, False])
def test_unit_gamma_without_shortcut(relu, b2):
    """gamma = 1 and no shortcut: x5 comes from one rounding, with b2 in its limits (|b2| <= 2^14) or by the general chain; ties at both parities."""
    d = oracle.ConvDesc(2, 9, 20, 32, 48, 3, 3, 1, 1)
    x0, w = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2710, 1), synth.normal_codes((d.c_out, d.kh, d.kw, d.c_in), 2711, 2, std_codes=40 if abs(b2) > 100 else 2)
    x0 = (x0 // 16 * 16).astype(np.int8)   # sums in steps of 16: every eighth is a tie
    ref = oracle.layer_forward(d, x0, -2, w, 128, b2, None, relu)
    out = (d.n, d.ho, d.wo, d.c_out)
    gd = G.gdesc(d)
    for keep in (False, True):   # without x2, and with it (the general chain)
        x5, mask = G.zeros(out, torch.int8), G.zeros((ref["x5"].size + 7) // 8, torch.uint8)
        x2 = G.zeros(out, torch.int16) if keep else None
        eoq.eoq_conv_fwd(G.handle(), gd, G.dev(x0), None, -2, G.dev(w), 128, b2, None, relu, x5, x2, mask, None, G.workspace(gd, eoq.EOQ_PASS_FWD))
        assert G.status_clear() == 0
        assert np.array_equal(G.host(x5), ref["x5"]) and np.array_equal(G.unpack_mask(mask, out), ref["mask"])


@pytest.mark.parametrize("c_in,c_out", [(16, 16), (32, 32), (16, 32), (48, 32), (32, 48), (32, 96), (96, 96), (160, 160)])
@pytest.mark.parametrize("n", [1, 8])
def test_error_back_propagation_in_72_registers(n, c_in, c_out):
    """The kernel of fewer registers is for a reduction of one 32-channel chunk into a column tile of at most 32: no layer of several
    chunks takes it, however narrow its column tiles are."""
    d = oracle.ConvDesc(n, 16, 16, c_in, c_out, 3, 3, 1, 1)
    gd = G.gdesc(d)
    plan = eoq.eoq_describe_plan(G.handle(), gd, eoq.EOQ_PASS_DGRAD)
    narrow = int(plan.split("tile_n=")[1].split()[0]) <= 32
    assert ("registers=72" in plan) == ("kernel=igemm_patch" in plan and c_out <= 32 and narrow)
    assert c_out > 32 or "kernel=igemm_patch" in plan
    e3, w = synth.normal_codes((n, 16, 16, c_out), 2720, c_in, std_codes=24), synth.normal_codes((c_out, 3, 3, c_in), 2721, c_out, std_codes=6)
    acc = oracle.conv_dgrad_acc(d, e3, w)
    want, p, _ = oracle.sq_int(acc, -9 - 7)
    e4, e4_exp, total = G.zeros(acc.shape, torch.int8), G.zeros(1, torch.int32), G.zeros(1, torch.int64)
    eoq.eoq_conv_dgrad(G.handle(), gd, G.dev(e3), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.dev(w), e4, e4_exp, total, None,
                       G.workspace(gd, eoq.EOQ_PASS_DGRAD))
    assert G.status_clear() == 0
    assert np.array_equal(G.host(e4), want) and e4_exp.item() == p and total.item() == int(want.astype(np.int64).sum())
