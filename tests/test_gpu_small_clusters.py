"""Kernels that take one cluster for small tensors, around the sizes where they hand over to the general ones, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import eoq, synth
import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [1, 511, 512, 513, 2047, 2049, 4097, 12287, 12288, 12289])
@pytest.mark.parametrize("gamma,with_x2", [(118, True), (128, False), (-700, True), (0, False)])
def test_error_head_sizes(groups, gamma, with_x2):
    """Groups of 16 codes: clusters of 1, 2, 4 and 8 blocks with up to two groups a thread, then two kernels."""
    n = 16 * groups
    e0 = synth.normal_codes(n, 2900, groups, std_codes=30)
    mask = (synth.int8_uniform(n, 2901, groups) > -20).astype(np.uint8)
    x2 = synth.int8_uniform(n, 2902, groups).astype(np.int16) * 200 if with_x2 else None
    e3, p = G.empty((n,), torch.int8), G.zeros(1, torch.int32)
    s1, s2 = G.zeros(1, torch.int64), G.zeros(1, torch.int64)
    for _ in range(2):
        eoq.eoq_err_prescale_dev(G.handle(), G.dev(e0), torch.tensor([-12], dtype=torch.int32, device="cuda:0"), G.dev(G.pack_mask(mask)),
                                 None if x2 is None else G.dev(x2), n, torch.tensor([gamma], dtype=torch.int32, device="cuda:0"), e3, p, s1,
                                 None if x2 is None else s2)
        e1 = e0.astype(np.int64) * mask
        assert G.status_clear() == (0 if (e1 * gamma).any() else eoq.EOQ_DEV_SQ_ZERO)
        assert s1.item() == int(e1.sum()) and (x2 is None or s2.item() == int((e1 * x2).sum()))
        want, pw, _ = oracle.sq_int(e1 * gamma, -12 - 7)
        assert np.array_equal(G.host(e3), want) and p.item() == pw


@pytest.mark.parametrize("groups", [4096, 189440, 189441, 3 * 189440 - 7])
@pytest.mark.parametrize("masked", [False, True])
def test_error_head_of_several_groups_to_a_thread(groups, masked):
    """The largest cluster, and two kernels whose threads take one to three groups (five blocks of 256 threads to an SM), a maximum that
    only the last group holds among them."""
    n = 16 * groups
    e0 = synth.normal_codes(n, 2910, groups, std_codes=9).clip(-60, 60).astype(np.int8)
    e0[n - 1] = -127
    mask = synth.bits(n, 2911, groups, 0.5) if masked else None
    if masked:
        mask[n - 1] = 1
    x2 = synth.int8_uniform(n, 2912, groups).astype(np.int16) * 250
    e1 = e0.astype(np.int64) * (1 if mask is None else mask)
    e3, p, s1, s2 = G.empty((n,), torch.int8), G.zeros(1, torch.int32), G.zeros(1, torch.int64), G.zeros(1, torch.int64)
    eoq.eoq_err_prescale(G.handle(), G.dev(e0), torch.tensor([-12], dtype=torch.int32, device="cuda:0"), G.dev(G.pack_mask(mask)) if masked else None,
                         G.dev(x2), n, 118, e3, p, s1, s2)
    want, pw, _ = oracle.sq_int(e1 * 118, -12 - 7)
    assert G.status_clear() == 0 and np.array_equal(G.host(e3), want) and p.item() == pw
    assert s1.item() == int(e1.sum()) and s2.item() == int((e1 * x2).sum())


GEOMETRIES = [
    oracle.ConvDesc(1, 1, 1, 16, 16, 1, 1, 1, 0),      # one pixel: most of the taps' sets are empty
    oracle.ConvDesc(8, 32, 32, 16, 16, 3, 3, 1, 1),    # a slice per pixel block
    oracle.ConvDesc(2, 5, 6, 32, 48, 3, 3, 1, 1),
    oracle.ConvDesc(3, 9, 7, 64, 256, 1, 1, 1, 0),     # 16,384 weights: the most that one cluster takes; two slabs of channels
    oracle.ConvDesc(3, 9, 7, 64, 272, 1, 1, 1, 0),     # more: three launches
    oracle.ConvDesc(2, 11, 13, 16, 112, 3, 3, 2, 1),   # strided, borders at the top and left only
    oracle.ConvDesc(1, 4, 3, 16, 32, 5, 5, 1, 2),      # every row and column a border
]


@pytest.mark.parametrize("d", GEOMETRIES, ids=lambda d: "n%d_%dx%d_%d_%d_k%ds%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.stride))
@pytest.mark.parametrize("b1", [0, -2, 900])
def test_weight_gradient_finish(d, b1):
    x0, e3 = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2910, d.c_in), synth.normal_codes((d.n, d.ho, d.wo, d.c_out), 2911, d.c_out, std_codes=30)
    acc = oracle.conv_wgrad_acc(d, e3, x0, b1)
    want, p, _ = oracle.sq_int(acc, -16)
    gd = G.gdesc(d)
    ws = G.workspace(gd, eoq.EOQ_PASS_WGRAD)
    ws.fill_(0x5a)
    for dump in (None, G.zeros(acc.shape, torch.int64)):
        g, ex = G.empty(acc.shape, torch.int8), G.zeros(1, torch.int32)
        eoq.eoq_conv_wgrad(G.handle(), gd, G.dev(e3), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.dev(x0), b1, g, ex, dump, ws)
        assert G.status_clear() == 0
        assert np.array_equal(G.host(g), want) and ex.item() == p
    assert np.array_equal(G.host(dump), acc)
