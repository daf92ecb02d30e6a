"""The weight gradient in two parts (eoq_conv_wgrad_gemm per layer, one eoq_wgrad_finish for all layers) against the
oracle and against the one-call form, bit for bit: both GEMM kernels, with and without the b1 term, more layers than
one launch batch holds."""
import numpy as np
import pytest
import torch

import oracle
from oracle import ConvDesc
from paper_2105_13890_b200 import eoq, synth

import gpu_util as G

pytestmark = pytest.mark.gpu

LAYERS = [  # n, h, w, c_in, c_out, k, stride, pad, b1 (None: no bias in front of the convolution)
    (2, 12, 12, 32, 32, 3, 1, 1, -2),       # patch kernel, int32 slices
    (3, 7, 7, 64, 128, 3, 1, 1, 5),
    (2, 10, 10, 32, 64, 3, 2, 1, 3),        # strided: per-tap kernel
    (2, 9, 11, 48, 32, 1, 1, 0, -7),
    (2, 16, 16, 16, 32, 7, 2, 3, None),     # a first-layer shape
    (1, 20, 20, 64, 64, 5, 1, 2, 0),        # b1 present and zero
]


def make(case, seed):
    n, h, w, c_in, c_out, k, stride, pad, b1 = case
    d = ConvDesc(n, h, w, c_in, c_out, k, k, stride, pad)
    e3 = synth.normal_codes((n, d.ho, d.wo, c_out), seed, 0)
    x0 = synth.relu_codes((n, h, w, c_in), seed, 1)
    S = oracle.conv_wgrad_acc(d, e3, x0, b1 or 0)
    g_o, pg_o, _ = oracle.sq_int(S, -12 - 7)
    return d, e3, x0, b1, g_o, pg_o


@pytest.mark.parametrize("repeat", [1, 4])     # 6 and 24 layers: the second needs two launch batches
def test_gemm_per_layer_and_one_finish_for_all(repeat):
    hd = G.handle()
    cases = [make(c, 8900 + 10 * r + i) for r in range(repeat) for i, c in enumerate(LAYERS)]
    descs, e3s, pes, b1s, gs, pgs, wss, parts = [], [], [], [], [], [], [], []
    for d, e3, x0, b1, _, _ in cases:
        gd = G.gdesc(d)
        ws = G.workspace(gd, eoq.EOQ_PASS_WGRAD)
        e3_d, pe = G.dev(e3), G.dev(np.array([-12], dtype=np.int32))
        parts.append(eoq.eoq_conv_wgrad_gemm(hd, gd, e3_d, pe, G.dev(x0), ws))
        descs.append(gd); e3s.append(e3_d); pes.append(pe); wss.append(ws)
        b1s.append(None if b1 is None else G.dev(np.array([b1], dtype=np.int32)))
        gs.append(G.zeros((d.c_out, d.kh, d.kw, d.c_in), torch.int8)); pgs.append(G.zeros(1, torch.int32))
    eoq.eoq_wgrad_finish(hd, descs, e3s, pes, b1s, gs, pgs, wss, parts)
    torch.cuda.synchronize()
    assert eoq.eoq_last_status(hd) == 0
    for (d, e3, x0, b1, g_o, pg_o), g, pg in zip(cases, gs, pgs):
        assert np.array_equal(G.host(g), g_o) and pg.item() == pg_o, (d, b1)
    # the same through the one-call form, on the same handle (its cells are clean)
    d, e3, x0, b1, g_o, pg_o = cases[0]
    gd = G.gdesc(d)
    g1, pg1 = G.zeros(g_o.shape, torch.int8), G.zeros(1, torch.int32)
    eoq.eoq_conv_wgrad_dev(hd, gd, G.dev(e3), G.dev(np.array([-12], dtype=np.int32)), G.dev(x0), G.dev(np.array([b1], dtype=np.int32)), g1, pg1,
                           G.workspace(gd, eoq.EOQ_PASS_WGRAD))
    torch.cuda.synchronize()
    assert np.array_equal(G.host(g1), g_o) and pg1.item() == pg_o


def test_a_zero_error_gives_zero_gradients_and_the_flag():
    hd = G.handle()
    d = ConvDesc(2, 8, 8, 32, 32, 3, 3, 1, 1)
    gd = G.gdesc(d)
    ws = G.workspace(gd, eoq.EOQ_PASS_WGRAD)
    e3, pe = G.zeros((2, 8, 8, 32), torch.int8), G.dev(np.array([-12], dtype=np.int32))
    parts = eoq.eoq_conv_wgrad_gemm(hd, gd, e3, pe, G.dev(synth.relu_codes((2, 8, 8, 32), 1, 0)), ws)
    g, pg = G.empty((32, 3, 3, 32), torch.int8), G.zeros(1, torch.int32)
    eoq.eoq_wgrad_finish(hd, [gd], [e3], [pe], [G.dev(np.array([4], dtype=np.int32))], [g], [pg], [ws], [parts])
    torch.cuda.synchronize()
    assert not G.host(g).any() and pg.item() == -19
    assert eoq.eoq_last_status(hd) == eoq.EOQ_DEV_SQ_ZERO
    G.status_clear()


@pytest.mark.parametrize("b1", [None, -3])
def test_profile_groups_of_a_weight_gradient(b1):
    """The GEMM, the b1 error sums and what follows them are timed as kinds of their own, per call and in two parts."""
    d, e3, x0, _, g_o, pg_o = make((2, 12, 12, 32, 32, 3, 1, 1, b1), 9100)
    gd, h = G.gdesc(d), eoq.eoq_create(0)
    e3_d, x_d, pe = G.dev(e3), G.dev(x0), G.dev(np.array([-12], dtype=np.int32))
    b1_d = None if b1 is None else G.dev(np.array([b1], dtype=np.int32))
    ws, g, pg = G.workspace(gd, eoq.EOQ_PASS_WGRAD), G.zeros(g_o.shape, torch.int8), G.zeros(1, torch.int32)
    kinds = dict.fromkeys(eoq.EOQ_PROF_NAMES, 0)
    kinds.update(wgrad_gemm=2, wgrad_aux=2, wgrad_taps=0 if b1 is None else 2)
    before = eoq.eoq_launch_count(h)
    eoq.eoq_profile_start(h)
    eoq.eoq_conv_wgrad_dev(h, gd, e3_d, pe, x_d, b1_d, g, pg, ws)
    parts = eoq.eoq_conv_wgrad_gemm(h, gd, e3_d, pe, x_d, ws)
    eoq.eoq_wgrad_finish(h, [gd], [e3_d], [pe], [b1_d], [g], [pg], [ws], [parts])
    n, ms = eoq.eoq_profile_stop(h)
    assert dict(zip(eoq.EOQ_PROF_NAMES, n)) == kinds
    assert all((t > 0) == (k > 0) for k, t in zip(n, ms))
    assert eoq.eoq_launch_count(h) - before == 6 + kinds["wgrad_taps"]
    assert np.array_equal(G.host(g), g_o) and pg.item() == pg_o and eoq.eoq_last_status(h) == 0
    eoq.eoq_destroy(h)


# from one slice of the GEMM to about one per SM: an incomplete round of loads, several rounds, groups of slices
SLICES = [
    oracle.ConvDesc(1, 7, 7, 128, 128, 3, 3, 1, 1),
    oracle.ConvDesc(2, 9, 9, 256, 256, 1, 1, 1, 0),
    oracle.ConvDesc(9, 7, 7, 256, 256, 3, 3, 1, 1),
    oracle.ConvDesc(16, 14, 14, 256, 256, 3, 3, 1, 1),
    oracle.ConvDesc(16, 28, 28, 128, 128, 3, 3, 1, 1),
    oracle.ConvDesc(64, 32, 32, 16, 16, 3, 3, 1, 1),
    oracle.ConvDesc(6, 56, 56, 64, 64, 3, 3, 1, 1),
]


@pytest.mark.parametrize("d", SLICES, ids=lambda d: "n%d_%dx%d_%d_%d" % (d.n, d.h, d.w, d.c_in, d.c_out))
@pytest.mark.parametrize("b1", [0, 3, -30000])
def test_sums_of_slices(d, b1):
    """32-bit sums, and 64-bit ones where pixels * 127 * (127 + |b1|) does not fit."""
    x0, e3 = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2960, d.c_in), synth.normal_codes((d.n, d.ho, d.wo, d.c_out), 2961, d.c_out, std_codes=30)
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


@pytest.mark.parametrize("d", [oracle.ConvDesc(4, 16, 16, 16, 16, 3, 3, 1, 1), oracle.ConvDesc(8, 28, 28, 64, 128, 3, 3, 1, 1),
                               oracle.ConvDesc(5, 17, 15, 32, 48, 3, 3, 2, 1)], ids=lambda d: "n%d_%d_%d_s%d" % (d.n, d.c_in, d.c_out, d.stride))
def test_error_sums_beside_the_gemm(d):
    """The error sums start beside the GEMM: errors that the kernel in front of it wrote, over and over into one buffer and one
    workspace, have to be the ones they see."""
    hd, rounds = G.handle(), 12
    shape = (d.n, d.ho, d.wo, d.c_out)
    n = int(np.prod(shape))
    x0 = synth.int8_uniform((d.n, d.h, d.w, d.c_in), 2970, d.c_in)
    e0s = [synth.normal_codes(shape, 2971, i, std_codes=10 + 6 * i) for i in range(rounds)]
    gd = G.gdesc(d)
    ws = G.workspace(gd, eoq.EOQ_PASS_WGRAD)
    e3, pe, gamma, p_in = G.empty(shape, torch.int8), G.zeros(1, torch.int32), torch.tensor([128], dtype=torch.int32, device="cuda:0"), G.zeros(1, torch.int32)
    b1, x, mask = torch.tensor([-37], dtype=torch.int32, device="cuda:0"), G.dev(x0), G.dev(G.pack_mask(np.ones(n, np.uint8)))
    ins = [G.dev(e) for e in e0s]
    outs = [(G.empty((d.c_out, d.kh, d.kw, d.c_in), torch.int8), G.zeros(1, torch.int32)) for _ in e0s]
    for e0, (g, pg) in zip(ins, outs):
        eoq.eoq_err_prescale_dev(hd, e0, p_in, mask, None, n, gamma, e3, pe, G.zeros(1, torch.int64), None)
        eoq.eoq_conv_wgrad_dev(hd, gd, e3, pe, x, b1, g, pg, ws)
    assert G.status_clear() == 0
    for e0, (g, pg) in zip(e0s, outs):
        e3_o, p3, _ = oracle.sq_int(e0.astype(np.int64) * 128, -7)
        want, p, _ = oracle.sq_int(oracle.conv_wgrad_acc(d, e3_o, x0, -37), p3 - 7)
        assert np.array_equal(G.host(g), want) and pg.item() == p


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("case", [
    (1, 5, 6, 16, 16, 3, 1, 1, 7),           # fewer rows than copies of the error sums
    (3, 70, 45, 16, 48, 3, 2, 1, -3),        # a slab of 32 channels and one of 16
    (5, 65, 64, 16, 32, 3, 1, 1, 9),         # more ranges of rows than copies: 21 alone, 6 in a batch
    (9, 66, 64, 32, 80, 1, 1, 0, 11),        # 38 and 10, in three slabs
    (33, 66, 65, 16, 32, 5, 1, 2, -128),     # 139 and 32, four border rows and columns
    (1, 3, 300, 16, 32, 7, 1, 3, 100),       # every row a class of its own
], ids=lambda c: "n%d_%dx%d_%d_%d_k%ds%d" % c[:7])
def test_error_sums_of_every_cluster_size(case, batched):
    """The b1 term against the oracle where a layer's error sums are formed by one block, by up to four that store a copy each, or by more
    that add; a single call (sums beside the GEMM) and a finish of two layers, twice on one workspace whose contents are arbitrary."""
    hd = G.handle()
    d, e3, x0, b1, g_o, pg_o = make(case, 8960)
    gd, ws = G.gdesc(d), G.workspace(G.gdesc(d), eoq.EOQ_PASS_WGRAD)
    ws.fill_(0x5A)
    e3_d, pe, x_d, b1_d = G.dev(e3), G.dev(np.array([-12], dtype=np.int32)), G.dev(x0), G.dev(np.array([b1], dtype=np.int32))
    for _ in range(2):
        g, pg = G.empty(g_o.shape, torch.int8), G.zeros(1, torch.int32)
        if batched:
            d2, e2, x2, c2, g2_o, pg2_o = make(LAYERS[1], 8961)
            ws2, g2, pg2 = G.workspace(G.gdesc(d2), eoq.EOQ_PASS_WGRAD), G.empty(g2_o.shape, torch.int8), G.zeros(1, torch.int32)
            e2_d = G.dev(e2)
            parts = [eoq.eoq_conv_wgrad_gemm(hd, gd, e3_d, pe, x_d, ws), eoq.eoq_conv_wgrad_gemm(hd, G.gdesc(d2), e2_d, pe, G.dev(x2), ws2)]
            eoq.eoq_wgrad_finish(hd, [gd, G.gdesc(d2)], [e3_d, e2_d], [pe, pe], [b1_d, G.dev(np.array([c2], dtype=np.int32))], [g, g2],
                                 [pg, pg2], [ws, ws2], parts)
            assert np.array_equal(G.host(g2), g2_o) and pg2.item() == pg2_o
        else:
            eoq.eoq_conv_wgrad_dev(hd, gd, e3_d, pe, x_d, b1_d, g, pg, ws)
        assert G.status_clear() == 0 and np.array_equal(G.host(g), g_o) and pg.item() == pg_o


@pytest.mark.parametrize("case", [
    (3, 70, 45, 16, 48, 3, 2, 1, -3),        # up to four copies, stored
    (5, 65, 64, 16, 32, 3, 1, 1, 9),         # 21 ranges that add where the device is free, 6 where GEMMs are capped
    (2, 65, 64, 16, 32, 3, 1, 1, 9),         # 9 that add, 4 that store
    (33, 66, 65, 16, 32, 1, 1, 0, -128),
], ids=lambda c: "n%d_%dx%d_%d_%d_k%ds%d" % c[:7])
def test_slices_finished_more_than_once(case):
    """The sums of one GEMM can be finished again, by handles whose plans store the error sums or add them, alone or together."""
    d, e3, x0, b1, g_o, pg_o = make(case, 8970)
    gd, capped, hd = G.gdesc(d), eoq.eoq_create(0), G.handle()
    eoq.eoq_set_gemm_ctas(capped, 20)
    ws = G.workspace(gd, eoq.EOQ_PASS_WGRAD)
    ws.fill_(0x5A)
    e3_d, pe, b1_d = G.dev(e3), G.dev(np.array([-12], dtype=np.int32)), G.dev(np.array([b1], dtype=np.int32))
    d2, e2, x2, c2, g2_o, pg2_o = make(LAYERS[1], 8971)
    ws2, e2_d, b2_d = G.workspace(G.gdesc(d2), eoq.EOQ_PASS_WGRAD), G.dev(e2), G.dev(np.array([c2], dtype=np.int32))
    parts = eoq.eoq_conv_wgrad_gemm(hd, gd, e3_d, pe, G.dev(x0), ws)
    parts2 = eoq.eoq_conv_wgrad_gemm(hd, G.gdesc(d2), e2_d, pe, G.dev(x2), ws2)
    for h, together in ((hd, False), (capped, False), (hd, False), (hd, True), (hd, False), (capped, True), (hd, False)):
        g, pg, g2, pg2 = G.empty(g_o.shape, torch.int8), G.zeros(1, torch.int32), G.empty(g2_o.shape, torch.int8), G.zeros(1, torch.int32)
        if together:
            eoq.eoq_wgrad_finish(h, [gd, G.gdesc(d2)], [e3_d, e2_d], [pe, pe], [b1_d, b2_d], [g, g2], [pg, pg2], [ws, ws2], [parts, parts2])
            assert np.array_equal(G.host(g2), g2_o) and pg2.item() == pg2_o
        else:
            eoq.eoq_wgrad_finish(h, [gd], [e3_d], [pe], [b1_d], [g], [pg], [ws], [parts])
        assert eoq.eoq_last_status(h) == 0 and np.array_equal(G.host(g), g_o) and pg.item() == pg_o
    eoq.eoq_destroy(capped)


@pytest.mark.parametrize("case", [(12, 32, 32, 16, 16, 3, 1, 1, -2), (7, 31, 33, 16, 32, 3, 1, 1, 5)], ids=["16", "32"])
def test_small_slices_finished_again_under_another_plan(case):
    """A small layer is finished by one launch that stores its error sums; a profile has them added up by a kernel of their own."""
    d, e3, x0, b1, g_o, pg_o = make(case, 8980)
    gd, h, capped = G.gdesc(d), eoq.eoq_create(0), eoq.eoq_create(0)
    eoq.eoq_set_gemm_ctas(capped, 40)   # (few slices: a small layer)
    ws = G.workspace(gd, eoq.EOQ_PASS_WGRAD)
    ws.fill_(0x5A)
    e3_d, pe, b1_d = G.dev(e3), G.dev(np.array([-12], dtype=np.int32)), G.dev(np.array([b1], dtype=np.int32))
    parts = eoq.eoq_conv_wgrad_gemm(capped, gd, e3_d, pe, G.dev(x0), ws)
    for profiled in (False, True, False, True):
        g, pg = G.empty(g_o.shape, torch.int8), G.zeros(1, torch.int32)
        if profiled:
            eoq.eoq_profile_start(h)
        before = eoq.eoq_launch_count(h)
        eoq.eoq_wgrad_finish(h, [gd], [e3_d], [pe], [b1_d], [g], [pg], [ws], [parts])
        assert eoq.eoq_launch_count(h) - before == (3 if profiled else 1)
        if profiled:
            eoq.eoq_profile_stop(h)
        assert eoq.eoq_last_status(h) == 0 and np.array_equal(G.host(g), g_o) and pg.item() == pg_o
    eoq.eoq_destroy(h)
    eoq.eoq_destroy(capped)


@pytest.mark.parametrize("n,extent,c_in,c_out", [(512, 56, 64, 64), (512, 56, 16, 32), (256, 112, 32, 32)])
def test_error_sums_of_few_channels_hide_beside_the_gemm(n, extent, c_in, c_out):
    """A bias in front of the convolution costs a large weight gradient the adding up of its error sums and little more: they are read beside
    the GEMM (with and without: 1.08 to 1.15; in front of it, by 32 blocks to 32 channels: 1.28 to 1.33)."""
    h, gd = eoq.eoq_create(0), eoq.conv_desc(n, extent, extent, c_in, c_out, 3, 3, 1, 1)
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(1)
    x, e3 = (torch.randint(-90, 91, (n, extent, extent, c), generator=gen, device="cuda:0", dtype=torch.int8) for c in (c_in, c_out))
    g, pe, pg, b1 = G.empty((c_out, 3, 3, c_in), torch.int8), G.zeros(1, torch.int32), G.zeros(1, torch.int32), torch.tensor([-2], dtype=torch.int32, device="cuda:0")
    ws, graphs = G.workspace(gd, eoq.EOQ_PASS_WGRAD), []
    for bias in (None, b1):
        eoq.eoq_conv_wgrad_dev(h, gd, e3, pe, x, bias, g, pg, ws)
        torch.cuda.synchronize()
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            for _ in range(10):
                eoq.eoq_conv_wgrad_dev(h, gd, e3, pe, x, bias, g, pg, ws)
    best = [1e9, 1e9]
    for _ in range(10):
        for k, graph in enumerate(graphs):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.replay()
            b.record()
            torch.cuda.synchronize()
            best[k] = min(best[k], a.elapsed_time(b))
    assert best[1] < 1.22 * best[0], best
    eoq.eoq_destroy(h)
