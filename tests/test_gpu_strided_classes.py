"""Error back-propagation by the im2col kernel: the residue classes of a strided layer share launches of up to four GEMMs, and the
weights are read where they are whatever the number of channels."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import eoq, synth
import gpu_util as G

pytestmark = pytest.mark.gpu

GEOMETRIES = [
    # reductions over odd multiples of 16 channels, whose MMAs span two sub-tiles, padded ones among them; column atoms of 16 to 128 bytes
    oracle.ConvDesc(3, 9, 10, 16, 16, 1, 1, 1, 0),
    oracle.ConvDesc(2, 9, 10, 48, 48, 1, 1, 1, 0),
    oracle.ConvDesc(2, 12, 9, 64, 80, 1, 1, 1, 0),
    oracle.ConvDesc(40, 14, 14, 256, 112, 1, 1, 1, 0),
    oracle.ConvDesc(5, 37, 29, 48, 80, 3, 3, 2, 1),
    oracle.ConvDesc(2, 15, 16, 160, 48, 3, 3, 2, 1),
    oracle.ConvDesc(3, 7, 7, 128, 144, 3, 3, 1, 1),
    oracle.ConvDesc(1, 14, 14, 256, 512, 3, 3, 2, 1),    # one split for four classes of 1 to 4 taps
    oracle.ConvDesc(2, 17, 13, 64, 128, 3, 3, 2, 1),     # classes of other sizes
    oracle.ConvDesc(9, 30, 30, 32, 64, 3, 3, 2, 1),      # many tiles to a CTA under a cap
    oracle.ConvDesc(3, 11, 11, 32, 96, 5, 5, 3, 2),      # nine classes in three launches
    oracle.ConvDesc(2, 13, 9, 48, 80, 7, 7, 4, 3),       # sixteen classes, 16 channels to a chunk
    oracle.ConvDesc(2, 1, 9, 32, 32, 3, 3, 2, 1),        # no odd rows
    oracle.ConvDesc(2, 8, 8, 32, 64, 1, 1, 3, 0),        # eight classes without a tap
    oracle.ConvDesc(2, 9, 9, 32, 64, 2, 2, 3, 0),        # some without
]


@pytest.mark.parametrize("cap", [0, 1, 7])
@pytest.mark.parametrize("d", GEOMETRIES, ids=lambda d: "n%d_%dx%d_%d_%d_k%ds%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.stride))
def test_strided_classes(d, cap):
    """With and without the dump of the sums, whatever share of the CTAs a class gets."""
    gd, h = G.gdesc(d), eoq.eoq_create(0)
    if cap:
        eoq.eoq_set_gemm_ctas(h, cap)
    e3, w = synth.normal_codes((d.n, d.ho, d.wo, d.c_out), 2730, d.h, std_codes=24), synth.normal_codes((d.c_out, d.kh, d.kw, d.c_in), 2731, d.w, std_codes=6)
    acc = oracle.conv_dgrad_acc(d, e3, w)
    want, p, _ = oracle.sq_int(acc, -9 - 7)
    e3_d, w_d, exp, ws = G.dev(e3), G.dev(w), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.workspace(gd, eoq.EOQ_PASS_DGRAD)
    for dump in (None, G.empty(acc.shape, torch.int32)):
        e4, e4_exp, total = G.empty(acc.shape, torch.int8), G.zeros(1, torch.int32), G.empty(1, torch.int64)
        eoq.eoq_conv_dgrad(h, gd, e3_d, exp, w_d, e4, e4_exp, total, dump, ws)
        assert eoq.eoq_last_status(h) == 0
        assert np.array_equal(G.host(e4), want) and e4_exp.item() == p and total.item() == int(want.astype(np.int64).sum())
        assert dump is None or np.array_equal(G.host(dump), acc)
    eoq.eoq_destroy(h)


@pytest.mark.parametrize("d", [
    oracle.ConvDesc(3, 7, 9, 16, 16, 1, 1, 2, 0),       # one group of channels
    oracle.ConvDesc(5, 40, 41, 48, 32, 1, 1, 3, 0),     # three, a stride of three
    oracle.ConvDesc(97, 28, 28, 112, 64, 1, 1, 2, 0),   # two rounds and a bit of items to a thread
    oracle.ConvDesc(1, 1, 260, 80, 16, 1, 1, 7, 0),     # one row
], ids=lambda d: "n%d_%dx%d_%d_%d_s%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.stride))
def test_scattered_codes(d):
    """Strided 1x1 filters: codes on the grid, zeros elsewhere, for groups, widths, heights and strides that are no powers of two."""
    gd = G.gdesc(d)
    e3, w = synth.normal_codes((d.n, d.ho, d.wo, d.c_out), 2740, d.h, std_codes=24), synth.normal_codes((d.c_out, 1, 1, d.c_in), 2741, d.w, std_codes=6)
    want, p, _ = oracle.sq_int(oracle.conv_dgrad_acc(d, e3, w), -9 - 7)
    e4, e4_exp, total = torch.full(want.shape, 77, dtype=torch.int8, device="cuda:0"), G.zeros(1, torch.int32), G.empty(1, torch.int64)
    eoq.eoq_conv_dgrad(G.handle(), gd, G.dev(e3), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.dev(w), e4, e4_exp, total, None,
                       G.workspace(gd, eoq.EOQ_PASS_DGRAD))
    assert G.status_clear() == 0 and np.array_equal(G.host(e4), want) and e4_exp.item() == p
    assert total.item() == int(want.astype(np.int64).sum())


@pytest.mark.parametrize("cap", [0, 7])
@pytest.mark.parametrize("d", GEOMETRIES, ids=lambda d: "n%d_%dx%d_%d_%d_k%ds%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.stride))
def test_the_report_names_what_is_launched(d, cap):
    """Classes that a tap reaches, with their tiles and their shares of the CTAs, and the launches of the call."""
    gd, h = G.gdesc(d), eoq.eoq_create(0)
    if cap:
        eoq.eoq_set_gemm_ctas(h, cap)
    plan = dict(f.split("=") for f in eoq.eoq_describe_plan(h, gd, eoq.EOQ_PASS_DGRAD).split())

    def pixels(extent, k, r):
        return len(range(r, extent, d.stride)) if any((r + d.pad - q) % d.stride == 0 for q in range(k)) else 0

    rows = [d.n * pixels(d.h, d.kh, py) * pixels(d.w, d.kw, px) for py in range(d.stride) for px in range(d.stride)]
    live = [m for m in rows if m]
    if plan["kernel"] == "igemm":
        launches = -(-len(live) // 4)
        numbers = {f: [[int(v) for v in part.split(",")] for part in plan[f].split("/")] for f in ("tile_n", "m_tiles", "n_tiles", "ctas", "split")}
        assert int(plan["classes"]) == len(live) and int(plan["launches"]) == launches
        assert sum(numbers["m_tiles"], []) == [-(-m // 128) for m in live]
        assert all(n == -(-d.c_in // t) for n, t in zip(sum(numbers["n_tiles"], []), sum(numbers["tile_n"], [])))
        for tiles_m, tiles_n, ctas, (split,) in zip(numbers["m_tiles"], numbers["n_tiles"], numbers["ctas"], numbers["split"]):
            assert sum(ctas) <= max(cap or torch.cuda.get_device_properties(0).multi_processor_count, len(ctas))
            assert all(c % split == 0 and c <= m * n * split for c, m, n in zip(ctas, tiles_m, tiles_n))
            assert split == 1 or ctas == [m * n * split for m, n in zip(tiles_m, tiles_n)]   # (a cluster has one tile)
        if (d.n, d.c_out, d.stride, cap) == (1, 512, 2, 0):
            assert numbers["split"][0][0] > 1
    else:
        launches = 1
    e4, e4_exp = G.empty((d.n, d.h, d.w, d.c_in), torch.int8), G.zeros(1, torch.int32)
    before = eoq.eoq_launch_count(h)
    eoq.eoq_conv_dgrad(h, gd, G.zeros((d.n, d.ho, d.wo, d.c_out), torch.int8), G.zeros(1, torch.int32), G.zeros((d.c_out, d.kh, d.kw, d.c_in), torch.int8),
                       e4, e4_exp, None, None, G.workspace(gd, eoq.EOQ_PASS_DGRAD))
    assert eoq.eoq_launch_count(h) - before == launches + 1   # Q_e behind them
    eoq.eoq_last_status(h)   # (an error that is all zero is flagged)
    eoq.eoq_destroy(h)


@pytest.mark.parametrize("cap", [1, 3, 5, 7, 148])
@pytest.mark.parametrize("d", [
    oracle.ConvDesc(512, 112, 112, 16, 16, 3, 3, 2, 1),   # 12,544 tiles a class
    oracle.ConvDesc(300, 61, 53, 96, 48, 3, 3, 2, 1),     # classes of other sizes
    oracle.ConvDesc(64, 64, 64, 32, 64, 2, 2, 2, 0),      # four classes of one tap
], ids=lambda d: "n%d_%dx%d_%d_%d_k%ds%d" % (d.n, d.h, d.w, d.c_in, d.c_out, d.kh, d.stride))
def test_shares_of_the_classes(d, cap):
    """The division of the CTAs is that of the least time that suffices, counted up one by one; a plan of many tiles under a small cap
    is quick on the host all the same (12,544 tiles a class under three CTAs, counted up: 0.36 ms)."""
    gd, h = G.gdesc(d), eoq.eoq_create(0)
    eoq.eoq_set_gemm_ctas(h, cap)
    quickest = 1.0
    for _ in range(20):
        t = time.perf_counter()
        text = eoq.eoq_describe_plan(h, gd, eoq.EOQ_PASS_DGRAD)
        quickest = min(quickest, time.perf_counter() - t)
    plan = dict(f.split("=") for f in text.split())
    taps = [sum((r + d.pad - k) % d.stride == 0 for k in range(d.kh)) for r in range(d.stride)]
    cost = [2 * a * b + 1 for a in taps for b in taps]
    tiles = [int(m) * int(n) for m, n in zip(plan["m_tiles"].split(","), plan["n_tiles"].split(","))]
    at = sum(c * t for c, t in zip(cost, tiles)) // cap
    while at < max(cost) or not (sum(-(-t // (at // c)) for c, t in zip(cost, tiles)) <= max(cap, len(tiles))):
        at += 1
    assert [int(c) for c in plan["ctas"].split(",")] == [-(-t // (at // c)) for c, t in zip(cost, tiles)]
    assert quickest < 1.5e-4
    eoq.eoq_destroy(h)
