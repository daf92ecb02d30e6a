"""Error back-propagation whose sums travel as 16-bit words: every size of sum that the words treat differently, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import eoq, synth
import gpu_util as G

pytestmark = pytest.mark.gpu

GEOMETRIES = {
    "patch": oracle.ConvDesc(2, 9, 13, 32, 48, 3, 3, 1, 1),
    "taps, strided": oracle.ConvDesc(2, 11, 7, 32, 64, 3, 3, 2, 1),
    "1x1": oracle.ConvDesc(3, 6, 7, 16, 512, 1, 1, 1, 0),
    "1x1 strided": oracle.ConvDesc(2, 9, 8, 48, 256, 1, 1, 2, 0),
    "unreached rows": oracle.ConvDesc(1, 7, 9, 16, 32, 1, 1, 2, 1),
    "cluster": oracle.ConvDesc(1, 7, 7, 128, 512, 3, 3, 1, 1),
}


def _errors(kind, shape, seed):
    """Codes whose sums stay below the code range, below 2^14 (kept whole), pass it in some pixels only, or in all of them."""
    if kind == "zero":
        return np.zeros(shape, np.int8)
    e = synth.normal_codes(shape, 2600, seed, std_codes={"tiny": 1, "whole": 6, "mixed": 4, "large": 60}[kind]).astype(np.int32)
    if kind == "tiny":
        e[...] = 0
        e.reshape(-1)[::97] = 1
    if kind == "mixed":   # a few pixels 25 times as large as the rest
        rows = e.reshape(-1, shape[-1])
        rows[::11] *= 25
    return np.clip(e, -127, 127).astype(np.int8)


@pytest.mark.parametrize("kind", ["zero", "tiny", "whole", "mixed", "large"])
@pytest.mark.parametrize("name", list(GEOMETRIES))
def test_sums_as_16_bit_words(name, kind):
    d = GEOMETRIES[name]
    e3 = _errors(kind, (d.n, d.ho, d.wo, d.c_out), len(name))
    w = np.clip(np.round(synth.normal_f32((d.c_out, d.kh, d.kw, d.c_in), 2601, d.c_in) * (1 if kind == "tiny" else 20)), -127, 127).astype(np.int8)
    if kind == "large" and name == "1x1":   # every product at its largest: 512 * 127 * 127, the same sign within a pixel
        e3[...], w[...] = 127, 127
        e3[1] = -127
    acc = oracle.conv_dgrad_acc(d, e3, w)
    want, p, _ = oracle.sq_int(acc, -9 - 7)
    desc = G.gdesc(d)
    exp = torch.tensor([-9], dtype=torch.int32, device="cuda:0")
    e4, e4_exp, total = G.empty(acc.shape, torch.int8), G.zeros(1, torch.int32), G.zeros(1, torch.int64)
    ws = G.workspace(desc, eoq.EOQ_PASS_DGRAD)
    for dump in (None, G.empty(acc.shape, torch.int32)):   # the words, then the int32 sums that a caller may ask for
        e4.fill_(99)
        eoq.eoq_conv_dgrad(G.handle(), desc, G.dev(e3), exp, G.dev(w), e4, e4_exp, total, dump, ws)
        assert G.status_clear() == (0 if acc.any() else eoq.EOQ_DEV_SQ_ZERO)
        assert np.array_equal(G.host(e4), want) and e4_exp.item() == p and total.item() == int(want.astype(np.int64).sum())
    assert np.array_equal(G.host(dump), acc)


def test_halves_and_neighbours_of_halves_in_shortened_groups():
    """A 1x1 layer whose sums are set one by one: multiples of half a code step, one below and one above, beside a sum that fixes the
    step and groups short enough to be cut by several numbers of bits."""
    c = 16
    top = 127 * 127 * c   # the largest sum of 16 products: 258,064 -> a step of 2^11
    n = 4096
    e3 = np.zeros((1, 1, n, c), np.int8)
    w = np.zeros((c, 1, 1, c), np.int8)
    w[0], w[1], w[2] = 127, 1, 0
    w[2, 0, 0, :8] = 127   # (error channel 2 reaches half of the columns)
    rng = np.random.default_rng(5)
    e3[0, 0, :, 0] = rng.integers(-127, 128, n)
    e3[0, 0, :, 1] = rng.integers(-127, 128, n)
    e3[0, 0, :, 2] = rng.integers(-127, 128, n)
    w[3:] = 127
    e3[0, 0, ::64, :] = 127   # (every 64th pixel: the largest sums)
    d = oracle.ConvDesc(1, 1, n, c, c, 1, 1, 1, 0)
    acc = oracle.conv_dgrad_acc(d, e3, w)
    want, p, _ = oracle.sq_int(acc, -16)
    shift = p + 16   # bits that the code drops
    rest = acc.astype(np.int64) & ((1 << shift) - 1)
    assert abs(int(np.abs(acc).max()) - top) < top // 8 and shift >= 8
    assert (rest == 1 << (shift - 1)).any() and (rest == (1 << (shift - 1)) + 1).any() and (rest == (1 << (shift - 1)) - 1).any()
    assert (np.abs(acc).max(axis=-1) >= 1 << 14).any() and (np.abs(acc).max(axis=-1) < 1 << 14).any()
    e4, e4_exp = G.empty(acc.shape, torch.int8), G.zeros(1, torch.int32)
    desc = G.gdesc(d)
    eoq.eoq_conv_dgrad(G.handle(), desc, G.dev(e3), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.dev(w), e4, e4_exp, None, None,
                       G.workspace(desc, eoq.EOQ_PASS_DGRAD))
    assert np.array_equal(G.host(e4), want) and e4_exp.item() == p


@pytest.mark.parametrize("first", [0, 4, 8])
@pytest.mark.parametrize("name", ["patch", "taps, strided", "1x1", "cluster"])
def test_dumped_sums_at_every_alignment(name, first):
    """The int32 sums for a caller, 32 bytes to a store where their buffer starts at a multiple of 32 bytes and 16 where it does not
    (`first` elements behind an allocation): all of them, and nothing beside them."""
    d = GEOMETRIES[name]
    e3 = _errors("large", (d.n, d.ho, d.wo, d.c_out), 40 + first)
    w = synth.int8_uniform((d.c_out, d.kh, d.kw, d.c_in), 2602, first)
    acc = oracle.conv_dgrad_acc(d, e3, w)
    want, p, _ = oracle.sq_int(acc, -9 - 7)
    buf = torch.full((first + acc.size + 8,), 77, dtype=torch.int32, device="cuda:0")
    dump = buf[first:first + acc.size]
    assert dump.data_ptr() % 32 == 4 * first % 32
    e4, e4_exp, desc = G.empty(acc.shape, torch.int8), G.zeros(1, torch.int32), G.gdesc(d)
    eoq.eoq_conv_dgrad(G.handle(), desc, G.dev(e3), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.dev(w), e4, e4_exp, None, dump,
                       G.workspace(desc, eoq.EOQ_PASS_DGRAD))
    assert G.status_clear() == 0
    assert np.array_equal(G.host(dump).reshape(acc.shape), acc) and (G.host(buf[:first]) == 77).all() and (G.host(buf[first + acc.size:]) == 77).all()
    assert np.array_equal(G.host(e4), want) and e4_exp.item() == p


@pytest.mark.parametrize("c_out,cut", [(3000, 12), (20000, 15), (40000, 16), (80000, 17), (100000, 17)])
def test_sums_cut_by_the_most_bits(c_out, cut):
    """Reductions so long that groups lose `cut` bits, up to the 17 that a 32-bit sum can (16 and above need every bit of the count that a
    group carries): halves of a code step, their neighbours, and short groups beside them."""
    c_out = c_out // 16 * 16
    e3, w = np.zeros((1, 1, 40, c_out), np.int8), np.zeros((c_out, 1, 1, 32), np.int8)
    v = np.concatenate([np.array([127, -127, 120, -120, 112, -112, 104, 96, -96, 80, 64, 48, 32, 16, 8, 4]), np.arange(1, 25)])
    e3[0, 0, :, :c_out - 16] = v[:, None]
    e3[0, 0, :, c_out - 1] = np.arange(40) % 3 - 1    # (one beside the multiples)
    ones = 1 << int(np.log2(c_out - 16))
    w[:, 0, 0, 0] = 127
    for i in range(1, 8):   # ones << k in all: sums of v << (log2(ones) + k)
        w[:ones, 0, 0, i] = -(1 << (i - 1)) if i == 3 else 1 << (i - 1)
    w[:, 0, 0, 8:16] = synth.int8_uniform((c_out, 8), 2610, c_out)
    w[:100, 0, 0, 16:] = synth.int8_uniform((100, 16), 2611, c_out)   # the other group of a pixel
    w[c_out - 1] = 1
    d = oracle.ConvDesc(1, 1, 40, 32, c_out, 1, 1, 1, 0)
    acc = oracle.conv_dgrad_acc(d, e3, w)
    largest = np.abs(acc.astype(np.int64)).reshape(-1, 16).max(axis=1)
    assert largest.max().item().bit_length() - 14 == cut and len(set(x.item().bit_length() for x in largest)) > 5
    want, p, _ = oracle.sq_int(acc, -9 - 7)
    step = p - (-9 - 7)   # log2 of a code step
    rest = np.abs(acc.astype(np.int64)) & ((1 << step) - 1)
    for beside in (-1, 0, 1):
        assert (rest == (1 << (step - 1)) + beside).any()
    desc = G.gdesc(d)
    e4, e4_exp, total = G.empty(acc.shape, torch.int8), G.zeros(1, torch.int32), G.zeros(1, torch.int64)
    eoq.eoq_conv_dgrad(G.handle(), desc, G.dev(e3), torch.tensor([-9], dtype=torch.int32, device="cuda:0"), G.dev(w), e4, e4_exp, total, None,
                       G.workspace(desc, eoq.EOQ_PASS_DGRAD))
    assert G.status_clear() == 0
    assert np.array_equal(G.host(e4), want) and e4_exp.item() == p and total.item() == int(want.astype(np.int64).sum())
