"""Kernel variants at the sizes where they change over or end in a remainder, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import eoq, synth
import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 32767, 32769, 262144, 262145, 262144 + 8192 + 3])
@pytest.mark.parametrize("mode", [eoq.EOQ_Q, eoq.EOQ_CQ, eoq.EOQ_SQ])
def test_quantize_float_sizes(n, mode):
    """SQ in one cluster of 1 to 8 blocks up to 262,144 floats, tiles of 8,192 beyond; remainders modulo 4."""
    x = synth.normal_f32(n, 1500, n)
    c, p, _ = oracle.quantize_f32(mode, x)
    out, ex = G.zeros(n, torch.int16 if mode == eoq.EOQ_Q else torch.int8), G.zeros(1, torch.int32)
    for _ in range(2):  # twice: the reduction cell must come back clean
        eoq.eoq_quantize(G.handle(), mode, G.dev(x), True, None, n, out, ex)
        assert G.status_clear() == 0
        assert np.array_equal(G.host(out).astype(np.int32), np.clip(c, -32768, 32767)) and ex.item() == (p if mode == eoq.EOQ_SQ else -7)


@pytest.mark.parametrize("shape,c_dst,margin", [((2, 5, 31, 3), 16, 0), ((1, 9, 257, 3), 8, 5), ((3, 3, 40, 20), 48, 1)])
def test_quantize_image_rows(shape, c_dst, margin):
    """Rows that end inside a block, rows wider than a block, and more than four source channels in several groups."""
    n, h, w, c = shape
    x = synth.normal_f32(shape, 1510, w)
    codes, p, _ = oracle.quantize_f32(eoq.EOQ_SQ, x.reshape(-1))
    want = np.zeros((n, h, w + 2 * margin, c_dst), np.int8)
    want[:, :, margin:margin + w, :c] = codes.reshape(shape)
    out, ex = torch.full(want.shape, 77, dtype=torch.int8, device="cuda:0"), G.zeros(1, torch.int32)
    eoq.eoq_quantize_image(G.handle(), G.dev(x), n, h, w, c, c_dst, margin, out, ex)
    assert G.status_clear() == 0 and np.array_equal(G.host(out), want) and ex.item() == p


@pytest.mark.parametrize("lr", [(1, -3), (37, -8), (255, 2), (1, -30)])
@pytest.mark.parametrize("stochastic", [False, True])
def test_update_one_block_per_tensor(lr, stochastic):
    """Tensors of at most 65,536 codes take one block each; two consecutive steps of a device-resident counter."""
    sizes = [1, 15, 16, 2304, 16384 + 7, 65536]
    ws = [synth.int8_uniform(n, 1520, i) for i, n in enumerate(sizes)]
    gs = [synth.normal_codes(n, 1521, i, std_codes=40) for i, n in enumerate(sizes)]
    gs[1][:] = 0
    pgs = [-9 - i for i in range(len(sizes))]
    w_d, step = [G.dev(w) for w in ws], torch.tensor([5], dtype=torch.int64, device="cuda:0")
    g_d, p_d = [G.dev(g) for g in gs], [G.dev(np.array([p], dtype=np.int32)) for p in pgs]
    for k in range(2):
        eoq.eoq_update_dev(G.handle(), w_d, g_d, p_d, lr[0], lr[1], eoq.EOQ_ROUND_STOCHASTIC if stochastic else eoq.EOQ_ROUND_RNE, 11, step)
        assert G.status_clear() == (eoq.EOQ_DEV_SQ_ZERO) and step.item() == 6 + k
        for i in range(len(sizes)):
            ws[i], _, _ = oracle.update(ws[i], gs[i], pgs[i], lr[0], lr[1], stochastic=stochastic, seed=11, step=5 + k, tensor_id=i)
            assert np.array_equal(G.host(w_d[i]).astype(np.int32), ws[i]), (k, i)
