"""The self-test of the bounded waits runs the wait of the GEMM kernels, and a handle is usable behind a wait that ran out."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2105_13890_b200 import build, eoq, synth


def source(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return f.read()


def test_self_test_runs_the_wait_that_the_gemms_use():
    """One definition of wait_bar; every GEMM kernel's file and the self-test's kernel call it."""
    names = [n for n in os.listdir(build.CSRC) if n.endswith((".cu", ".cuh"))]
    assert [n for n in names if re.search(r"bool wait_bar\(", source(n))] == ["eoq_epilogue.cuh"]
    gemms = [n for n in build.SOURCES if re.match(r"eoq_(igemm|wgrad)", n)]
    assert len(gemms) == 6 and all("wait_bar" in source(n) for n in gemms)
    text = source("eoq_elementwise.cu")
    kernel = text[text.index("wait_self_test_kernel("):]
    kernel = kernel[:kernel.index("\n}\n")]
    assert "wait_bar(" in kernel and "wait_bar<64>(" in kernel and "RoleCtx" in kernel


@pytest.mark.gpu
def test_cells_are_clear_behind_a_wait_that_ran_out():
    """The self-test leaves every reduction cell as a kernel that gave up may; calls that use them then give the oracle's results, and
    those of a handle on which nothing ran out."""
    import gpu_util as G

    n_el = 1 << 20   # (beyond the calls that need no cells)
    e0, mask = synth.normal_codes(n_el, 8600, 1), synth.bits(n_el, 8601, 0)
    b = synth.normal_codes(n_el, 8602, 1)
    x2 = synth.normal_codes(n_el, 8603, 1).astype(np.int16) * 200
    x = synth.normal_f32((n_el,), 8604, 0)
    e3_ref, p3, s1, s2, _ = oracle.err_prescale(e0, -12, mask, x2, 118)
    d_e0, d_b, d_x2, d_x, d_mask = G.dev(e0), G.dev(b), G.dev(x2), G.dev(x), G.dev(G.pack_mask(mask))

    def i32(v):
        return G.dev(np.array([v], dtype=np.int32))

    def results(h):
        out = [G.zeros(n_el, torch.int8) for _ in range(4)]
        exps, sums = [G.zeros(1, torch.int32) for _ in range(4)], [G.zeros(1, torch.int64) for _ in range(4)]
        eoq.eoq_err_prescale(h, d_e0, i32(-12), d_mask, d_x2, n_el, 118, out[0], exps[0], sums[0], sums[1])
        eoq.eoq_aux_join_head(h, d_e0, i32(-12), d_b, i32(-10), d_mask, n_el, out[1], exps[1], sums[2], d_mask, None, i32(100), out[2], exps[2],
                              sums[3])
        eoq.eoq_quantize(h, eoq.EOQ_SQ, d_x, True, None, n_el, out[3], exps[3])
        assert eoq.eoq_last_status(h) == 0
        return [G.host(t) for t in out + exps + sums]

    fresh, h = eoq.eoq_create(0), eoq.eoq_create(0)
    try:
        want = results(fresh)
        for _ in range(2):
            e3 = torch.full((n_el,), 55, dtype=torch.int8, device="cuda:0")
            eoq.eoq_debug_force_wait_timeout(h)
            eoq.eoq_err_prescale(h, d_e0, i32(-12), d_mask, d_x2, n_el, 118, e3, G.zeros(1, torch.int32))
            assert eoq.eoq_last_status(h) == eoq.EOQ_DEV_TIMEOUT
            assert (G.host(e3) == 55).all()
            got = results(h)
            assert all(np.array_equal(a, c) for a, c in zip(got, want))
        assert np.array_equal(got[0], e3_ref) and got[4].item() == p3 and got[8].item() == s1 and got[9].item() == s2
    finally:
        eoq.eoq_destroy(h)
        eoq.eoq_destroy(fresh)
