"""Cycles of one hierarchy at changing widths, and which sweep forms they take."""
import numpy as np
import pytest
import torch

from paper_1308_5992_gb300 import wilson_amg as W
from wl_inputs import workload, cgauss

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.fixture(scope="module")
def c2():
    w = workload("C2")
    op = W.wilson_create(T(w["U"]), w["N"], w["m"])
    return w, op


def setup(c2, **params):
    w, op = c2
    p = W.amg_params_default(k_r=w["k"], k_e=w["k"], seed=w["seed"], zero_guess=1, setup_mu=w["setup_mu"],
                             block=w["blocks"], levels=len(w["blocks"]) + 1, **params)
    return W.amg_setup(op, p)


def cycle(amg, f, prec):
    x = torch.zeros_like(f)
    W.amg_cycle(amg, f, x, f.shape[0], prec)
    return x


def test_cycles_at_changing_widths(c2):
    """One hierarchy used at widths (and precisions) that grow and shrink gives each width the
    bits it gave at first."""
    amg = setup(c2)
    n = amg.n(0)
    f = T(np.stack([cgauss(700, r, n) for r in range(16)]))
    first = {}
    for nrhs, prec in ((9, 0), (16, 1), (9, 0), (5, 0), (9, 0), (16, 0), (5, 0), (9, 0), (16, 1)):
        x = cycle(amg, f[:nrhs].contiguous(), prec)
        assert torch.equal(x, first.setdefault((nrhs, prec), x)), (nrhs, prec)
    amg.close()


@pytest.mark.parametrize("prec", [W.WL_FP32, W.WL_FP32_BF16])
@pytest.mark.parametrize("nrhs", [1, 3, 11])
def test_row_block_chunks_agree_bitwise(c2, prec, nrhs):
    """The tuner may choose any chunk of the row-block form: a right-hand side's numbers do not
    depend on it."""
    amg = setup(c2, kacz_order=1, precision=prec)
    n = amg.n(0)
    x0, r0 = (np.stack([cgauss(s, r, n) for r in range(nrhs)]).astype(np.complex64).astype(complex) for s in (710, 720))
    outs = []
    for param in (1 | 1 << 8, 2 | 1 << 8, 4 | 1 << 8, 8 | 1 << 8, 8 | 2 << 8):
        x, r = T(x0), T(r0)
        W.amg_kaczmarz_form(amg, 0, x, r, nrhs, 2, prec, 4, param)
        outs.append((x, r))
        assert torch.equal(x, outs[0][0]) and torch.equal(r, outs[0][1]), param
    amg.close()


@pytest.mark.parametrize("prec,order", [(W.WL_FP64, 0), (W.WL_FP64, 1), (W.WL_FP32, 1), (W.WL_FP32_BF16, 1)])
def test_two_hierarchies_agree_bitwise(c2, prec, order):
    """The same cycle of two hierarchies, each tuned on its own, gives the same bits."""
    a, b = (setup(c2, kacz_order=order, precision=prec) for _ in range(2))
    f = T(np.stack([cgauss(730, r, a.n(0)) for r in range(6)]))
    for nrhs in (1, 2, 6):
        assert torch.equal(cycle(a, f[:nrhs].contiguous(), prec), cycle(b, f[:nrhs].contiguous(), prec)), nrhs
    a.close()
    b.close()


@pytest.mark.parametrize("prec,order", [(W.WL_FP64, 0), (W.WL_FP32, 1)])
def test_pinned_cycle_forms_give_the_same_bits(c2, prec, order):
    """The forms that amg_cycle_form reports, pinned on another hierarchy, give the same bits; in
    FP64 every row-block form gives the cycle to rounding (1e-12, as the other cycles)."""
    a, b = (setup(c2, kacz_order=order, precision=prec) for _ in range(2))
    f = T(np.stack([cgauss(740, r, a.n(0)) for r in range(2)]))
    x = cycle(a, f, prec)
    L = len(c2[0]["blocks"])
    for l in range(L):
        W.amg_pin_sweep_form(b, l, 2, prec, *W.amg_cycle_form(a, l, 2, prec)[:2])
    assert torch.equal(cycle(b, f, prec), x)
    b.close()
    if prec == W.WL_FP64:
        for param in (0, 2):
            c = setup(c2)
            W.amg_pin_sweep_form(c, 0, 2, prec, 6, param)
            assert float((cycle(c, f, prec) - x).abs().max() / x.abs().max()) <= 1e-12, param
            c.close()
    a.close()


@pytest.mark.parametrize("N,nrhs", [(16, 1), (16, 3), (32, 5)])
def test_residual_of_small_lattices(O, N, nrhs):
    """The FP64 residual of few site-vectors (a hop on two lanes each) on the smallest lattices
    against the oracle's operator; relative to 1e-12 (sums of 10 terms of order one, 1e-15 each)."""
    U = np.exp(2j * np.pi * np.random.default_rng(5).random((2, N, N)))
    op = W.wilson_create(T(U), N, 0.3)
    amg = W.amg_setup(op, W.amg_params_default(zero_guess=1, block=[2], levels=2, k_r=4, k_e=4, max_restarts=1, fgmres_m=1))
    bh = np.stack([cgauss(750, r, N * N) for r in range(nrhs)])
    x = torch.zeros_like(T(bh))
    _, info = W.amg_fgmres(amg, T(bh), x, nrhs, 1e-14)
    for r in range(nrhs):
        res = np.linalg.norm(bh[r] - O.dhat_apply(N, U, 0.3, x[r].cpu().numpy())) / np.linalg.norm(bh[r])
        assert abs(info[r]["true_relres"] - res) <= 1e-12 * res, (r, info[r], res)
    amg.close()
