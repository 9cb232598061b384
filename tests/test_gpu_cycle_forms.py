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
