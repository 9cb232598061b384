"""wl_apply's tiled Dhat kernel on the GPU: both tile sizes, wrap-around and the FP32 rounding."""
import numpy as np
import pytest
import torch

from paper_1308_5992_gb300 import wilson_amg as W
from wl_inputs import metropolis_u1, cgauss

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("N,nrhs", [(16, 1), (16, 5), (32, 1), (32, 160), (64, 40), (256, 3), (512, 1)])
def test_dhat_tile(N, nrhs):
    """Against wl_dhat_apply_noalloc (two launches through global memory), FP64 to 1e-15 and FP32 to
    1e-6 of the largest value; 32 and 64 with the large batches and 512 take the 32 x 16 tiles."""
    op = W.wilson_create(torch.from_numpy(metropolis_u1(N, 6.0, 5, 3)).to(DEV), N, -0.05)
    x = torch.from_numpy(np.stack([cgauss(600 + r, 1, N * N) for r in range(nrhs)])).to(DEV)
    ref, y, y32 = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
    for r in range(nrhs):
        W.wl_dhat_apply_noalloc(op, x[r:r + 1], ref[r:r + 1], 1)
    W.wl_apply(op, W.WL_OP_DHAT, x, y, nrhs, W.WL_FP64)
    W.wl_apply(op, W.WL_OP_DHAT, x, y32, nrhs, W.WL_FP32)
    top = float(ref.abs().max())
    assert float((y - ref).abs().max()) <= 1e-15 * top
    assert float((y32 - ref).abs().max()) <= 1e-6 * top
    op.close()


def test_fp32_rounds_to_nearest():
    """A vector with one non-zero site: its own value comes back as the nearest float exactly (the
    hops out and back cancel), for ties, carries, subnormal and zero floats."""
    N = 16
    op = W.wilson_create(torch.from_numpy(metropolis_u1(N, 6.0, 5, 3)).to(DEV), N, -0.05)
    rng = np.random.RandomState(4)
    vals = list(rng.standard_normal(40) * 10.0 ** rng.randint(-44, 30, 40))
    vals += [1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, 2.0 - 2.0 ** -25, 1.0 + 2.0 ** -24 + 2.0 ** -50, 0.0, -0.0, 1e-46, 7e-46]
    vals += [2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -25), -(2.0 ** -149), 3.0e38, 1.5 * 2.0 ** -149]
    for i, v in enumerate(vals):
        x = torch.zeros(1, N * N, dtype=torch.complex128, device=DEV)
        k = (37 * i) % (N * N)
        x[0, k] = complex(v, -v)
        y = torch.zeros_like(x)
        W.wl_apply(op, W.WL_OP_DHAT, x, y, 1, W.WL_FP32)
        got = complex(y[0, k].item())
        with np.errstate(over="ignore"):
            f = float(np.float32(v))
        assert got.real == f and got.imag == -f, (v, got, f)
    op.close()


@pytest.mark.parametrize("N,nrhs", [(16, 1), (64, 3), (256, 3), (512, 1)])
@pytest.mark.parametrize("prec", [W.WL_FP64, W.WL_FP32])
def test_in_place(N, nrhs, prec):
    """y = x, and y one right-hand side into x: the same bits as a call on separate arrays."""
    op = W.wilson_create(torch.from_numpy(metropolis_u1(N, 6.0, 5, 3)).to(DEV), N, -0.05)
    x = torch.from_numpy(np.stack([cgauss(620 + r, 1, N * N) for r in range(nrhs)])).to(DEV)
    ref = torch.zeros_like(x)
    W.wl_apply(op, W.WL_OP_DHAT, x, ref, nrhs, prec)
    buf = torch.zeros(nrhs + 1, N * N, dtype=torch.complex128, device=DEV)
    for shift in (0, 1):
        buf[:nrhs] = x
        W.wl_apply(op, W.WL_OP_DHAT, buf[:nrhs], buf[shift:shift + nrhs], nrhs, prec)
        assert torch.equal(buf[shift:shift + nrhs], ref)
    op.close()
