"""Row-block forms of the Kaczmarz sweep on the GPU (launch forms 4 and 5 of amg_kaczmarz_form)."""
import numpy as np
import pytest
import torch

from paper_1308_5992_gb300 import wilson_amg as W
from oracle import oracle as O
from wl_inputs import workload, cgauss

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PARAMS = [1 | 1 << 8, 2 | 1 << 8, 4 | 1 << 8, 8 | 1 << 8, 8 | 2 << 8]


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


def f32(a):
    return a.astype(np.complex64).astype(np.complex128)


@pytest.fixture(scope="module")
def hier(tmp_path_factory):
    from oracle.hierfile import write_hierarchy
    out = {}
    # fine grids 64, 128 and 256, coarse levels of side 64, 32 and (deep) 16
    for name, blocks in (("T64", [2, 2]), ("T128", [2, 2, 2]), ("deep", [2, 2, 2]), ("wide", [4, 4])):
        w = workload({"deep": "T64", "wide": "S02"}.get(name, name))
        more = dict(mu1=1, mu2=1) if name == "wide" else {}  # the oracle's setup of 256 x 256 is slow
        h = O.Hierarchy.setup(w["N"], w["U"], w["m"], O.setup_params(blocks, k_r=w["k"], k_e=w["k"], seed=w["seed"],
                                                                     **more))
        path = str(tmp_path_factory.mktemp("rows") / (name + ".wlh"))
        write_hierarchy(path, h)
        out[name] = (h, W.wilson_create(T(w["U"]), w["N"], w["m"]), path)
    return out


@pytest.mark.parametrize("name", ["T64", "T128"])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 5, 17])
def test_row_block_sweep(hier, name, nrhs):
    """Two sweeps against the oracle's tile order, every chunk of right-hand sides (ragged ones
    too), to the bound of the other FP32 forms (1e-6 from the FP32 values of the inputs)."""
    h, op, path = hier[name]
    amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, kacz_order=1, precision=W.WL_FP32))
    for l in range(h.L - 1):
        if h.Nl[l] < 64:
            continue
        n = h.n(l)
        x0 = f32(0.1 * np.stack([cgauss(410 + l, r, n) for r in range(nrhs)]))
        r0 = f32(np.stack([cgauss(420 + l, r, n) for r in range(nrhs)]))
        ref = [h.kaczmarz(l, x0[r], r0[r], order=O.ORDER_TILE, sweeps=2) for r in range(nrhs)]
        xr, rr = np.stack([a for a, _ in ref]), np.stack([b for _, b in ref])
        for param in PARAMS:
            xg, rg = T(x0), T(r0)
            W.amg_kaczmarz_form(amg, l, xg, rg, nrhs, 2, W.WL_FP32, 4, param)
            assert rel(xg.cpu().numpy(), xr) <= 1e-6 and rel(rg.cpu().numpy(), rr) <= 1e-6, (l, param)
    amg.close()


@pytest.mark.parametrize("prec", [W.WL_FP32, W.WL_FP32_BF16])
def test_row_block_sweep_relaxed(hier, prec):
    """omega = 0.8 and BF16-stored stencils, against the tile kernel on the same stored numbers
    (each within 1e-6 of the exact sweep, so 2e-6 of each other)."""
    h, op, path = hier["T64"]
    amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, kacz_order=1, precision=prec, omega=0.8))
    n, nrhs = h.n(0), 3
    x0 = f32(0.1 * np.stack([cgauss(430, r, n) for r in range(nrhs)]))
    r0 = f32(np.stack([cgauss(440, r, n) for r in range(nrhs)]))
    xa, ra, xb, rb = T(x0), T(r0), T(x0), T(r0)
    W.amg_kaczmarz(amg, 0, xa, ra, nrhs, 2, prec)
    W.amg_kaczmarz_form(amg, 0, xb, rb, nrhs, 2, prec, 4, 4 | 1 << 8)
    assert rel(xb.cpu().numpy(), xa.cpu().numpy()) <= 2e-6 and rel(rb.cpu().numpy(), ra.cpu().numpy()) <= 2e-6
    amg.close()


def test_row_block_form_refused(hier):
    """FP64 sweeps, the 16-colour ordering and unknown chunks have no row-block form."""
    h, op, path = hier["T64"]
    z = T(np.zeros((1, h.n(0)), dtype=complex))
    for order, prec, param in ((1, W.WL_FP64, 1 | 1 << 8), (0, W.WL_FP32, 1 | 1 << 8), (1, W.WL_FP32, 3 | 1 << 8)):
        amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, kacz_order=order))
        with pytest.raises(W.WilsonAMGError):
            W.amg_kaczmarz_form(amg, 0, z, z.clone(), 1, 1, prec, 4, param)
        amg.close()


@pytest.mark.parametrize("nrhs", [1, 5])
def test_small_level_sweeps(hier, nrhs):
    """The one-launch form on the 32x32 and 16x16 levels: three sweeps against the oracle's colour
    order (1e-6 as above), and BF16-stored against the per-colour launches."""
    h, op, path = hier["deep"]
    assert h.Nl == [64, 32, 16, 8]
    amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, precision=W.WL_FP32))
    for l in (1, 2):
        n = h.n(l)
        x0 = f32(0.1 * np.stack([cgauss(450 + l, r, n) for r in range(nrhs)]))
        r0 = f32(np.stack([cgauss(460 + l, r, n) for r in range(nrhs)]))
        ref = [h.kaczmarz(l, x0[r], r0[r], order=O.ORDER_COLOUR, sweeps=3) for r in range(nrhs)]
        xr, rr = np.stack([a for a, _ in ref]), np.stack([b for _, b in ref])
        xg, rg = T(x0), T(r0)
        W.amg_kaczmarz_form(amg, l, xg, rg, nrhs, 3, W.WL_FP32, 5, 0)
        assert rel(xg.cpu().numpy(), xr) <= 1e-6 and rel(rg.cpu().numpy(), rr) <= 1e-6, l
        xa, ra, xb, rb = T(x0), T(r0), T(x0), T(r0)
        W.amg_kaczmarz_form(amg, l, xa, ra, nrhs, 3, W.WL_FP32_BF16, 0, 0)
        W.amg_kaczmarz_form(amg, l, xb, rb, nrhs, 3, W.WL_FP32_BF16, 5, 0)
        assert rel(xb.cpu().numpy(), xa.cpu().numpy()) <= 2e-6 and rel(rb.cpu().numpy(), ra.cpu().numpy()) <= 2e-6, l
    z = T(np.zeros((1, h.n(0)), dtype=complex))
    with pytest.raises(W.WilsonAMGError):  # a 64x64 level
        W.amg_kaczmarz_form(amg, 0, z, z.clone(), 1, 1, W.WL_FP32, 5, 0)
    amg.close()


@pytest.mark.parametrize("name", ["T128", "deep", "wide"])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 9])
def test_fp64_ring_sweeps(hier, name, nrhs):
    """The FP64 forms on every 16-colour level (256x256 down to 16x16; every lane split
    of the inner products, ragged chunks of right-hand sides) against the oracle, to the bound of
    the other FP64 forms (1e-13 for one sweep, two here: 2e-13)."""
    h, op, path = hier[name]
    for omega in (1.0, 0.8):
        amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, omega=omega))
        for l in range(h.L - 1):
            n = h.n(l)
            x0 = 0.1 * np.stack([cgauss(470 + l, r, n) for r in range(nrhs)])
            r0 = np.stack([cgauss(480 + l, r, n) for r in range(nrhs)])
            xg, rg = T(x0), T(r0)
            W.amg_kaczmarz_form(amg, l, xg, rg, nrhs, 2, W.WL_FP64, 6, 0)
            outs = [(xg, rg)]
            for param in [1] * (h.Nl[l] in (32, 64)) + [2] * (h.Nl[l] >= 32 and nrhs <= 4):  # clusters
                xc, rc = T(x0), T(r0)
                W.amg_kaczmarz_form(amg, l, xc, rc, nrhs, 2, W.WL_FP64, 6, param)
                outs.append((xc, rc))
            if omega == 1.0:
                ref = [h.kaczmarz(l, x0[r], r0[r], order=O.ORDER_COLOUR, sweeps=2) for r in range(nrhs)]
                xr, rr = np.stack([a for a, _ in ref]), np.stack([b for _, b in ref])
            else:
                xa, ra = T(x0), T(r0)
                W.amg_kaczmarz_form(amg, l, xa, ra, nrhs, 2, W.WL_FP64, 0, 0)
                xr, rr = xa.cpu().numpy(), ra.cpu().numpy()
            for xg, rg in outs:
                assert rel(xg.cpu().numpy(), xr) <= 2e-13 and rel(rg.cpu().numpy(), rr) <= 2e-13, (l, omega)
        amg.close()
    amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, kacz_order=1))
    z = T(np.zeros((1, h.n(0)), dtype=complex))
    with pytest.raises(W.WilsonAMGError):  # a tile-ordered level
        W.amg_kaczmarz_form(amg, 0, z, z.clone(), 1, 1, W.WL_FP64, 6, 0)
    amg.close()


@pytest.mark.parametrize("nrhs", [1, 3, 7])
def test_small_batch_cycle(hier, nrhs):
    """Cycles whose stencil applies and restrictions take several lanes a site (cells of 2, levels
    64 to 8), V and W, against the oracle: FP64 1e-12, FP32 1e-5 as for the other batches."""
    h, op, path = hier["deep"]
    n = h.n(0)
    f = np.stack([cgauss(495, q, n) for q in range(nrhs)])
    for cycle in (W.WL_CYCLE_V, W.WL_CYCLE_W):
        ref = np.stack([h.cycle(f[q], nu1=2, nu2=2, gamma=cycle + 1) for q in range(nrhs)])
        for prec, tol in ((W.WL_FP64, 1e-12), (W.WL_FP32, 1e-5)):
            amg = W.amg_import(op, path, W.amg_params_default(zero_guess=1, cycle=cycle, precision=prec))
            xg = torch.zeros_like(T(f))
            W.amg_cycle(amg, T(f), xg, nrhs, prec)
            assert rel(xg.cpu().numpy(), ref) <= tol, (cycle, prec)
            amg.close()
