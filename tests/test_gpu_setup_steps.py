"""Steps of the GPU setup: the Galerkin product and the coarsest inverse."""
import numpy as np
import pytest
import torch

from paper_1308_5992_gb300 import wilson_amg as W
from oracle import oracle as O
from wl_inputs import workload, cgauss

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("blocks", [[2, 2], [4], [4, 2], [2, 4], [2, 2, 2]])
def test_galerkin_and_coarsest(blocks, tmp_path):
    """A set-up hierarchy of a 64x64 field, cells of 2 and 4, coarsest grids of 16 and 8: every
    coarse operator is P^H A P of the exported interpolation (random vectors, 1e-12 of the largest
    entry: sums of at most 9 * 49 products and the oracle's own), and the coarsest solve is the
    oracle's dense LU solve (1e-11, as for the other hierarchies)."""
    from oracle.hierfile import read
    w = workload("T64")
    op = W.wilson_create(T(w["U"]), w["N"], w["m"])
    p = W.amg_params_default(k_r=6, k_e=6, seed=5, block=blocks, levels=len(blocks) + 1)
    amg = W.amg_setup(op, p)
    path = str(tmp_path / "h.wlh")
    W.amg_export(amg, path)
    d = read(path)
    h = O.Hierarchy.from_arrays(w["N"], w["U"], d["m"], d["Nl"], d["Bl"], d["Pw"], d["As"])
    for l in range(h.L - 1):
        x = cgauss(510 + l, 0, h.n(l + 1))
        ref = h.restrict(l, h.apply(l, h.prolong(l, x, np.zeros(h.n(l), dtype=complex))))
        got = h.apply(l + 1, x)
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max(), l
    n = h.n(h.L - 1)
    f = np.stack([cgauss(520, q, n) for q in range(2)])
    xg = torch.zeros_like(T(f))
    W.amg_coarsest(amg, T(f), xg, 2)
    ref = np.stack([h.coarsest_solve(f[q]) for q in range(2)])
    assert np.abs(xg.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    amg.close()
    op.close()
