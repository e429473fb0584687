"""Ring stage over transform lengths: every power of two up to 8192 and its
neighbours (Bluestein rings), aliased (n < 2 l_max) and not, with and without
an equator ring, against the oracle.  Few rings, so each length is cheap.

Tolerances as in the transforms' parity tests: relative L2 1e-10 in FP64 (the
synthesis, the transpose and the fused stage of the operator), 1e-5 in FP32.
"""
import numpy as np
import pytest

from oracle import sht as osht
from oracle import solver as osol
from tests._util import rand_alm, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = ([(7, n, 20) for n in (1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33)] +
         [(6, n, 40) for n in (63, 64, 65, 96, 127, 128, 129, 255, 256, 257, 500, 512, 513)] +
         [(5, n, 300) for n in (511, 600, 601, 1000, 1024, 1025)] +
         [(4, n, 9) for n in (2047, 2048, 2049, 4095, 4096, 8192)] +
         [(4, n, 1100) for n in (1024, 2048, 2199, 2200)])


@pytest.mark.parametrize("nring,nphi,L", SIZES)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_ring_lengths(nring, nphi, L, prec):
    from paper_2306_15511_gb300 import Plan
    nb = 3
    plan, g = Plan(gauss=(nring, nphi), lmax=L, max_batch=nb), osht.gauss_legendre(nring, nphi)
    rng = np.random.default_rng(nphi + L)
    ct, rt = (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)
    tol = 1e-10 if prec == "fp64" else max(1e-5, 3.0 * 2.0 ** -24 * L)
    a, m = rand_alm(L, rng, (nb,)), rng.normal(size=(nb, g.npix))
    s = plan.alm2map(torch.tensor(a, dtype=ct, device="cuda")).cpu().numpy()
    t = plan.alm2map_adjoint(torch.tensor(m, dtype=rt, device="cuda")).cpu().numpy()
    for b in range(nb):
        assert rel_l2(s[b], osht.alm2map(g, L, a[b])) < tol
        assert rel_l2(t[b], osht.alm2map_adjoint(g, L, m[b])) < tol
    if prec == "fp64":
        cl, bl = 1.0 / (1.0 + np.arange(L + 1.0)), np.linspace(1.0, 0.5, L + 1)
        ninv = rng.uniform(0.0, 2.0, g.npix)
        prob = osol.Problem(g, L, cl, bl, ninv)
        y = plan.apply_operator(cl, bl, torch.tensor(ninv, device="cuda"),
                                torch.tensor(a[:, None], device="cuda")).cpu().numpy()
        for b in range(nb):
            assert rel_l2(y[b, 0], prob.matvec(a[b][None])[0]) < tol
