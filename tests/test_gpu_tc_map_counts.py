"""Tensor-core transforms over the number of maps of a call (8 maps per CTA, 16
at spin 0 beyond 8) and l_max around the chunks of 32 l and the flushes of the
accumulators, against the oracle.

Tolerance: the FP32 bound of the transforms' parity tests, relative L2
max(1e-5, 3 u l_max) (u = 2^-24).
"""
import numpy as np
import pytest

from oracle import sht as osht
from tests._util import rand_alm, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,L", [(8, 3), (16, 31), (16, 32), (48, 127), (48, 130), (96, 257), (100, 288)])
@pytest.mark.parametrize("nb", [1, 8, 9, 16, 17])
def test_map_counts(nside, L, nb):
    from paper_2306_15511_gb300 import Plan
    plan, g = Plan(nside=nside, lmax=L, max_batch=nb, spin2=True), osht.healpix(nside)
    rng = np.random.default_rng(100 * nb + L)
    tol = max(1e-5, 3.0 * 2.0 ** -24 * L)
    a0, a2 = rand_alm(L, rng, (nb,)), rand_alm(L, rng, (nb, 2))
    m0, m2 = rng.normal(size=(nb, g.npix)), rng.normal(size=(nb, 2, g.npix))
    cx = lambda x: torch.tensor(x, dtype=torch.complex64, device="cuda")  # noqa: E731
    re = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda")  # noqa: E731
    s0 = plan.alm2map(cx(a0), tensor_cores=True).cpu().numpy()
    s2 = plan.alm2map(cx(a2), spin=2, tensor_cores=True).cpu().numpy()
    t0 = plan.alm2map_adjoint(re(m0), tensor_cores=True).cpu().numpy()
    t2 = plan.alm2map_adjoint(re(m2), spin=2, tensor_cores=True).cpu().numpy()
    for b in {0, nb // 2, nb - 1}:
        assert rel_l2(s0[b], osht.alm2map(g, L, a0[b])) < tol
        assert rel_l2(s2[b], np.stack(osht.alm2map_spin2(g, L, a2[b, 0], a2[b, 1]))) < tol
        assert rel_l2(t0[b], osht.alm2map_adjoint(g, L, m0[b])) < tol
        assert rel_l2(t2[b], np.stack(osht.alm2map_spin2_adjoint(g, L, m2[b, 0], m2[b, 1]))) < tol
