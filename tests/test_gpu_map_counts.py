"""FP64-accurate transforms over the number of maps of a call.

The shapes of the Legendre kernels follow the number of maps (maps per pass,
maps per CTA), so every count from one to a full group and beyond is checked
against the oracle, at sizes with ragged tails along l (segments of 32 and
rows of 128) and along the ring pairs.  Tolerance: the 1e-10 relative L2 of
the FP64 transforms' parity tests.
"""
import numpy as np
import pytest

from oracle import sht as osht
from tests._util import rand_alm, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,L", [(8, 12), (16, 33), (24, 70), (48, 141)])
@pytest.mark.parametrize("nb", [1, 2, 3, 4, 5, 6, 7, 9, 12])
@pytest.mark.parametrize("double_float", [False, True])
def test_map_counts(nside, L, nb, double_float):
    from paper_2306_15511_gb300 import Plan
    plan, g = Plan(nside=nside, lmax=L, max_batch=nb, spin2=True), osht.healpix(nside)
    rng = np.random.default_rng(1000 * nb + L)
    dev = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    a0, a2 = rand_alm(L, rng, (nb,)), rand_alm(L, rng, (nb, 2))
    m0, m2 = rng.normal(size=(nb, g.npix)), rng.normal(size=(nb, 2, g.npix))
    how = dict(double_float=double_float)
    s0 = plan.alm2map(dev(a0), **how).cpu().numpy()
    s2 = plan.alm2map(dev(a2), spin=2, **how).cpu().numpy()
    t0 = plan.alm2map_adjoint(dev(m0), **how).cpu().numpy()
    t2 = plan.alm2map_adjoint(dev(m2), spin=2, **how).cpu().numpy()
    for b in range(nb):
        assert rel_l2(s0[b], osht.alm2map(g, L, a0[b])) < 1e-10
        assert rel_l2(s2[b], np.stack(osht.alm2map_spin2(g, L, a2[b, 0], a2[b, 1]))) < 1e-10
        assert rel_l2(t0[b], osht.alm2map_adjoint(g, L, m0[b])) < 1e-10
        assert rel_l2(t2[b], np.stack(osht.alm2map_spin2_adjoint(g, L, m2[b, 0], m2[b, 1]))) < 1e-10
