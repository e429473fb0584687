"""FP64 Legendre sums on small grids (synthesis: a warp per 32-l segment;
transpose: two groups of threads per CTA) around the segments, the 32-pair
stages and the largest l_max that takes them, against the oracle.

Tolerance: the FP64 bound of the transforms' parity tests, relative L2 1e-10.
"""
import numpy as np
import pytest

from oracle import sht as osht
from tests._util import rand_alm, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,L", [(1, 2), (8, 31), (15, 32), (16, 33), (17, 64), (32, 65), (33, 96), (64, 128),
                                     (64, 151), (64, 152)])
@pytest.mark.parametrize("nb", [1, 2, 3, 5, 9])
def test_small_grids(nside, L, nb):
    from paper_2306_15511_gb300 import Plan
    plan, g = Plan(nside=nside, lmax=L, max_batch=nb, spin2=True), osht.healpix(nside)
    rng = np.random.default_rng(100 * nb + L)
    a0, a2 = rand_alm(L, rng, (nb,)), rand_alm(L, rng, (nb, 2))
    m0, m2 = rng.normal(size=(nb, g.npix)), rng.normal(size=(nb, 2, g.npix))
    dev = lambda x: torch.tensor(x, device="cuda")  # noqa: E731
    s0 = plan.alm2map(dev(a0)).cpu().numpy()
    s2 = plan.alm2map(dev(a2), spin=2).cpu().numpy()
    t0 = plan.alm2map_adjoint(dev(m0)).cpu().numpy()
    t2 = plan.alm2map_adjoint(dev(m2), spin=2).cpu().numpy()
    for b in {0, nb // 2, nb - 1}:
        assert rel_l2(s0[b], osht.alm2map(g, L, a0[b])) < 1e-10
        assert rel_l2(s2[b], np.stack(osht.alm2map_spin2(g, L, a2[b, 0], a2[b, 1]))) < 1e-10
        assert rel_l2(t0[b], osht.alm2map_adjoint(g, L, m0[b])) < 1e-10
        assert rel_l2(t2[b], np.stack(osht.alm2map_spin2_adjoint(g, L, m2[b, 0], m2[b, 1]))) < 1e-10
