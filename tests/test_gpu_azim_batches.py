"""Azimuthal blocks over batch sizes (right-hand sides per pass) and block
sizes around the 32-row blocks of the factorization and the 128-row tiles of
the application: one application against the oracle's.

Tolerances: FP64 application, block rows within 1e-9 of the largest entry (as
the preconditioner's parity test); the FP32 application of the mixed solver,
relative L2 of 1e-5: entries of M^-1 and r rounded to 2^-24, sums of up to
n = 310 terms.
"""
import numpy as np
import pytest

from inputs import configs as C
from oracle import sht as osht
from oracle import solver as osol

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lb", [31, 32, 63, 127, 128, 154])
@pytest.mark.parametrize("nb", [1, 4, 5, 9])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_batches(lb, nb, ncomp):
    from paper_2306_15511_gb300 import Plan
    nside, L = 64, 154
    g = osht.healpix(nside)
    rng = np.random.default_rng(lb + 10 * nb)
    cl = C.cl_damped(L)
    if ncomp == 3:
        cl = np.stack([cl, 0.05 * cl, 5e-5 * cl, 0.3 * np.sqrt(0.05) * cl])
    bl = C.gauss_beam(L, 1.5 * np.pi / L)
    z, _ = C.pixel_centres(nside)
    ninv = np.where(np.abs(z) < 0.2, 0.0, rng.uniform(0.5, 1.5, z.size) / 400.0)
    if ncomp == 3:
        ninv = np.stack([ninv, 0.5 * ninv])
    P = (L + 1) * (L + 2) // 2
    r = rng.normal(size=(nb, ncomp, P)) + 1j * rng.normal(size=(nb, ncomp, P))
    r[..., osht.ms_of(L) == 0] = r[..., osht.ms_of(L) == 0].real
    plan = Plan(nside=nside, lmax=L, max_batch=nb, spin2=ncomp == 3)
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    z64 = plan.precond_apply(cl, bl, dev(ninv), dev(r), precond="azim", block_lmax=lb).cpu().numpy()
    z32 = plan.precond_apply(cl, bl, dev(ninv), dev(r), precond="azim", block_lmax=lb, fp32=True).cpu().numpy()
    ap = osol.azimuthal_precond(osol.Problem(g, L, cl, bl, ninv), lb)
    rows = osht.ls_of(L) <= lb
    for b in range(nb):
        ref = ap(r[b])
        for c in range(min(ncomp, 2)):
            err = np.abs(z64[b, c][rows] - ref[c][rows]).max()
            assert err <= 1e-9 * np.abs(ref[c]).max()
            assert np.linalg.norm(z32[b, c][rows] - ref[c][rows]) <= 1e-5 * np.linalg.norm(ref[c][rows])
