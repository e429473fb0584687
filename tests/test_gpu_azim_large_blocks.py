"""Azimuthal blocks of more than 512 rows (the application stages 512 columns at
a time and sums eight column ranges; the factorization has more than ten block
columns), a few m against NumPy's inverse of the oracle's blocks.

Tolerances, from the block A of n rows (u = 2^-53, v = 2^-24):
- FP64: 4 n u cond(A), relative to the largest entry of the result (Cholesky
  factorization and inverse, and NumPy's own);
- FP32 application: relative to | |A^-1| |r| |, (n / 8 + 8) v (an eighth of the
  columns in order, then three additions; entries of A^-1 and r rounded).
"""
import numpy as np
import pytest

from inputs import configs as C
from oracle import sht as osht
from oracle import solver as osol

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NSIDE, L, LB = 140, 528, 525


def problem(ncomp):
    rng = np.random.default_rng(7)
    cl = C.cl_damped(L)
    if ncomp == 3:
        cl = np.stack([cl, 0.05 * cl, 5e-5 * cl, 0.3 * np.sqrt(0.05) * cl])
    bl = C.gauss_beam(L, 1.5 * np.pi / L)
    z, _ = C.pixel_centres(NSIDE)
    ninv = np.where(np.abs(z) < 0.2, 0.0, rng.uniform(0.5, 1.5, z.size) / 400.0)
    if ncomp == 3:
        ninv = np.stack([ninv, 0.5 * ninv])
    return cl, bl, ninv


def blocks(ncomp, ms):
    cl, bl, ninv = problem(ncomp)
    prob = osol.Problem(osht.healpix(NSIDE), L, cl, bl, ninv)
    wsum = osol.ring_sum_weights(prob)
    return {m: osol.azimuthal_te_block(prob, m, LB, wsum)[1] for m in ms}


@pytest.mark.parametrize("ncomp,ms", [(1, (0, 12, 14)), (3, (0, 1, 12, 14, 270, 510))])
def test_large_blocks(ncomp, ms):
    from paper_2306_15511_gb300 import Plan
    nb = 5
    cl, bl, ninv = problem(ncomp)
    rng = np.random.default_rng(11)
    P = (L + 1) * (L + 2) // 2
    r = rng.normal(size=(nb, ncomp, P)) + 1j * rng.normal(size=(nb, ncomp, P))
    all_m, all_l = osht.ms_of(L), osht.ls_of(L)
    r[..., all_m == 0] = r[..., all_m == 0].real
    plan = Plan(nside=NSIDE, lmax=L, max_batch=nb, spin2=ncomp == 3)
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731

    def apply(n, fp32):   # the first n realizations
        return plan.precond_apply(cl, bl, dev(ninv), dev(r[:n]), precond="azim", block_lmax=LB,
                                  fp32=fp32).cpu().numpy()

    got = {(n, fp32): apply(n, fp32) for n in (1, nb) for fp32 in (False, True)}
    comps = range(min(ncomp, 2))
    for m, A in blocks(ncomp, ms).items():
        n = A.shape[0]
        Ai = np.linalg.inv(A)
        tol64 = 4 * n * 2.0 ** -53 * np.linalg.cond(A)
        assert tol64 < 1e-7
        rows = np.where((all_m == m) & (all_l <= LB))[0]
        for (nr, fp32), z in got.items():
            for b in range(nr):
                v = np.concatenate([r[b, c, rows] for c in comps])
                w = np.concatenate([z[b, c, rows] for c in comps])
                for part in (np.real, np.imag):
                    ref = Ai @ part(v)
                    err = np.abs(part(w) - ref)
                    if fp32:
                        scale = np.linalg.norm(np.abs(Ai) @ np.abs(part(v)))
                        assert np.linalg.norm(err) <= (n / 8 + 8) * 2.0 ** -24 * scale, (m, nr, b)
                    else:
                        assert err.max() <= tol64 * np.abs(ref).max(), (m, nr, b)
