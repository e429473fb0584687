"""T+E+B solves with the spin-0 and spin-2 Legendre launches side by side
(graph replay and eager) against the same solve with one launch after the
other (while profiling): the launches write different rows and take the same
shapes, so every bit is the same.
"""
import numpy as np
import pytest

from inputs import configs as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp64", "mixed_tc"])
@pytest.mark.parametrize("nside,lmax,nb", [(8, 16, 1), (32, 64, 3), (48, 101, 9)])
def test_overlap_changes_no_bit(mode, nside, lmax, nb):
    from paper_2306_15511_gb300 import Plan
    cl = C.cl_damped(lmax)
    cl = np.stack([cl, 0.05 * cl, 5e-5 * cl, 0.3 * np.sqrt(0.05) * cl])
    bl = C.gauss_beam(lmax, 1.5 * np.pi / lmax)
    z, _ = C.pixel_centres(nside)
    rng = np.random.default_rng(nside + nb)
    ninv = np.where(np.abs(z) < 0.2, 0.0, rng.uniform(0.5, 1.5, z.size) / 400.0)
    ninv = np.stack([ninv, 0.5 * ninv])
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    d, w2 = dev(rng.normal(size=(nb, 3, z.size))), dev(rng.normal(size=(nb, 3, z.size)))
    P = (lmax + 1) * (lmax + 2) // 2
    w1 = dev(rng.normal(size=(nb, 3, P)) + 1j * rng.normal(size=(nb, 3, P)))
    plan = Plan(nside=nside, lmax=lmax, max_batch=nb, spin2=True)

    def solve(**kw):
        out = plan.cg_sample(cl, bl, dev(ninv), d, w1, w2, tol=1e-7, maxiter=24, mode=mode,
                             allow_not_converged=True, **kw)
        return (out[0] if isinstance(out, tuple) else out).cpu()
    ref = solve(profile=True)
    for kw in (dict(), dict(graphs=False), dict()):
        assert torch.equal(solve(**kw), ref)
