"""Every shape that the autotuner may choose for the FP64 and FP32 CUDA-core
Legendre sums, forced one after the other (SHTG_TUNE_FORCE, read once per
process, so the transforms run in child processes: this file run as a program).

Synthesis: every bit as with the first shape.  Transposes sum in other orders:
relative L2 from the first shape within twice the transforms' parity bounds
(each side is within one of the exact value): 1e-10 in FP64, max(1e-5, 3 u l_max)
in FP32 (u = 2^-24).
"""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# ring pairs up to 256 and up to 512 (the FP64 spin-0 transpose then has four and
# two shapes), more CTAs than SMs; ragged along l and along the pairs
SIZES = [(50, 165), (151, 170)]
MAPS = (1, 2, 3, 5)   # the shapes follow the number of maps


def transforms(path):
    import torch

    from paper_2306_15511_gb300 import Plan
    out = {}
    for nside, lmax in SIZES:
        plan = Plan(nside=nside, lmax=lmax, max_batch=max(MAPS), spin2=True)
        gen = torch.Generator(device="cuda").manual_seed(nside)
        for bits, real, cplx in ((64, torch.float64, torch.complex128), (32, torch.float32, torch.complex64)):
            for nb in MAPS:
                for spin in (0, 2):
                    lead = (nb, 2) if spin else (nb,)
                    m = torch.randn(*lead, plan.npix, dtype=torch.float64, device="cuda", generator=gen).to(real)
                    a = torch.randn(*lead, plan.nalm, dtype=torch.complex128, device="cuda", generator=gen).to(cplx)
                    key = f"{bits} {nside} {lmax} {nb} {spin}"
                    out[key + " adjoint"] = plan.alm2map_adjoint(m, spin=spin).cpu().numpy()
                    out[key + " synthesis"] = plan.alm2map(a, spin=spin).cpu().numpy()
        plan.close()
    np.savez(path, **out)


def child(tmp_path, shape):
    path = str(tmp_path / "out.npz")
    subprocess.run([sys.executable, os.path.abspath(__file__), path], check=True, cwd=ROOT, timeout=300,
                   env={**os.environ, "SHTG_TUNE_FORCE": str(shape)})
    with np.load(path) as z:
        return {k: z[k] for k in z.files}


@pytest.fixture(scope="module")
def first(tmp_path_factory):
    return child(tmp_path_factory.mktemp("first"), 0)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [1, 2, 3])
def test_every_shape(tmp_path, first, shape):
    got = child(tmp_path, shape)
    assert got.keys() == first.keys()
    for k in first:
        if k.endswith("synthesis"):
            assert np.array_equal(got[k], first[k]), k
        else:
            lmax = int(k.split()[2])
            tol = 2e-10 if k.startswith("64") else 2 * max(1e-5, 3 * 2.0 ** -24 * lmax)
            assert np.linalg.norm(got[k] - first[k]) <= tol * np.linalg.norm(first[k]), k


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    transforms(sys.argv[1])
