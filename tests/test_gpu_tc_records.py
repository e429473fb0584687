"""The tensor-core transforms' operand records live in an optional buffer of the
plan: a plan that makes no tensor-core call has none, and with a small buffer
(several passes over map groups and over m) or none at all (the CTAs build their
own operands) every bit of the result is the same.

The shapes and the buffer are set through SHTG_TUNE_FORCE and
SHTG_TC_RECORD_BYTES, the first of which is read once per process, so the
transforms run in child processes (this file run as a program).
"""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# (N_side, l_max, maps): map groups of 8 (spin 2, and spin 0 synthesis with fewer
# CTAs than SMs) and 16 (spin 0); the second grid's transpose records of one m are
# larger than its synthesis records of a quarter of the m, so a small buffer
# splits the map groups there
SIZES = [(32, 64, 40), (64, 16, 40), (24, 60, 5), (96, 160, 40)]


def transforms(path):
    import torch

    from paper_2306_15511_gb300 import Plan
    out = {}
    for nside, lmax, nb in SIZES:
        plan = Plan(nside=nside, lmax=lmax, max_batch=nb, spin2=True)
        gen = torch.Generator(device="cuda").manual_seed(nside)
        for spin in (0, 2):
            lead = (nb, 2) if spin else (nb,)
            m = torch.randn(*lead, plan.npix, device="cuda", generator=gen)
            a = plan.alm2map_adjoint(m, spin=spin, tensor_cores=True)
            key = f"{nside} {lmax} {nb} {spin}"
            out[key + " adjoint"] = a.cpu().numpy()
            out[key + " synthesis"] = plan.alm2map(a, spin=spin, tensor_cores=True).cpu().numpy()
        plan.close()
    np.savez(path, **out)


def child(tmp_path, shape, room=None):
    path = str(tmp_path / "out.npz")
    env = {k: v for k, v in os.environ.items() if k != "SHTG_TC_RECORD_BYTES"}
    env["SHTG_TUNE_FORCE"] = str(shape)
    if room is not None:
        env["SHTG_TC_RECORD_BYTES"] = str(room)
    subprocess.run([sys.executable, os.path.abspath(__file__), path], check=True, env=env, cwd=ROOT, timeout=300)
    with np.load(path) as z:
        return {k: z[k] for k in z.files}


@pytest.fixture(scope="module")
def whole(tmp_path_factory):
    """Records of every map in one pass."""
    return child(tmp_path_factory.mktemp("whole"), 0)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,room", [
    (0, 4000000), (0, 1000000), (0, 200000), (0, 80000),   # several passes over m, over map groups
    (1, 200000),                             # (two A buffers; synthesis without records)
    (0, 0), (1, 0),                          # no buffer
    (1, None), (2, None), (3, None),         # every shape that the tuner may choose
])
def test_every_buffer_and_shape_gives_the_same_bits(tmp_path, whole, shape, room):
    got = child(tmp_path, shape, room)
    assert got.keys() == whole.keys()
    for k in whole:
        assert np.array_equal(got[k], whole[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("nside,lmax", [(64, 128), (96, 160)])
def test_map_groups_give_the_same_bits(nside, lmax):
    """Spin 0 by groups of 8 or 16 maps (as the grid is small or large, or the
    call has more than 8 maps) against 8 maps per call."""
    torch = pytest.importorskip("torch")
    from paper_2306_15511_gb300 import Plan
    nb = 21
    many = Plan(nside=nside, lmax=lmax, max_batch=nb)
    few = Plan(nside=nside, lmax=lmax, max_batch=8)
    m = torch.randn(nb, many.npix, device="cuda", generator=torch.Generator(device="cuda").manual_seed(lmax))
    a = many.alm2map_adjoint(m, tensor_cores=True)
    s = many.alm2map(a, tensor_cores=True)
    for k in range(0, nb, 8):
        ak = few.alm2map_adjoint(m[k:k + 8].contiguous(), tensor_cores=True)
        assert torch.equal(ak, a[k:k + 8])
        assert torch.equal(few.alm2map(ak, tensor_cores=True), s[k:k + 8])
    many.close()
    few.close()


def device_bytes(plan):
    from paper_2306_15511_gb300 import _native as N
    info = N.PlanInfo()
    N.check(plan._lib.shtg_plan_get_info(plan._h, C.byref(info)))
    return int(info.device_bytes)


@pytest.mark.gpu
def test_buffer_belongs_to_the_tensor_core_calls():
    torch = pytest.importorskip("torch")
    from paper_2306_15511_gb300 import Plan
    plan = Plan(nside=32, lmax=64, max_batch=2, spin2=True)
    start = device_bytes(plan)
    for dtype, kw in ((torch.float64, {}), (torch.float64, {"double_float": True}), (torch.float32, {})):
        for spin in (0, 2):
            m = torch.ones((2, 2, plan.npix) if spin else (2, plan.npix), dtype=dtype, device="cuda")
            plan.alm2map(plan.alm2map_adjoint(m, spin=spin, **kw), spin=spin, **kw)
    assert device_bytes(plan) == start
    m = torch.ones(2, plan.npix, device="cuda")
    plan.alm2map_adjoint(m, tensor_cores=True)
    spin0 = device_bytes(plan)
    assert spin0 > start
    plan.alm2map_adjoint(torch.ones(2, 2, plan.npix, device="cuda"), spin=2, tensor_cores=True)
    assert device_bytes(plan) > spin0
    both = device_bytes(plan)
    plan.alm2map(plan.alm2map_adjoint(m, tensor_cores=True), tensor_cores=True)
    assert device_bytes(plan) == both
    plan.close()


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    transforms(sys.argv[1])
