"""Tensor-core transpose whose operand records do not fit the plan's record
buffer at once (48 maps at N_side 512, l_max 1536: 4.8 GB in two passes over m),
and the synthesis that uses the same buffer, against a plan that takes 8 maps at a time in one pass: every map group
is worked by the same kernels, so every bit is the same.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_several_passes_give_the_same_bits():
    from paper_2306_15511_gb300 import Plan
    nside, lmax, nb = 512, 1536, 48
    big = Plan(nside=nside, lmax=lmax, max_batch=nb, spin2=True)
    gen = torch.Generator(device="cuda").manual_seed(5)
    m = torch.randn(nb, 2, big.npix, device="cuda", generator=gen)
    a = big.alm2map_adjoint(m, spin=2, tensor_cores=True)
    s = big.alm2map(a, spin=2, tensor_cores=True)
    big.close()
    small = Plan(nside=nside, lmax=lmax, max_batch=8, spin2=True)
    for k in range(0, nb, 8):
        ak = small.alm2map_adjoint(m[k:k + 8].contiguous(), spin=2, tensor_cores=True)
        assert torch.equal(ak, a[k:k + 8])
        assert torch.equal(small.alm2map(ak, spin=2, tensor_cores=True), s[k:k + 8])
    small.close()
