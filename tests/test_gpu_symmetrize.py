"""SSE_FLAG_SYMMETRIZE is FP64 arithmetic on the stored Sigma in the FP32 transform modes too: on general inputs the
result is (S - S^H) / 2 of the unflagged result to the bit, and with anti-Hermitian inputs each pair of independently
rounded elements is averaged, which leaves values that FP32 cannot hold. Norb = 9 with NB = 3 runs the tensor-core
products in F16X3_FFT, the other shapes the FP32 ones; the transform lengths 32, 36 and 72 take the codelet E-transforms,
243 the Stockham kernel."""
import pytest
import torch

from conftest import normwise
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, ring_neighbours

pytestmark = pytest.mark.gpu

SHAPES = [Dims(NA=6, NB=2, Norb=4, NE=33, Nkz=3, Nqz=2, Nw=3), Dims(NA=5, NB=3, Norb=9, NE=68, Nkz=4, Nqz=4, Nw=4),
          Dims(NA=5, NB=1, Norb=1, NE=28, Nkz=1, Nqz=1, Nw=4), Dims(NA=7, NB=2, Norb=7, NE=238, Nkz=8, Nqz=5, Nw=5)]


def ident(d):
    return f"Norb{d.Norb}_NE{d.NE}_Nkz{d.Nkz}"


@pytest.mark.parametrize("mode", ["fp32_fft", "f16x3_fft"])
@pytest.mark.parametrize("d", SHAPES, ids=ident)
def test_general_inputs_to_the_bit(d, mode):
    g = make_inputs(d, seed=8, nbr=ring_neighbours(d.NA, d.NB), general=True).to("cuda")
    args = (g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr)
    for atoms in ((0, d.NA), (2, 3)):
        S = B.sigma(*args, mode=mode, symmetrize=True, atoms=atoms)
        R = B.sigma(*args, mode=mode, atoms=atoms)
        for s, r in zip(S, R):
            s, r = s[:, :, atoms[0]:atoms[1]], r[:, :, atoms[0]:atoms[1]]
            assert torch.equal(s, 0.5 * (r - r.conj().transpose(-1, -2)))


@pytest.mark.parametrize("mode", ["fp32_fft", "f16x3_fft"])
@pytest.mark.parametrize("d", [s for s in SHAPES if s.Norb > 1], ids=ident)
def test_antihermitian_inputs_are_averaged(d, mode):
    g = make_inputs(d, seed=9, nbr=ring_neighbours(d.NA, d.NB)).to("cuda")
    args = (g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr)
    S = B.sigma(*args, mode=mode, antihermitian=True, symmetrize=True, check=True)
    R = B.sigma(*args, mode="fp64_fft", antihermitian=True, symmetrize=True)
    for s, r in zip(S, R):
        assert torch.equal(s, -s.conj().transpose(-1, -2))
        assert normwise(s.cpu().numpy(), r.cpu().numpy()) <= 2e-6
        assert not torch.equal(s, s.to(torch.complex64).to(torch.complex128))
