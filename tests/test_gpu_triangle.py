"""Transforms of the upper triangle's columns (sse_tri.cuh), with SSE_FLAG_ANTIHERMITIAN against the general path of the
same mode on the same anti-Hermitian inputs.

kz grids with and without an instantiation (Nkz = 9 takes the full columns), odd and even transform lengths (self-paired
rows eps = 0 and L / 2), block sizes down to 1, atom ranges for which the scratch holds the triangle or not, with and
without symmetrisation. Bounds: the tolerances of the modes against the oracle (FP64 1e-12, FP32 transforms 2e-6)."""
import pytest
import torch

from conftest import normwise
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, ring_neighbours

pytestmark = pytest.mark.gpu

SHAPES = [Dims(NA=6, NB=2, Norb=1 + 2 * k % 11, NE=20 + 5 * k, Nkz=k, Nqz=(k + 1) // 2, Nw=3) for k in range(1, 10)] + [
    Dims(NA=5, NB=3, Norb=10, NE=24, Nkz=3, Nqz=2, Nw=3),     # L = 27
    Dims(NA=5, NB=1, Norb=16, NE=76, Nkz=2, Nqz=2, Nw=5),     # L = 81
    Dims(NA=40, NB=4, Norb=10, NE=61, Nkz=7, Nqz=7, Nw=9),    # L = 72
]


@pytest.mark.parametrize("mode,bound", [("fp64_fft", 1e-12), ("fp32_fft", 2e-6), ("f16x3_fft", 2e-6)])
@pytest.mark.parametrize("d", SHAPES, ids=lambda d: f"Norb{d.Norb}_NE{d.NE}_Nkz{d.Nkz}_NA{d.NA}")
def test_sigma_equals_general_path(d, mode, bound):
    if mode == "f16x3_fft" and d.Norb > 10:
        pytest.skip("the tensor-core products take Norb <= 10")
    g = make_inputs(d, seed=5, nbr=ring_neighbours(d.NA, d.NB)).to("cuda")
    args = (g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr)
    for atoms in ((0, d.NA), (1, d.NA), (2, 3)):
        for sym in (False, True):
            S = B.sigma(*args, mode=mode, antihermitian=True, symmetrize=sym, check=True, atoms=atoms)
            R = B.sigma(*args, mode=mode, symmetrize=sym, atoms=atoms)
            for s, r in zip(S, R):
                s, r = s[:, :, atoms[0]:atoms[1]], r[:, :, atoms[0]:atoms[1]]
                assert normwise(s.cpu().numpy(), r.cpu().numpy()) <= bound
                if sym:
                    assert torch.equal(s, -s.conj().transpose(-1, -2))


@pytest.mark.parametrize("mode,bound", [("fp64_fft", 1e-12), ("fp32_fft", 2e-6)])
@pytest.mark.parametrize("d", SHAPES, ids=lambda d: f"Norb{d.Norb}_NE{d.NE}_Nkz{d.Nkz}_NA{d.NA}")
def test_pi_equals_general_path(d, mode, bound):
    g = make_inputs(d, seed=6, nbr=ring_neighbours(d.NA, d.NB)).to("cuda")
    for sym in (False, True):
        kw = dict(mode=mode, symmetrize=sym)
        P = B.pi(g.G_less, g.G_greater, g.dH, g.nbr, d.Nqz, d.Nw, antihermitian=True, check=True, **kw)
        R = B.pi(g.G_less, g.G_greater, g.dH, g.nbr, d.Nqz, d.Nw, **kw)
        for p, r in zip(P, R):
            assert normwise(p.cpu().numpy(), r.cpu().numpy()) <= bound


@pytest.mark.parametrize("mode,bound", [("fp64_fft", 1e-12), ("fp32_fft", 2e-6), ("f16x3_fft", 2e-6)])
@pytest.mark.parametrize("d", SHAPES, ids=lambda d: f"Norb{d.Norb}_NE{d.NE}_Nkz{d.Nkz}_NA{d.NA}")
def test_projection_of_general_inputs(d, mode, bound):
    """SSE_FLAG_SYMMETRIZE on inputs without symmetry: (S - S^H) / 2 of the unflagged result, exactly anti-Hermitian."""
    if mode == "f16x3_fft" and d.Norb > 10:
        pytest.skip("the tensor-core products take Norb <= 10")
    g = make_inputs(d, seed=7, nbr=ring_neighbours(d.NA, d.NB), general=True).to("cuda")
    args = (g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr)
    for atoms in ((0, d.NA), (2, 3)):
        S = B.sigma(*args, mode=mode, symmetrize=True, atoms=atoms)
        R = B.sigma(*args, mode=mode, atoms=atoms)
        for s, r in zip(S, R):
            s, r = s[:, :, atoms[0]:atoms[1]], r[:, :, atoms[0]:atoms[1]]
            want = 0.5 * (r - r.conj().transpose(-1, -2))
            assert normwise(s.cpu().numpy(), want.cpu().numpy()) <= bound
            assert torch.equal(s, -s.conj().transpose(-1, -2))
