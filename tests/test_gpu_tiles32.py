"""FP32 register-tile kernels of the adjoint (spec_adj32_kernel) and of Pi (spec_pi32_kernel), mode FP32_FFT, against the
FP64 oracle at the edges of their tiles.

Every block size Norb = 1 .. 16 (odd sizes are padded to even tiles, the groups of threads change with the size),
frequency counts below, at and just above a CTA's tile, several tiles and several chunks per bond, and a bond count whose
coupling blocks do not stay resident in shared memory. Bound: 2e-6 normwise per output tensor, as for the mode (FP32
rounding 6e-8 times the transform stages, the Norb-term products and sums of at most 192 FP32 terms, a
few 1e-7)."""
import math

import pytest

import oracle
from conftest import normwise
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, make_upstream, ring_neighbours

pytestmark = pytest.mark.gpu
SCALE = 1.0 / (2.0 * math.pi)
BOUND = 2e-6

SHAPES = [Dims(NA=3, NB=1 + n % 3, Norb=n, NE=9 + n, Nkz=1 + n % 3, Nqz=1, Nw=3) for n in range(1, 17)] + [
    Dims(NA=4, NB=2, Norb=10, NE=6, Nkz=1, Nqz=1, Nw=2),      # 8 frequencies: less than a tile
    Dims(NA=4, NB=2, Norb=10, NE=10, Nkz=5, Nqz=2, Nw=2),     # 60: whole tiles of 10
    Dims(NA=4, NB=2, Norb=10, NE=25, Nkz=1, Nqz=1, Nw=2),     # 27: a partial last tile
    Dims(NA=17, NB=16, Norb=10, NE=13, Nkz=2, Nqz=2, Nw=3),   # coupling blocks of Pi restaged per bond
    Dims(NA=11, NB=5, Norb=16, NE=11, Nkz=1, Nqz=1, Nw=3),
    Dims(NA=70, NB=4, Norb=9, NE=60, Nkz=3, Nqz=2, Nw=4),     # several tiles per CTA
]


@pytest.mark.parametrize("d", SHAPES, ids=lambda d: f"Norb{d.Norb}_NB{d.NB}_NE{d.NE}_Nkz{d.Nkz}_NA{d.NA}")
def test_adjoint_and_pi(d):
    nbr = ring_neighbours(d.NA, d.NB)
    x = make_inputs(d, seed=41 + d.Norb, nbr=nbr, general=True)
    g = x.to("cuda")
    W = make_upstream(d, seed=42)
    R = B.sigma_grad(g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr, W[0].cuda(), W[1].cuda(),
                     mode="fp32_fft", check=True)
    O = oracle.sigma_grad(x.nbr, x.dH, x.D_less, x.D_greater, x.G_less, x.G_greater, SCALE, W[0], W[1])
    for s, o in zip(R, O):
        assert normwise(s.cpu().numpy(), o) <= BOUND
    P = B.pi(g.G_less, g.G_greater, g.dH, g.nbr, d.Nqz, d.Nw, mode="fp32_fft", check=True)
    O = oracle.pi(x.nbr, x.dH, x.G_less, x.G_greater, SCALE, d.Nqz, d.Nw)
    for s, o in zip(P, O):
        assert normwise(s.cpu().numpy(), o) <= BOUND
