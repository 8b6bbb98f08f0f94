"""FP32 register-tile products (spec_prod32_kernel: Sigma forward and the gradient in G, mode FP32_FFT) against the
FP64 oracle at the edges of the kernel's tiles.

Every block size Norb = 1 .. 16 (odd sizes are padded to even tiles; one or two frequencies per thread), frequency
counts below, at and just above a CTA's tile, a bond count whose coupling blocks do not stay resident in shared
memory, and target atoms without an incoming bond. Bound: 2e-6 normwise per output tensor, as for the mode (FP32
rounding 6e-8 times the transform stages and the Norb-term products, a few 1e-7)."""
import math

import pytest
import torch

import oracle
from conftest import normwise
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, make_upstream, ring_neighbours

pytestmark = pytest.mark.gpu
SCALE = 1.0 / (2.0 * math.pi)
BOUND = 2e-6

SHAPES = [Dims(NA=3, NB=1 + n % 3, Norb=n, NE=9 + n, Nkz=1 + n % 3, Nqz=1, Nw=3) for n in range(1, 17)] + [
    Dims(NA=4, NB=2, Norb=10, NE=22, Nkz=1, Nqz=1, Nw=2),     # 24 frequencies: one full tile
    Dims(NA=4, NB=2, Norb=10, NE=25, Nkz=1, Nqz=1, Nw=2),     # 27: one full tile and three more
    Dims(NA=17, NB=16, Norb=10, NE=13, Nkz=2, Nqz=2, Nw=3),   # coupling blocks restaged per bond
    Dims(NA=11, NB=10, Norb=16, NE=11, Nkz=1, Nqz=1, Nw=3),
    Dims(NA=70, NB=4, Norb=9, NE=60, Nkz=3, Nqz=2, Nw=4),     # several tiles per CTA
]


@pytest.mark.parametrize("d", SHAPES, ids=lambda d: f"Norb{d.Norb}_NB{d.NB}_NE{d.NE}_NA{d.NA}")
def test_forward_and_gradient_in_g(d):
    nbr = ring_neighbours(d.NA, d.NB)
    nbr[:, 0] = nbr[0, 0]  # some atoms with many incoming bonds, some with none
    x = make_inputs(d, seed=31 + d.Norb, nbr=nbr, general=True)
    g = x.to("cuda")
    S = B.sigma(g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr, mode="fp32_fft", check=True)
    O = oracle.sigma(x.nbr, x.dH, x.D_less, x.D_greater, x.G_less, x.G_greater, SCALE)
    for s, o in zip(S, O):
        assert normwise(s.cpu().numpy(), o) <= BOUND
    W = make_upstream(d, seed=32)
    R = B.sigma_grad_G(g.dH, g.D_less, g.D_greater, g.nbr, W[0].cuda(), W[1].cuda(), mode="fp32_fft", check=True)
    O = oracle.sigma_grad_G(x.nbr, x.dH, x.D_less, x.D_greater, SCALE, W[0], W[1])
    for s, o in zip(R, O):
        assert normwise(s.cpu().numpy(), o) <= BOUND
