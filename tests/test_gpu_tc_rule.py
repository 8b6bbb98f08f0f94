"""Mode F16X3_FFT on both sides of the rule that picks its block products: tensor cores for Norb >= 9 with at least three
bonds, the FP32 products otherwise. Every (Norb, NB) around the line against the FP64 oracle (2e-6 normwise, the mode's
bound), and the kernel that ran, from the profile."""
import math

import pytest
import torch

import oracle
from conftest import normwise
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, ring_neighbours

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("NB", [1, 2, 3, 4])
@pytest.mark.parametrize("Norb", [8, 9, 10])
def test_products_by_block_size_and_bonds(Norb, NB):
    d = Dims(NA=6, NB=NB, Norb=Norb, NE=27, Nkz=2, Nqz=2, Nw=4)
    x = make_inputs(d, seed=Norb + NB, nbr=ring_neighbours(d.NA, d.NB), general=True)
    g = x.to("cuda")
    B.sse_profile_read()
    S = B.sigma(g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr, mode="f16x3_fft", profile=True)
    torch.cuda.synchronize()
    names = [name for name, _, _ in B.sse_profile_read()]
    assert ("spec_prod_tc_kernel" in names) == (Norb >= 9 and NB >= 3)
    O = oracle.sigma(x.nbr, x.dH, x.D_less, x.D_greater, x.G_less, x.G_greater, 1.0 / (2.0 * math.pi))
    for s, o in zip(S, O):
        assert normwise(s.cpu().numpy(), o) <= 2e-6
