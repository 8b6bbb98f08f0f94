"""FP32 E-transforms at every transform length L = 2^a 3^b up to 1296: the codelet kernels (every pair of factors, both
column widths, partial column tiles, with and without the prefetched FP64 tile) and the Stockham kernel for the lengths
without two balanced factors. Sigma and Pi in FP32_FFT against FP64_FFT on the same inputs; bound 2e-6 normwise, the
mode's."""
import pytest

from conftest import normwise
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, ring_neighbours

pytestmark = pytest.mark.gpu

LENGTHS = sorted(2 ** a * 3 ** b for a in range(11) for b in range(7) if 6 <= 2 ** a * 3 ** b <= 1296)


@pytest.mark.parametrize("L", LENGTHS)
def test_every_length(L):
    Nw = 2 if L < 40 else 5
    d = Dims(NA=5, NB=1, Norb=3, NE=L - Nw, Nkz=2, Nqz=1, Nw=Nw)
    g = make_inputs(d, seed=L, nbr=ring_neighbours(d.NA, d.NB), general=True).to("cuda")
    S, R = [B.sigma(g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr, mode=m) for m in ("fp32_fft", "fp64_fft")]
    P, Q = [B.pi(g.G_less, g.G_greater, g.dH, g.nbr, d.Nqz, d.Nw, mode=m) for m in ("fp32_fft", "fp64_fft")]
    for x, y in zip(tuple(S) + tuple(P), tuple(R) + tuple(Q)):
        assert normwise(x.cpu().numpy(), y.cpu().numpy()) <= 2e-6
