"""The FP32 adjoint's coupling gradient is summed over the groups of threads in FP64 (spec_adj32_kernel).

Small whole numbers on a 4 x 4 frequency grid (L = 4, Nkz = 4: every twiddle is 1, -1, i or -i): the transforms, the
block products and each group's sum are whole numbers below 2^24, exact in FP32, while the sum over the 16 frequencies
needs more than 24 bits. Added in FP64 the gradient equals the oracle's to the bit; one FP32 addition of two groups'
sums would round it. The magnitudes are asserted from a numpy model of the terms (one (frequency, l) per group at
Norb = 1 and 2)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import Dims, make_inputs, ring_neighbours

pytestmark = pytest.mark.gpu


def whole(shape, most, rng):
    return torch.from_numpy(rng.integers(-most, most + 1, shape) + 1j * rng.integers(-most, most + 1, shape))


def terms_of_type(x, t, W):
    """The terms X_mu[:, l] conj(G[:, l]) and conj(W[l, :]) U_mu[l, :] of one type, per bond [f][l][mu][m][n], each with a
    bound of every partial product of its complex multiplication."""
    d = x.dims
    Gl, Ds = (x.G_less, x.G_greater)[t].numpy(), (x.D_less.numpy(), x.D_greater.numpy())

    def spectrum(v):
        p = np.zeros((4, 4) + v.shape[2:], complex)
        p[:v.shape[0], :v.shape[1]] = v
        return np.round(np.fft.fft2(p, axes=(0, 1))).reshape((16,) + v.shape[2:])

    k = np.zeros((d.Nqz, 4) + Ds[0].shape[2:], complex)
    k[:, 1], k[:, 3] = Ds[t][:, 0], Ds[1 - t][:, 0]
    Gh, Wh, Kh = spectrum(Gl), spectrum(W), spectrum(k)
    for a in range(d.NA):
        for s in range(d.NB):
            A, w, g, kk = x.dH[a, s].numpy(), Wh[:, a], Gh[:, x.nbr[a, s]], Kh[:, a, s]
            X = np.einsum("fmj,fjab->fmab", -1j * np.conj(kk), np.stack([w @ A[j] for j in range(3)], 1))
            U = np.einsum("fim,fiab->fmab", 1j * kk, np.stack([A[i] @ g for i in range(3)], 1))
            for spec, p, q in (("fmxl,fyl->flmxy", X, np.conj(g)), ("flx,fmly->flmxy", np.conj(w), U)):
                yield np.einsum(spec, p, q), np.einsum(spec, abs(p.real) + abs(p.imag), abs(q.real) + abs(q.imag))


@pytest.mark.parametrize("Norb,most", [(1, 80), (2, 55)])
def test_whole_numbers_survive(Norb, most):
    d = Dims(NA=3, NB=1, Norb=Norb, NE=3, Nkz=4, Nqz=4, Nw=1)
    x = make_inputs(d, seed=3, nbr=ring_neighbours(d.NA, d.NB), general=True)
    rng = np.random.default_rng(Norb)
    for name in ("G_less", "G_greater", "dH", "D_less", "D_greater"):
        setattr(x, name, whole(getattr(x, name).shape, 3, rng))
    W = [whole(d.g_shape(), 3, rng) for _ in range(2)]
    for t in range(2):  # one large entry a lag of one apart: the terms of all frequencies have a common part
        (x.G_less, x.G_greater)[t][0, 0] += most
        (x.D_less, x.D_greater)[t][0, 0] += most
        W[t][0, 1] += most * 1j
    lossy = 0
    for t in range(2):
        v, bound = (np.array(p) for p in zip(*terms_of_type(x, t, W[t].numpy())))
        assert bound.max() < 2 ** 24
        total = v[0::2].sum((1, 2)) + v[1::2].sum((1, 2))
        seq = np.stack([v[0::2], v[1::2]], 1).reshape((d.NA * d.NB, -1) + v.shape[3:]).astype(np.complex64)
        f32 = np.zeros_like(seq[:, 0])
        for i in range(seq.shape[1]):
            f32 = f32 + seq[:, i]
        lossy += int((f32 != total).sum())
    assert lossy > 0, "the FP32 sum is exact too: the inputs show nothing"
    g = x.to("cuda")
    got = B.sigma_grad(g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr, W[0].cuda(), W[1].cuda(), scale=1.0,
                       mode="fp32_fft", check=True)[0].cpu().numpy()
    ref = oracle.sigma_grad(x.nbr, x.dH, x.D_less, x.D_greater, x.G_less, x.G_greater, 1.0, W[0], W[1])[0]
    assert np.array_equal(got, np.asarray(ref))
