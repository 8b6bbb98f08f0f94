"""Tensor-core block products on the transform path (sse_sigma_fwd, mode F16X3_FFT) against the FP64 oracle.

FP32 transforms with the per-frequency block products as FP16 hi/lo split GEMMs on tcgen05 (three products,
FP32 accumulation, power-of-two scales). Stated bound: 2e-6 normwise per output tensor (max|gpu - oracle| /
max|oracle|), the FP32_FFT bound: the split keeps ~22 significant bits per operand, so the products add ~2^-22
relative per term to the FP32 transforms' few 1e-7.

The mode runs the tensor-core kernel for Norb >= 9 with NB >= 3 and the FP32 products otherwise. Every device call here
checks from its profile which of the two ran, and every behaviour is tested on both sides: both block sizes of the kernel
(27 of 32 rows per group and element copies at Norb = 9, 30 rows and bulk copies at Norb = 10), three and four bonds,
ragged last tiles, several frequency-tile groups, Nqz < Nkz, both flags, atom ranges, scales over the whole tensor, per
atom and per bond, neighbours out of range, host buffers, autograd and the FinFET workload on sampled blocks.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from conftest import normwise
from oracle.subproblem import oracle_blocks
from paper_1912_10024_gb300 import binding as B
from paper_1912_10024_gb300.inputs import FINFET, TINY, Dims, make_inputs, ring_neighbours

pytestmark = pytest.mark.gpu
SCALE = 1.0 / (2.0 * math.pi)
BOUND = 2e-6


TC10 = Dims(NA=6, NB=4, Norb=10, NE=37, Nkz=3, Nqz=2, Nw=7)  # bulk copies, a ragged last tile, Nqz < Nkz
TC9 = Dims(NA=5, NB=3, Norb=9, NE=26, Nkz=3, Nqz=3, Nw=6)    # 27 of 32 rows per group, element copies


def on_tensor_cores(d):
    return d.Norb >= 9 and d.NB >= 3


def gpu_sigma(inp, **kw):
    """The device call; its profile has to name the tensor-core kernel exactly where the rule says so."""
    g = inp.to("cuda")
    B.sse_profile_read()
    try:
        return B.sigma(g.G_less, g.G_greater, g.dH, g.D_less, g.D_greater, g.nbr, mode="f16x3_fft", profile=True, **kw)
    finally:
        torch.cuda.synchronize()
        names = [name for name, _, _ in B.sse_profile_read()]
        assert ("spec_prod_tc_kernel" in names) == on_tensor_cores(inp.dims), names


def inputs(d, seed, **kw):
    return make_inputs(d, seed=seed, nbr=None if d is TINY else ring_neighbours(d.NA, d.NB), **kw)


def oracle_sigma(inp, **kw):
    return oracle.sigma(inp.nbr, inp.dH, inp.D_less, inp.D_greater, inp.G_less, inp.G_greater, SCALE, **kw)


SHAPES = [
    TINY,  # the FP32 products up to Norb = 8 and for fewer than three bonds
    Dims(NA=5, NB=2, Norb=10, NE=40, Nkz=3, Nqz=2, Nw=11),
    Dims(NA=6, NB=3, Norb=1, NE=300, Nkz=2, Nqz=2, Nw=9),
    Dims(NA=7, NB=1, Norb=3, NE=61, Nkz=4, Nqz=3, Nw=5),
    Dims(NA=4, NB=4, Norb=5, NE=33, Nkz=3, Nqz=3, Nw=6),
    Dims(NA=3, NB=2, Norb=7, NE=50, Nkz=2, Nqz=1, Nw=13),
    Dims(NA=4, NB=3, Norb=8, NE=29, Nkz=5, Nqz=5, Nw=4),
    Dims(NA=3, NB=4, Norb=9, NE=26, Nkz=3, Nqz=3, Nw=8),    # the tensor cores
    TC9,
    TC10,
    Dims(NA=5, NB=3, Norb=10, NE=4, Nkz=1, Nqz=1, Nw=2),    # six frequencies: half a tile
    Dims(NA=5, NB=3, Norb=10, NE=59, Nkz=3, Nqz=3, Nw=5),   # 192: sixteen full tiles, two whole groups
    Dims(NA=5, NB=4, Norb=9, NE=103, Nkz=4, Nqz=3, Nw=5),   # 432: 36 tiles, the last group half full
]


@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: f"Norb{d.Norb}_NB{d.NB}_NE{d.NE}_Nkz{d.Nkz}")
def test_shapes(dims):
    inp = inputs(dims, seed=dims.Norb + 2000)
    Sl, Sg = gpu_sigma(inp, check=True)
    Ol, Og = oracle_sigma(inp)
    errs = [normwise(Sl.cpu().numpy(), Ol), normwise(Sg.cpu().numpy(), Og)]
    print("f16x3_fft", dims, errs)
    assert max(errs) <= BOUND


@pytest.mark.parametrize("dims", [TINY, Dims(NA=5, NB=2, Norb=10, NE=40, Nkz=3, Nqz=2, Nw=11), TC9, TC10],
                         ids=["tiny", "norb10", "tc9", "tc10"])
def test_antihermitian_half_spectrum(dims):
    inp = inputs(dims, seed=2100)
    Sl, Sg = gpu_sigma(inp, check=True, antihermitian=True)
    Ol, Og = oracle_sigma(inp)
    assert max(normwise(Sl.cpu().numpy(), Ol), normwise(Sg.cpu().numpy(), Og)) <= BOUND


@pytest.mark.parametrize("dims,atoms", [(TINY, (5, 12)), (TC9, (1, 3)), (TC10, (2, 5))], ids=["tiny", "tc9", "tc10"])
def test_symmetrize_and_atom_range(dims, atoms):
    inp = inputs(dims, seed=2200)
    Sl, Sg = gpu_sigma(inp, symmetrize=True)
    Ol, Og = oracle_sigma(inp)
    for S, O in ((Sl, Ol), (Sg, Og)):
        assert normwise(S.cpu().numpy(), 0.5 * (O - O.conj().swapaxes(-1, -2))) <= BOUND
    out = tuple(torch.full(dims.g_shape(), 3 + 3j, dtype=torch.complex128, device="cuda") for _ in range(2))
    a0, a1 = atoms
    gpu_sigma(inp, atoms=atoms, out=out)
    Ol, Og = oracle_sigma(inp, a_range=atoms)
    for S, O in zip(out, (Ol, Og)):
        S = S.cpu().numpy()
        assert normwise(S[:, :, a0:a1], O[:, :, a0:a1]) <= BOUND
        assert np.all(S[:, :, :a0] == 3 + 3j) and np.all(S[:, :, a1:] == 3 + 3j)


@pytest.mark.parametrize("d", [Dims(NA=5, NB=2, Norb=10, NE=40, Nkz=3, Nqz=2, Nw=11), TC9, TC10],
                         ids=["norb10", "tc9", "tc10"])
def test_scaled_inputs_keep_the_error(d):
    """Power-of-two normalisation: inputs scaled by 2^40 and 2^-40 give the same relative error (FP16 alone would
    overflow or flush)."""
    inp = inputs(d, seed=2300)
    for f in (2.0 ** 40, 2.0 ** -40):
        big = inputs(d, seed=2300)
        big.G_less, big.G_greater, big.D_less = inp.G_less * f, inp.G_greater * f, inp.D_less / f
        Sl, Sg = gpu_sigma(big)
        Ol, Og = oracle_sigma(big)
        assert max(normwise(Sl.cpu().numpy(), Ol), normwise(Sg.cpu().numpy(), Og)) <= BOUND, f


@pytest.mark.parametrize("d", [TC9, TC10], ids=["tc9", "tc10"])
def test_scales_per_atom_and_per_bond(d):
    """G of atom b scaled by 2^(-24 .. 24), or the couplings of slot s by 2^(-20 .. 20): the scales are per block and per
    bond, so every atom's Sigma keeps the error relative to its own largest element."""
    for what in ("atom", "bond"):
        inp = inputs(d, seed=2310, general=True)
        if what == "atom":
            f = 2.0 ** torch.linspace(-24, 24, d.NA).round().reshape(-1, 1, 1)
            inp.G_less, inp.G_greater = inp.G_less * f, inp.G_greater * f
        else:
            f = 2.0 ** torch.linspace(-20, 20, d.NB).round().reshape(1, -1, 1, 1, 1)
            inp.dH = inp.dH * f
        for S, O in zip(gpu_sigma(inp), oracle_sigma(inp)):
            S = S.cpu().numpy()
            for a in range(d.NA):
                assert normwise(S[:, :, a], O[:, :, a]) <= BOUND, (what, a)


@pytest.mark.parametrize("d,atom,slot", [(TINY, 2, 3), (TC9, 2, 1), (TC10, 0, 0), (TC10, 5, 3)],
                         ids=["tiny", "tc9", "tc10_first", "tc10_last"])
def test_bad_neighbour_reported_and_contributes_zero(d, atom, slot):
    inp = inputs(d, seed=2400)
    inp.nbr[atom, slot] = -7
    with pytest.raises(B.SseError) as e:
        gpu_sigma(inp, check=True)
    assert e.value.status == 5
    torch.cuda.synchronize()
    S = gpu_sigma(inp)
    ref = inp.dH.clone()
    ref[atom, slot] = 0
    inp.dH = ref
    inp.nbr[atom, slot] = 0
    for s, o in zip(S, oracle_sigma(inp)):
        assert normwise(s.cpu().numpy(), o) <= BOUND


def test_matches_fp32_fft_at_the_adjoint_workload():
    """NA=256, Norb=10, NE=256, Nkz=Nqz=5, Nw=16 (diamond list): the same transforms, products on the tensor
    cores; the two differ by the products' rounding only."""
    from paper_1912_10024_gb300.inputs import ADJOINT
    inp = make_inputs(ADJOINT, seed=7, device="cuda")
    args = (inp.G_less, inp.G_greater, inp.dH, inp.D_less, inp.D_greater, inp.nbr)
    tc = B.sigma(*args, mode="f16x3_fft", check=True)
    f32 = B.sigma(*args, mode="fp32_fft")
    f64 = B.sigma(*args, mode="fp64_fft")
    e_tc = max(float((x - y).abs().max() / y.abs().max()) for x, y in zip(tc, f64))
    e_32 = max(float((x - y).abs().max() / y.abs().max()) for x, y in zip(f32, f64))
    print("adjoint workload: f16x3_fft", e_tc, "fp32_fft", e_32)
    assert e_tc <= BOUND


def test_finfet_sampled():
    inp = make_inputs(FINFET, seed=0, device="cuda")
    Sl, Sg = B.sigma(inp.G_less, inp.G_greater, inp.dH, inp.D_less, inp.D_greater, inp.nbr, mode="f16x3_fft",
                     check=True)
    torch.cuda.synchronize()
    worst = 0.0
    for (a, E0, E1) in [(0, 0, 2), (511, 255, 257), (1023, 510, 512), (77, 100, 101)]:
        Ol, Og = oracle_blocks(inp.nbr, inp.dH, inp.D_less, inp.D_greater, inp.G_less, inp.G_greater, SCALE,
                               a, E0, E1)
        for S, O in ((Sl, Ol), (Sg, Og)):
            worst = max(worst, normwise(S[:, E0:E1, a].cpu().numpy(), O))
    print("f16x3_fft finfet sampled", worst)
    assert worst <= BOUND


@pytest.mark.parametrize("d", [Dims(NA=5, NB=2, Norb=10, NE=40, Nkz=3, Nqz=2, Nw=11), TC9, TC10],
                         ids=["norb10", "tc9", "tc10"])
def test_host_buffer_entry(d):
    inp = inputs(d, seed=2500)
    pin = [t.pin_memory() for t in (inp.G_less, inp.G_greater, inp.dH, inp.D_less, inp.D_greater, inp.nbr)]
    S = B.sigma_host(*pin, mode="f16x3_fft", check=True)
    for s, o, t in zip(S, oracle_sigma(inp), gpu_sigma(inp)):
        assert normwise(s.numpy(), o) <= BOUND
        assert torch.equal(s, t.cpu())


@pytest.mark.parametrize("d", [Dims(NA=6, NB=2, Norb=3, NE=20, Nkz=3, Nqz=2, Nw=4), TC9, TC10],
                         ids=["norb3", "tc9", "tc10"])
def test_autograd_after_tensor_core_forward(d):
    """sigma_autograd in mode f16x3_fft: the forward on the tensor cores (the same bytes as the plain call), the adjoint in
    FP32_FFT."""
    inp = inputs(d, seed=2600)
    g = inp.to("cuda")
    W = torch.randn(d.g_shape(), dtype=torch.complex128, generator=torch.Generator().manual_seed(1))
    V = torch.randn(d.g_shape(), dtype=torch.complex128, generator=torch.Generator().manual_seed(2))
    leaves = [t.clone().requires_grad_(True) for t in (g.dH, g.D_less, g.D_greater)]
    Sl, Sg = B.sigma_autograd(*leaves, g.G_less, g.G_greater, g.nbr, SCALE, "f16x3_fft")
    assert all(torch.equal(s.detach(), t) for s, t in zip((Sl, Sg), gpu_sigma(inp)))
    loss = (W.cuda().conj() * Sl).real.sum() + (V.cuda().conj() * Sg).real.sum()
    loss.backward()
    ref = oracle.sigma_grad(inp.nbr, inp.dH, inp.D_less, inp.D_greater, inp.G_less, inp.G_greater, SCALE, W, V)
    for leaf, r in zip(leaves, ref):
        assert normwise(leaf.grad.cpu().numpy(), r) <= 1e-5
