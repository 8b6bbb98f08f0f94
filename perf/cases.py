"""The calls of this library whose speed is measured: one pass per case, through the Python entry points of
``paper_1912_10024_gb300.binding``, on the seeded synthetic inputs of ``paper_1912_10024_gb300.inputs``.

A case names an operation (``op``), an arithmetic mode and the problem sizes:

* ``sigma``   Sigma^<, Sigma^> of Eq. (3) on device tensors, with the output and workspace tensors that a
              self-consistent loop keeps from one iteration to the next;
* ``step``    the autograd step: forward, then the gradients of dH, D^<, D^>, G^<, G^>;
* ``grad``    the adjoint alone (gradients of dH, D^<, D^>), with a kept workspace;
* ``grad_g``  the gradient with respect to G^<, G^> alone, with a kept workspace;
* ``pi``      Pi^<, Pi^> of Eq. (4), with kept output and workspace;
* ``dcomb``   the bond weights from the raw phonon functions, and their adjoint;
* ``host``    Sigma from page-locked host tensors to page-locked host tensors.

``exact`` evaluates the same sums with torch.fft and torch matrix products in complex128. The direct tensor-core modes
(bf16x3, tf32) are left out: they are kept as cross-checks of the transform modes, which replace them in use.
"""
import math

import torch

from paper_1912_10024_gb300 import binding as sse
from paper_1912_10024_gb300.inputs import ADJOINT, FINFET, TINY, Dims, default_neighbours, make_inputs, make_upstream

SCALE = 1.0 / (2.0 * math.pi)
SIZES = ("NA", "NB", "Norb", "NE", "Nkz", "Nqz", "Nw")


def _case(name, op, mode, dims, antihermitian=False, symmetrize=False):
    c = {"op": op, "mode": mode, "antihermitian": antihermitian, "symmetrize": symmetrize}
    c.update({n: getattr(dims, n) for n in SIZES})
    return dict(c, name=name) if name else c


def listed():
    return [
        # the first call of a new user: the tiny structure in the Python default mode (direct FP64 sums)
        _case("sigma_tiny_default", "sigma", "fp64", TINY),
        # the smallest differentiable step (gradient checks, fits of a few parameters): many launches, little work
        _case("step_tiny_fp64", "step", "fp64_fft", TINY),
        # an ordinary odd-sized run: odd blocks, three bonds, truncated qz grid, a transform length of no special form
        _case("sigma_ragged_f16x3", "sigma", "f16x3_fft", Dims(NA=90, NB=3, Norb=7, NE=301, Nkz=4, Nqz=3, Nw=21),
              symmetrize=True),
        # the FinFET structure in the two mixed precisions: one iteration of the self-consistent loop
        _case("sigma_finfet_f16x3", "sigma", "f16x3_fft", FINFET),
        _case("sigma_finfet_fp32", "sigma", "fp32_fft", FINFET),
        # the same iteration in FP64 with the symmetry that lesser and greater functions have
        _case("sigma_finfet_fp64", "sigma", "fp64_fft", FINFET, antihermitian=True),
        # inverse design on the adjoint structure: one training step, every gradient
        _case("step_adjoint_fp32", "step", "fp32_fft", ADJOINT),
        # the adjoint at the FinFET sizes (gradients of the couplings and the phonon weights)
        _case("grad_finfet_fp32", "grad", "fp32_fft", FINFET),
        # the phonon half of the iteration
        _case("pi_finfet_fp32", "pi", "fp32_fft", FINFET),
        # sensitivities with respect to G for twelve orbitals (the paper's "Small" block size) on ragged grids
        _case("grad_g_norb12_fp32", "grad_g", "fp32_fft", Dims(NA=200, NB=4, Norb=12, NE=350, Nkz=3, Nqz=3, Nw=45)),
        # a host program that owns the Green's functions: upload, compute, download
        _case("host_f16x3", "host", "f16x3_fft", Dims(NA=128, NB=4, Norb=10, NE=256, Nkz=5, Nqz=5, Nw=16)),
        # the phonon weights of the FinFET iteration and their adjoint: pure memory traffic
        _case("dcomb_finfet", "dcomb", "fp64", FINFET),
    ]


def draw(rng):
    op, mode = rng.choice([("sigma", "fp64"), ("sigma", "f16x3_fft"), ("sigma", "f16x3_fft"), ("sigma", "fp32_fft"),
                           ("sigma", "fp64_fft"), ("step", "fp32_fft"), ("grad", "fp32_fft"), ("pi", "fp32_fft"),
                           ("pi", "fp64_fft"), ("grad_g", "fp32_fft"), ("host", "f16x3_fft"), ("dcomb", "fp64")])

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    NA, NE, Nkz = spread(16, 1024), spread(32, 512), rng.randint(1, 7)
    Norb = rng.randint(4, 10 if mode == "f16x3_fft" else 12)
    NB = rng.choice([2, 4]) if op == "dcomb" else rng.randint(1, 4)
    Nw = min(rng.randint(4, 45), NE // 2)
    Nqz = rng.randint(max(1, Nkz - 2), Nkz)
    # multiply-adds of the block products; FP64 runs on a pipe about sixty times narrower, the direct sums cost
    # about Nqz * Nw times more, and host buffers are page-locked, which takes long
    cap = 3e9 if mode == "fp64" else 5e10 if mode == "fp64_fft" else 4e10 if op == "host" else 6e11
    while NA > 16 and _macs(Dims(NA, NB, Norb, NE, Nkz, Nqz, Nw)) > cap and op != "dcomb":
        NA = max(16, NA * 2 // 3)
    while op != "dcomb" and NE > 32 and _macs(Dims(NA, NB, Norb, NE, Nkz, Nqz, Nw)) > cap:
        NE = max(32, NE * 2 // 3)
        Nw = min(Nw, NE // 2)
    ah = op in ("sigma", "pi") and mode != "fp64" and rng.random() < 0.4
    sym = op != "dcomb" and rng.random() < 0.3
    return _case(None, op, mode, Dims(NA, NB, Norb, NE, Nkz, Nqz, Nw), ah, sym)


def _dims(c):
    return Dims(**{n: c[n] for n in SIZES})


def _symmetric_neighbours(d):
    """A list in which every bond has its reverse: the diamond slab where the sizes fit, a two-way ring otherwise."""
    if d.NB == 4 and d.NA in (256, 1024, 4096):
        return default_neighbours(d)
    steps = [s for k in range(1, d.NB // 2 + 1) for s in (k, -k)]
    a = torch.arange(d.NA).unsqueeze(1)
    return ((a + torch.tensor(steps)) % d.NA).to(torch.int32)


def _raw_phonon(d, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return [torch.complex(*(0.01 * torch.randn(d.Nqz, d.Nw, d.NA, n, 3, 3, dtype=torch.float64, device="cuda",
                                               generator=gen) for _ in range(2)))
            for n in (d.NB + 1, d.NB + 1, d.NB, d.NB)]


def prepare(case, seed):
    d, op = _dims(case), case["op"]
    st = {"case": case, "d": d}
    if op == "dcomb":
        st["raw"] = _raw_phonon(d, seed)
        st["nbr"] = _symmetric_neighbours(d).cuda()
        return st
    x = make_inputs(d, seed=seed, device="cuda")
    st["x"] = x
    m = sse.MODES[case["mode"]]
    flags = (sse.SSE_FLAG_SYMMETRIZE if case["symmetrize"] else 0)
    flags |= sse.SSE_FLAG_ANTIHERMITIAN if case["antihermitian"] else 0
    cd = sse.dims_of(x.G_less, x.D_less, x.dH)

    def buf(n):
        return torch.empty(n, dtype=torch.uint8, device="cuda")

    if op == "sigma":
        st["out"] = (torch.empty_like(x.G_less), torch.empty_like(x.G_greater))
        st["ws"] = buf(sse.sse_workspace_bytes(cd, m, flags))
    elif op == "pi":
        shape = (d.Nqz, d.Nw, d.NA, d.NB + 1, 3, 3)
        st["out"] = tuple(torch.empty(shape, dtype=torch.complex128, device="cuda") for _ in range(2))
        st["ws"] = buf(sse.sse_pi_workspace_bytes(cd, m, flags))
    elif op in ("grad", "grad_g", "step"):
        st["W"] = make_upstream(d, seed=seed + 1, device="cuda")
        if op == "grad":
            st["ws"] = buf(sse.sse_workspace_bytes(cd, m, flags))
        elif op == "grad_g":
            st["ws"] = buf(sse.sse_sigma_bwd_g_workspace_bytes(cd, m, flags))
        else:
            st["leaves"] = [t.requires_grad_() for t in (x.dH, x.D_less, x.D_greater, x.G_less, x.G_greater)]
    elif op == "host":
        st["host"] = [t.cpu().pin_memory() for t in (x.G_less, x.G_greater, x.dH, x.D_less, x.D_greater, x.nbr)]
        st["out"] = tuple(torch.zeros(d.g_shape(), dtype=torch.complex128).pin_memory() for _ in range(2))
        st["buf"] = buf(sse.sse_sigma_fwd_host_bytes(cd, m, flags))
        st["copy"] = torch.cuda.Stream()
        del st["x"]
    return st


def run(st):
    c, op = st["case"], st["case"]["op"]
    mode, sym, ah = c["mode"], c["symmetrize"], c["antihermitian"]
    if op == "dcomb":
        rl, rg, gl, gg = st["raw"]
        return sse.dcomb(rl, rg, st["nbr"]) + sse.dcomb_grad(gl, gg, st["nbr"])
    if op == "host":
        return sse.sigma_host(*st["host"], mode=mode, symmetrize=sym, out=st["out"], device_buf=st["buf"],
                              copy_stream=st["copy"], antihermitian=ah)
    x = st["x"]
    if op == "sigma":
        return sse.sigma(x.G_less, x.G_greater, x.dH, x.D_less, x.D_greater, x.nbr, mode=mode, symmetrize=sym,
                         antihermitian=ah, out=st["out"], ws=st["ws"])
    if op == "pi":
        return sse.pi(x.G_less, x.G_greater, x.dH, x.nbr, c["Nqz"], c["Nw"], mode=mode, symmetrize=sym,
                      antihermitian=ah, out=st["out"], ws=st["ws"])
    if op == "grad":
        return sse.sigma_grad(x.G_less, x.G_greater, x.dH, x.D_less, x.D_greater, x.nbr, *st["W"], mode=mode,
                              symmetrize=sym, ws=st["ws"])
    if op == "grad_g":
        return sse.sigma_grad_G(x.dH, x.D_less, x.D_greater, x.nbr, *st["W"], mode=mode, symmetrize=sym, ws=st["ws"])
    S = sse.sigma_autograd(*st["leaves"], x.nbr, mode=mode, symmetrize=sym)
    return tuple(S) + torch.autograd.grad(S, st["leaves"], st["W"])


# ---- the work of one pass --------------------------------------------------------------------------------------

def _macs(d, products=6):
    """Complex multiply-adds of the block products of both types: `products` Norb^3 and 9 Norb^2 per bond and
    frequency, on the shortest grid that holds the linear convolution."""
    return 2 * d.Nkz * (d.NE + d.Nw) * d.NA * d.NB * (products * d.Norb ** 3 + 9 * d.Norb ** 2)


def work(case):
    d, op = _dims(case), case["op"]
    G = 16 * d.Nkz * d.NE * d.NA * d.Norb ** 2
    D = 16 * d.Nqz * d.Nw * d.NA * d.NB * 9
    H = 16 * d.NA * d.NB * 3 * d.Norb ** 2
    nb = 4 * d.NA * d.NB
    if op == "dcomb":
        raw = 16 * d.Nqz * d.Nw * d.NA * (d.NB + 1) * 9
        return {"bytes": 4 * (raw + D) + 2 * nb, "flops": 2 * 2 * 3 * (D // 8) * 1.0}
    n = d.Nkz * (d.NE + d.Nw)
    fft = 5.0 * n * math.log2(n) * d.NA * d.Norb ** 2  # one block-valued transform
    half = 0.5 if case["antihermitian"] else 1.0
    fwd = 8.0 * _macs(d) * half + 4 * fft
    adj = 8.0 * _macs(d, 12) + 4 * fft
    if op in ("sigma", "host"):
        return {"bytes": 4 * G + 2 * D + H + nb, "flops": fwd}
    if op == "pi":
        return {"bytes": 2 * G + H + nb + 2 * 16 * d.Nqz * d.Nw * d.NA * (d.NB + 1) * 9,
                "flops": 8.0 * _macs(d) * half + 2 * fft}
    if op == "grad":
        return {"bytes": 4 * G + 4 * D + 2 * H + nb, "flops": adj}
    if op == "grad_g":
        return {"bytes": 4 * G + 2 * D + H + nb, "flops": fwd}
    return {"bytes": 8 * G + 4 * D + 2 * H + nb, "flops": 2 * fwd + adj}


def tolerance(case):
    """About four times the 2-norm error measured against `exact` over the listed and drawn sizes: 1.4e-15 in FP64,
    5.8e-7 in the mixed modes. The bond weights are sums of four terms, equal to the bit in the order of Eq. (3)."""
    if case["op"] == "dcomb":
        return {"rel": 1e-15}
    if case["mode"] in ("fp64", "fp64_fft"):
        return {"rel": 6e-15}
    return {"rel": 2.4e-6}


# ---- the same sums in 64 bits with torch alone -----------------------------------------------------------------

def _length(n):
    """The smallest 2^a 3^b 5^c >= n."""
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def _spectrum(X, L):
    """[Nkz, NE, NA, N, N] -> [NA, Nkz * L, N, N], zero-padded along E, transformed along E and kz."""
    Nkz, NE, NA, N, _ = X.shape
    Y = torch.fft.fft(torch.fft.fft(X, n=L, dim=1), dim=0)
    return Y.reshape(Nkz * L, NA, N, N).permute(1, 0, 2, 3).contiguous()


def _back(Y, Nkz, L, NE):
    """[c, Nkz * L, ...] -> [Nkz, NE, c, ...]."""
    Y = Y.reshape((Y.shape[0], Nkz, L) + Y.shape[2:])
    Y = torch.fft.ifft(torch.fft.ifft(Y, dim=1), dim=2)[:, :, :NE]
    return Y.movedim(0, 2)


def _lags(Dt, Do, Nkz, L):
    """Transformed lag kernel [c, NB, F, 3, 3] from the phonon weights [Nqz, Nw, c, NB, 3, 3] of the two types."""
    Nqz, Nw = Dt.shape[:2]
    K = torch.cat([torch.zeros_like(Dt[:, :1]), Dt,
                   torch.zeros((Nqz, L - 1 - 2 * Nw) + Dt.shape[2:], dtype=Dt.dtype, device=Dt.device), Do.flip(1)],
                  dim=1)
    K = torch.fft.fft(torch.fft.fft(K, n=Nkz, dim=0), dim=1)
    return K.reshape((Nkz * L,) + K.shape[2:]).permute(1, 2, 0, 3, 4)


def _forward(Gh, dH, Dt, Do, nb, Nkz, L, NE, sym):
    """Sigma [Nkz, NE, c, N, N] of a chunk of atoms: dH, Dt, Do are theirs, nb [c, NB] their neighbours."""
    c, NB, _, N, _ = dH.shape
    F = Nkz * L
    K = _lags(Dt, Do, Nkz, L)
    acc = None
    for s in range(NB):
        right = dH[:, s].conj().permute(0, 3, 1, 2).reshape(c, N, 3 * N)      # [l, (j, n)] = conj(dH_j[n][l])
        P = torch.bmm(Gh[nb[:, s].long()].reshape(c, F * N, N), right).reshape(c, F, N, 3, N)
        U = torch.stack([sum(K[:, s, :, i, j, None, None] * P[:, :, :, j] for j in range(3)) for i in range(3)], 1)
        U = U.permute(0, 1, 3, 2, 4).reshape(c, 3 * N, F * N)                  # [(i, m), (f, n)]
        left = dH[:, s].permute(0, 2, 1, 3).reshape(c, N, 3 * N)              # [m', (i, m)] = dH_i[m'][m]
        v = torch.bmm(left, U)
        acc = v if acc is None else acc + v
    S = _back((1j * SCALE * acc).reshape(c, N, F, N).permute(0, 2, 1, 3), Nkz, L, NE)
    return 0.5 * (S - S.conj().transpose(-1, -2)) if sym else S


def _exact_sigma(x, d, sym, W=None, want_g=False):
    L = _length(d.NE + d.Nw)
    Gh = [_spectrum(G, L).requires_grad_(want_g) for G in (x.G_less, x.G_greater)]
    S = [torch.empty_like(x.G_less) for _ in range(2)]
    gH, gD = torch.zeros_like(x.dH), [torch.zeros_like(x.D_less), torch.zeros_like(x.D_greater)]
    D = (x.D_less, x.D_greater)
    step = max(1, int(2.5e9 // (16 * d.Nkz * L * max(d.Norb ** 2, 9 * d.NB) * 12)))
    for a0 in range(0, d.NA, step):
        r = slice(a0, min(d.NA, a0 + step))
        dH = x.dH[r].clone().requires_grad_(W is not None)
        Dc = [t[:, :, r].clone().requires_grad_(W is not None) for t in D]
        for t in range(2):
            with torch.set_grad_enabled(W is not None):
                s = _forward(Gh[t], dH, Dc[t], Dc[1 - t], x.nbr[r], d.Nkz, L, d.NE, sym)
                if W is not None:
                    s.backward(W[t][:, :, r])
            S[t][:, :, r] = s.detach()
            del s
        if W is not None:
            gH[r] = dH.grad
            for t in range(2):
                gD[t][:, :, r] = Dc[t].grad
    gG = [_back(g.grad * (d.Nkz * L), d.Nkz, L, d.NE).contiguous() for g in Gh] if want_g else []
    return tuple(S), (gH, gD[0], gD[1]), tuple(gG)


def _exact_pi(x, d, sym):
    L = _length(d.NE + d.Nw)
    F = d.Nkz * L
    Gh = [_spectrum(G, L) for G in (x.G_less, x.G_greater)]
    k, e = torch.arange(d.Nkz, device="cuda"), torch.arange(L, device="cuda")
    neg = (((-k) % d.Nkz)[:, None] * L + ((-e) % L)[None, :]).reshape(-1)
    out = [torch.empty((d.Nqz, d.Nw, d.NA, d.NB + 1, 3, 3), dtype=torch.complex128, device="cuda") for _ in range(2)]
    step = max(1, int(2.5e9 // (16 * F * d.Norb ** 2 * 10)))
    N = d.Norb
    for a0 in range(0, d.NA, step):
        r = slice(a0, min(d.NA, a0 + step))
        dH, nb = x.dH[r], x.nbr[r].long()
        c = dH.shape[0]
        for t in range(2):
            total = None
            for s in range(d.NB + 1):
                if s < d.NB:
                    h = dH[:, s]
                    E = torch.bmm(Gh[t][r].reshape(c, F * N, N), h.permute(0, 2, 1, 3).reshape(c, N, 3 * N))
                    Y = Gh[1 - t][nb[:, s]][:, neg].reshape(c, F * N, N)
                    Q = torch.bmm(Y, h.conj().permute(0, 3, 1, 2).reshape(c, N, 3 * N))  # Y dH_i^H
                    E = E.reshape(c * F, N, 3, N).permute(0, 2, 1, 3).reshape(c * F, 3, N * N)   # j, (m, n)
                    Q = Q.reshape(c * F, N, 3, N).permute(0, 2, 3, 1).reshape(c * F, 3, N * N)   # i, (m, n) <- [n, m]
                    C = torch.bmm(Q, E.transpose(1, 2)).reshape(c, F, 3, 3)
                    total = C if total is None else total + C
                else:
                    C = total
                v = -1j * SCALE * _back(C, d.Nkz, L, d.Nw + 1)[:d.Nqz, 1:]
                out[t][:, :, r, s] = 0.5 * (v - v.conj().transpose(-1, -2)) if sym else v
    return tuple(out)


def _reverse_slots(nbr):
    """rev[a, s] = the slot s' with nbr[nbr[a, s], s'] = a (the first one)."""
    nb = nbr.long()
    hit = nb[nb] == torch.arange(nb.shape[0], device=nb.device)[:, None, None]
    return hit.to(torch.int64).argmax(-1)


def _exact_dcomb(st):
    nb = st["nbr"].long()
    rev = _reverse_slots(nb)
    NB = nb.shape[1]
    rl, rg, gl, gg = st["raw"]

    def pick(x):
        return x[:, :, nb, rev]

    fwd = [pick(r) - r[:, :, :, NB][:, :, nb] - r[:, :, :, NB:NB + 1] + r[:, :, :, :NB] for r in (rl, rg)]
    bwd = []
    for g in (gl, gg):
        both = g + pick(g)
        bwd.append(torch.cat([both, -both.sum(3, keepdim=True)], dim=3))
    return tuple(fwd) + tuple(bwd)


def exact(case, seed):
    d, op, sym = _dims(case), case["op"], case["symmetrize"]
    if op == "dcomb":
        return _exact_dcomb(prepare(case, seed))
    x = make_inputs(d, seed=seed, device="cuda")
    if op == "pi":
        return _exact_pi(x, d, sym)
    if op in ("sigma", "host"):
        return _exact_sigma(x, d, sym)[0]
    W = make_upstream(d, seed=seed + 1, device="cuda")
    S, g, gG = _exact_sigma(x, d, sym, W, want_g=op in ("step", "grad_g"))
    return g if op == "grad" else gG if op == "grad_g" else S + g + gG
