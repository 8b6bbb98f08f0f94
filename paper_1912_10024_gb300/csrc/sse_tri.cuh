// Transforms of anti-Hermitian blocks (SSE_FLAG_ANTIHERMITIAN) by their upper triangle. With G(E, k) = -G(E, k)^H block by
// block, G^_nm(f) = -conj(G^_mn(-f)): the Norb (Norb + 1) / 2 elements m <= n hold the whole spectrum, and the same is true
// of Sigma. So G is transformed along E for those columns only, the kz DFT that follows writes the full blocks of the
// computed half of the frequencies (and of the other half where Pi needs it), and after the products the inverse kz DFT
// reads that half and writes the triangle's columns for every frequency. 0.55 of the E-transforms at Norb = 10, half of
// the kz passes, no mirror pass, no separate symmetrisation (symmetrised FP32 spectra excepted: mirrored, transformed back
// in full and averaged in FP64). The 3 x 3 blocks of the lag kernel are taken the same way (six columns of nine). FinFET in FP64 (the transforms are bound by the FP64 pipe): E-transforms of G and S 102 -> 58 ms, of K
// 17.6 -> 11.8; kz passes 36 -> 21 ms, mirror 3.6 -> 0: the call 830 -> 761 ms.
#pragma once

#include "sse_spectral.cuh"

namespace sse {
namespace {

constexpr int kTriMaxNorb = 16, kTriMax = kTriMaxNorb * (kTriMaxNorb + 1) / 2;
// kz grids with an instantiation of the kernels below: up to 8 the two FP64 columns of a thread leave registers for two CTAs
// per SM (compress: 124 at Nkz = 8, 170 at 12, 230 at 16). Larger grids take the full columns; not measured there.
constexpr int kTriMaxNk = 8;

struct TriMap {  // the upper triangle of an n x n block, row by row
    int nt, nel;
    uint8_t at[kTriMax], tr[kTriMax];  // offset of (m, n) and of (n, m) in the block
};
inline TriMap make_tri_map(int n) {
    TriMap t{};
    t.nel = n * n;
    for (int r = 0; r < n; ++r)
        for (int c = r; c < n; ++c) {
            t.at[t.nt] = (uint8_t)(r * n + c);
            t.tr[t.nt++] = (uint8_t)(c * n + r);
        }
    return t;
}

// G^t[k][E][atom][mn] of the triangle's columns, rows E >= NE are zero
template <class CC>
struct LoadGTri {
    using C = CC;
    const double2* G;
    int NE;
    size_t rowlen;
    TriMap t;
    __device__ C operator()(int k, int r, size_t col) const {
        if (r >= NE) return CT<C>::mk(0, 0);
        const unsigned a = (unsigned)col / (unsigned)t.nt;
        const double2 v = G[((size_t)k * NE + r) * rowlen + (size_t)a * t.nel + t.at[(unsigned)col - a * t.nt]];
        return CT<C>::mk(v.x, v.y);
    }
};

// lag kernel of one qz slice (LoadLagT) for the triangle of its 3 x 3 blocks: row w + 1 <- D^t(q, w), row L - (w + 1) <-
// D^t'(q, w), else zero
template <class CC>
struct LoadLagTri {
    using C = CC;
    const double2* Dt;
    const double2* Dtb;
    int Nw, L;
    size_t rowlen, col0;
    TriMap t;
    __device__ C operator()(int q, int r, size_t col) const {
        const bool up = r >= 1 && r <= Nw, down = r >= L - Nw;
        if (!up && !down) return CT<C>::mk(0, 0);
        const unsigned b = (unsigned)col / (unsigned)t.nt;
        const size_t at = (size_t)b * t.nel + t.at[(unsigned)col - b * t.nt];
        const double2 v = (up ? Dt : Dtb)[((size_t)q * Nw + (up ? r - 1 : L - 1 - r)) * rowlen + col0 + at];
        return CT<C>::mk(v.x, v.y);
    }
};

// S[k][E][a_begin * nel + atom * nel + mn] = conj(v) * inv and its partner -conj at nm, E < NE; with sym the diagonal's
// real part (rounding) is cleared, as (S - S^H) / 2 does
template <class C>
struct StoreSigmaTri {
    double2* S;
    int NE;
    size_t rowlen, col0;
    double inv;
    int rows, sym;
    TriMap t;
    __device__ void operator()(int k, int r, size_t col, C v) const {
        using R = typename CT<C>::R;
        const R s = (R)inv;
        const unsigned a = (unsigned)col / (unsigned)t.nt, i = (unsigned)col - a * t.nt;
        double2* o = S + ((size_t)k * NE + r) * rowlen + col0 + (size_t)a * t.nel;
        const double2 w = make_double2((double)(v.x * s), (double)(-v.y * s));
        const int at = t.at[i], tr = t.tr[i];
        if (at == tr) {
            o[at] = make_double2(sym ? 0.0 : w.x, w.y);
        } else {
            o[at] = w;
            o[tr] = make_double2(-w.x, w.y);
        }
    }
};

__device__ __forceinline__ double2 cnegconj(double2 a) { return make_double2(-a.x, a.y); }
__device__ __forceinline__ float2 cnegconj(float2 a) { return make_float2(-a.x, a.y); }

// forward kz DFT of the triangle's columns X[k < n_in][eps][block][i] into full blocks G[kappa][eps][block][mn] for eps <= L / 2,
// and for every eps with `both`. A thread takes the rows eps and L - eps of one column.
template <class C, int NK>
__global__ void __launch_bounds__(256) dft_kz_expand_kernel(const C* __restrict__ X, C* __restrict__ G, TriMap t, int n_in,
                                                            int L, unsigned ncols, int both) {
    const size_t total = (size_t)(L / 2 + 1) * ncols;
    const size_t gcols = (size_t)(ncols / t.nt) * t.nel;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int e = (int)(i / ncols), em = e == 0 ? 0 : L - e;
        const unsigned col = (unsigned)(i - (size_t)e * ncols), a = col / (unsigned)t.nt, k0 = col - a * t.nt;
        const int at = t.at[k0], tr = t.tr[k0];
        C x[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) x[k] = k < n_in ? X[((size_t)k * L + e) * ncols + col] : CT<C>::mk(0, 0);
        C* g = G + (size_t)e * gcols + (size_t)a * t.nel;    // row eps
        C* gm = G + (size_t)em * gcols + (size_t)a * t.nel;  // row -eps
        const size_t slab = (size_t)L * gcols;
        const bool self = e == em, diag = at == tr;
        kz_dft<C, NK>(x, 0, [&](int kap, C v) {
            const int km = kap == 0 ? 0 : NK - kap;
            g[kap * slab + at] = v;
            if (self ? !diag : both) gm[km * slab + tr] = cnegconj(v);
        });
        if (self || diag) continue;
#pragma unroll
        for (int k = 0; k < NK; ++k) x[k] = k < n_in ? X[((size_t)k * L + em) * ncols + col] : CT<C>::mk(0, 0);
        kz_dft<C, NK>(x, 0, [&](int kap, C v) {
            const int km = kap == 0 ? 0 : NK - kap;
            g[km * slab + tr] = cnegconj(v);
            if (both) gm[kap * slab + at] = v;
        });
    }
}

// inverse kz DFT of the full blocks S[kappa][eps][atom][mn], eps <= L / 2 (on the rows eps = -eps: kappa <= NK / 2), into
// the triangle's columns X[k][eps][atom][i] of every eps
template <class C, int NK>
__global__ void __launch_bounds__(256) dft_kz_compress_kernel(const C* __restrict__ S, C* __restrict__ X, TriMap t, int L,
                                                              unsigned ncols) {
    const size_t total = (size_t)(L / 2 + 1) * ncols;
    const size_t scols = (size_t)(ncols / t.nt) * t.nel;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int e = (int)(i / ncols), em = e == 0 ? 0 : L - e;
        const unsigned col = (unsigned)(i - (size_t)e * ncols), a = col / (unsigned)t.nt, k0 = col - a * t.nt;
        const C* s = S + (size_t)e * scols + (size_t)a * t.nel;
        const size_t slab = (size_t)L * scols;
        const bool self = e == em;
        C x[NK], u[NK];  // rows eps and -eps of element (m, n)
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const int km = k == 0 ? 0 : NK - k;
            if (!self || k <= NK / 2) x[k] = s[k * slab + t.at[k0]];
            if (!self || km <= NK / 2) u[k] = cnegconj(s[km * slab + t.tr[k0]]);
        }
        if (self)
#pragma unroll
            for (int k = NK / 2 + 1; k < NK; ++k) x[k] = u[k];
        kz_dft<C, NK>(x, 1, [&](int k, C v) { X[((size_t)k * L + e) * ncols + col] = v; });
        if (!self) kz_dft<C, NK>(u, 1, [&](int k, C v) { X[((size_t)k * L + em) * ncols + col] = v; });
    }
}

// Symmetrised Sigma of general inputs, FP64 spectra: the spectrum of (S - S^H) / 2 is (S^_mn(f) - conj(S^_nm(-f))) / 2,
// anti-Hermitian, so its triangle is enough. Inverse kz DFT of twice that from the full blocks S[kappa][eps][atom][mn] into
// the triangle's columns (the store halves it): the symmetrisation costs no pass of its own and 0.45 of the inverse
// E-transform goes away. FP64_FFT, both types, kz pass, inverse E-transform and symmetrisation: NA = 90, Norb = 7, NE = 301,
// Nkz = 4 993 -> 585 us, NA = 256, Norb = 10, NE = 256, Nkz = 5 6.01 -> 3.27 ms. Not for FP32 spectra: there the projection would round to 24 bits what symmetrize_kernel averages
// in FP64.
template <class C, int NK>
__global__ void __launch_bounds__(256) dft_kz_project_kernel(const C* __restrict__ S, C* __restrict__ X, TriMap t, int L,
                                                             unsigned ncols) {
    const size_t total = (size_t)(L / 2 + 1) * ncols;
    const size_t scols = (size_t)(ncols / t.nt) * t.nel;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int e = (int)(i / ncols), em = e == 0 ? 0 : L - e;
        const unsigned col = (unsigned)(i - (size_t)e * ncols), a = col / (unsigned)t.nt, k0 = col - a * t.nt;
        const C* s = S + (size_t)e * scols + (size_t)a * t.nel;    // row eps
        const C* sm = S + (size_t)em * scols + (size_t)a * t.nel;  // row -eps
        const int at = t.at[k0], tr = t.tr[k0];
        const size_t slab = (size_t)L * scols;
        C x[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) x[k] = cadd(s[k * slab + at], cnegconj(sm[((NK - k) % NK) * slab + tr]));
        kz_dft<C, NK>(x, 1, [&](int k, C v) { X[((size_t)k * L + e) * ncols + col] = v; });
        if (e == em) continue;
#pragma unroll
        for (int k = 0; k < NK; ++k) x[k] = cadd(sm[k * slab + at], cnegconj(s[((NK - k) % NK) * slab + tr]));
        kz_dft<C, NK>(x, 1, [&](int k, C v) { X[((size_t)k * L + em) * ncols + col] = v; });
    }
}

// The triangle's columns fit 32 bits and the kz grid has an instantiation; `room` complex entries of scratch hold the
// triangle's spectrum of all atoms (the region of S^: large enough unless few of the atoms are targets).
inline bool tri_applies(const sse_dims& d, int L, size_t room) {
    const size_t cols = (size_t)d.NA * (d.Norb * (d.Norb + 1) / 2);
    return d.Norb <= kTriMaxNorb && d.Nkz <= kTriMaxNk && cols <= 0x7fffffffu && (size_t)d.Nkz * L * cols <= room;
}

template <class F>
cudaError_t tri_with_nk(int nk, F&& f) {
    switch (nk) {
        case 1: return f(std::integral_constant<int, 1>{});
        case 2: return f(std::integral_constant<int, 2>{});
        case 3: return f(std::integral_constant<int, 3>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 7: return f(std::integral_constant<int, 7>{});
        case 8: return f(std::integral_constant<int, 8>{});
        default: return cudaErrorInvalidValue;
    }
}

template <class C>
cudaError_t launch_kz_expand(const char* name, const C* X, C* G, const TriMap& t, int Nk, int n_in, int L, size_t ncols,
                             bool both, cudaStream_t st) {
    return tri_with_nk(Nk, [&](auto nk) {
        SSE_TIMED(name, st,
                  dft_kz_expand_kernel<C, decltype(nk)::value>
                  <<<grid_for((size_t)(L / 2 + 1) * ncols, 256), 256, 0, st>>>(X, G, t, n_in, L, (unsigned)ncols, both ? 1 : 0));
        return cudaGetLastError();
    });
}

template <class C>
cudaError_t launch_kz_compress(const char* name, const C* S, C* X, const TriMap& t, int Nk, int L, size_t ncols,
                               cudaStream_t st) {
    return tri_with_nk(Nk, [&](auto nk) {
        SSE_TIMED(name, st,
                  dft_kz_compress_kernel<C, decltype(nk)::value>
                  <<<grid_for((size_t)(L / 2 + 1) * ncols, 256), 256, 0, st>>>(S, X, t, L, (unsigned)ncols));
        return cudaGetLastError();
    });
}

template <class C>
cudaError_t launch_kz_project(const char* name, const C* S, C* X, const TriMap& t, int Nk, int L, size_t ncols,
                              cudaStream_t st) {
    return tri_with_nk(Nk, [&](auto nk) {
        SSE_TIMED(name, st,
                  dft_kz_project_kernel<C, decltype(nk)::value>
                  <<<grid_for((size_t)(L / 2 + 1) * ncols, 256), 256, 0, st>>>(S, X, t, L, (unsigned)ncols));
        return cudaGetLastError();
    });
}

}  // namespace
}  // namespace sse
