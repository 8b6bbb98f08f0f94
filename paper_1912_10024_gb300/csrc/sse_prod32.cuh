// FP32 block products of the transform path on wide register tiles (Sigma forward and the gradient in G, mode
// FP32_FFT). Per target atom and frequency f, over the bonds of the target,
//
//   P_j = X(f) T_j^H  (j = 0..2),   U_i = sum_j k_ij(f) P_j,   acc += sum_i T_i U_i,
//
// with X = G^_b, T_j = dH_j, k = K^ for the forward, and X = W^_a, T_j = dH_j^H, k = conj(K^) over the incoming bonds
// for the gradient in G: one kernel serves both.
//
// What bounds it: the shared-memory return path (128 bytes per clock and SM, also for a broadcast: a 16-byte load by a warp
// takes 4 clocks, the issue time of 16 warp-wide FMAs) and, next to it, the FP32 pipe (128 FMA per clock and SM, 80
// TFLOP/s). A thread therefore owns half of the rows and two columns of the block, for the three j together and for NF
// frequencies: at Np = 10 (NF = 1) P takes 5.5 FMAs and acc 2.9 per float loaded, against 2 on 2 x 2 tiles for the P_j one
// frequency at a time. FinFET workload, per step of two types: 52.3 -> 36.6 ms (0.62 of the FP32 pipe; ncu at the
// adjoint workload: shared-memory wavefronts 72% of peak, FMA pipe 69% active, three warps per scheduler).
#pragma once

#include "sse_spectral.cuh"

namespace sse {
namespace {

__device__ __forceinline__ float2 f2dup(float a) { return make_float2(a, a); }

// c + a * b on a pair of floats: one issue slot for two FMAs, the same rate on the FP32 pipe (measured 79.8 against
// 76.2 TFLOP/s for chains of fmaf). The slots it frees carry the operand loads: Sigma's products at the FinFET
// workload take 37.2 ms per step with it, 42.3 with fmaf.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n.reg .b64 ra, rb, rc, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nmov.b64 rc, {%6, %7};\n"
        "fma.rn.f32x2 rd, ra, rb, rc;\nmov.b64 {%0, %1}, rd;\n}\n"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

// -a on the integer pipe (the FMA pipe is the busy one)
__device__ __forceinline__ float2 f2neg(float a, float b) {
    return make_float2(__uint_as_float(__float_as_uint(a) ^ 0x80000000u), __uint_as_float(__float_as_uint(b) ^ 0x80000000u));
}

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

template <int B>
__device__ __forceinline__ void tile_cp_async(float* dst, const void* src, bool ok) {
    cp_async_elem<B>((uint32_t)__cvta_generic_to_shared(dst), src, ok);
}
__device__ __forceinline__ void tile_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tile_cp_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// One N x N complex block (row-major in global memory) into rows of NP complex; ok = false fills with zeros. Work item
// i < ITEMS.
template <int NP, int ODD>
struct TileCopy {
    static constexpr int N = NP - ODD;
    static constexpr int ITEMS = ODD ? N * N : N * N / 2;
    __device__ __forceinline__ static void run(float* dst, const float2* src, int i, bool ok) {
        if constexpr (ODD) {
            tile_cp_async<8>(dst + ((i / N) * NP + i % N) * 2, src + i, ok);
        } else {
            tile_cp_async<16>(dst + i * 4, src + 2 * i, ok);
        }
    }
};

template <int NP>
struct TileShape {
    static constexpr int RH = NP / 2;               // rows per thread
    static constexpr int CP = NP / 2;               // column pairs
    static constexpr int TPF = 2 * CP;              // threads per frequency set
    static constexpr int NF = NP <= 6 ? 2 : 1;      // frequencies per thread: two while their tiles fit in registers
    // CTAs per SM that the registers (P 12 Np NF / 2, acc 2 Np NF, operands) leave room for with at most 16 bytes of spills
    // (Np = 4, 6, 8 and 12; none at 10). Measured at Norb = 10: NF = 1 with three CTAs 36.6 ms per FinFET step, NF = 2 with two 37.1, NF = 1 with four (spills) 45.8; at
    // Norb = 12 (gradient in G, NA = 200): NF = 1 with three CTAs 3.8 ms, with two 4.2. Norb = 8 (NA = 256, NE = 256, Nkz = 5):
    // NF = 1 with four CTAs 1.79 ms, NF = 2 with two 1.84, NF = 1 with three 1.90; Norb = 6: NF = 2 0.90, NF = 1 0.97.
    static constexpr int CTAS = NP <= 4 || NP == 8 ? 4 : NP <= 12 ? 3 : 2;
    static constexpr int XS = NP * NP * 2;          // floats of X per frequency
    static constexpr int US = 3 * NP * NP * 2;      // floats of U per frequency
    static constexpr int RSTR = (NP + 1) * 4;       // floats per column pair of the right operand (odd: bank spread)
    static constexpr int RB = 3 * CP * RSTR;        // floats of the right operand per bond
    static constexpr int LB = 3 * NP * NP * 2;      // floats of the left operand per bond
    static constexpr int FGMAX = 128 / TPF;         // frequency sets per CTA
};

struct TileCfg {
    int fg, F, threads, fchunk, nchunks, nres;
    int off_L, off_R, off_X, off_U, off_K, off_F, smem;
};

// nb: bonds a target may have (their dH operands stay resident where they fit beside the
// buffers of S::CTAS CTAs), ntgt: targets
template <int NP>
TileCfg make_tile_cfg(int nb, size_t ntgt, size_t nfreq) {
    using S = TileShape<NP>;
    auto a16 = [](int x) { return (x + 15) & ~15; };
    TileCfg c{};
    auto place = [&](int fg, int nres) {
        c.fg = fg;
        c.nres = nres;
        c.F = fg * S::NF;
        c.threads = (fg * S::TPF + 31) / 32 * 32;
        c.off_L = 0;
        c.off_R = a16(c.off_L + nres * S::LB * 4);
        c.off_X = a16(c.off_R + nres * S::RB * 4);
        c.off_U = a16(c.off_X + c.F * S::XS * 4);
        c.off_K = a16(c.off_U + c.F * S::US * 4);
        c.off_F = a16(c.off_K + c.F * 9 * 8);
        c.smem = c.off_F + 2 * c.F * 8;
        return c.smem;
    };
    const int room = (227 / S::CTAS - 1) * 1024;
    bool ok = false;
    for (int fg = S::FGMAX; !ok && fg >= 1 && 2 * fg >= S::FGMAX; --fg) ok = place(fg, nb) <= room;
    if (!ok) place(S::FGMAX, 1);  // the operands of one bond at a time
    // tiles per CTA: enough CTAs for ~8 waves, at most 8 tiles (the dH operands are staged per CTA)
    const size_t tiles = (nfreq + c.F - 1) / c.F;
    const size_t want = (size_t)152 * S::CTAS * 8;
    size_t per = tiles * ntgt / want;
    per = per < 1 ? 1 : per > 8 ? 8 : per;
    c.fchunk = (int)per;
    c.nchunks = (int)((tiles + per - 1) / per);
    return c;
}

struct TileArgs {
    sse_dims d;
    FreqMap fm;
    const int32_t* nbr;   // forward: neighbour list
    const int* off;       // gradient in G: incoming bonds of each atom
    const int* list;
    const double2* dH;
    const float2* X;      // forward: G^ [f][NA][nel]; gradient: W^ [f][nA][nel]
    const float2* K;      // [f][nA][NB][9]
    float2* out;          // forward: S^ [f][nA][nel]; gradient: R^ [f][NA][nel]
    double scale;
    unsigned* status;
};

template <int NP, int ODD, bool GRADG>
__global__ void __launch_bounds__(128, TileShape<NP>::CTAS) spec_prod32_kernel(TileCfg c, TileArgs p) {
    using S = TileShape<NP>;
    using Cp = TileCopy<NP, ODD>;
    constexpr int N = NP - ODD, nel = N * N, RH = S::RH, CP = S::CP, NF = S::NF;
    extern __shared__ __align__(16) unsigned char smem[];
    float* sL = reinterpret_cast<float*>(smem + c.off_L);   // [res][3 i][NP m'][NP m] T_i
    float* sR = reinterpret_cast<float*>(smem + c.off_R);   // [res][3 j][CP][NP + 1 l] (re, re, im, im) of conj(T_j[n][l])
    float* sX = reinterpret_cast<float*>(smem + c.off_X);   // [F][NP m][NP l]
    float* sU = reinterpret_cast<float*>(smem + c.off_U);   // [F][3 i][NP m][CP] (re, re, im, im)
    float2* sK = reinterpret_cast<float2*>(smem + c.off_K);  // [F][9]
    long long* sF = reinterpret_cast<long long*>(smem + c.off_F);  // [2 tiles][F] frequency of each slot, -1: none
    const int tid = threadIdx.x, nt = blockDim.x;
    const sse_dims& d = p.d;
    const int nA = d.a_end - d.a_begin;
    const int tgt = blockIdx.x;
    const int i0 = GRADG ? p.off[tgt] : 0;
    const int nb = GRADG ? p.off[tgt + 1] - i0 : d.NB;
    const size_t nX = GRADG ? (size_t)nA : (size_t)d.NA, nK = (size_t)nA * d.NB;
    const size_t nO = GRADG ? (size_t)d.NA : (size_t)nA;
    const int ntiles_all = (int)((p.fm.count + c.F - 1) / c.F);
    const int tile0 = blockIdx.y * c.fchunk, tile1 = min(ntiles_all, tile0 + c.fchunk);
    const bool resident = nb <= c.nres;

    const int fs = tid / S::TPF, tt = tid - fs * S::TPF;
    const int m0 = (tt / CP) * RH, cp = tt % CP;
    const bool lane = fs < c.fg;

    // bond ib of the target: row of X (-1: neighbour out of range, contributes zero) and bond index in K
    auto bond = [&](int ib, int& xrow, int& kidx) {
        if (GRADG) {
            kidx = p.list[i0 + ib];
            xrow = kidx / d.NB;
        } else {
            kidx = tgt * d.NB + ib;
            const int b = p.nbr[(size_t)d.a_begin * d.NB + kidx];
            xrow = (b >= 0 && b < d.NA) ? b : -1;
        }
    };
    auto stage_T = [&](int ib, int slot) {
        int xrow, kidx;
        bond(ib, xrow, kidx);
        const double2* H = p.dH + ((size_t)d.a_begin * d.NB + kidx) * 3 * nel;
        float* L = sL + (size_t)slot * S::LB;
        float* R = sR + (size_t)slot * S::RB;
        for (int i = tid; i < 3 * NP * NP; i += nt) {
            const int j = i / (NP * NP), e = i - j * (NP * NP), r = e / NP, q = e - r * NP;
            float2 v = make_float2(0.f, 0.f);  // T_j[r][q]
            if (r < N && q < N) {
                const double2 h = GRADG ? H[j * nel + q * N + r] : H[j * nel + r * N + q];
                v = make_float2((float)h.x, GRADG ? -(float)h.y : (float)h.y);
            }
            reinterpret_cast<float2*>(L)[i] = v;
            float* o = R + (j * CP + r / 2) * S::RSTR + q * 4 + (r & 1);
            o[0] = v.x;
            o[2] = -v.y;
        }
        if (!GRADG && xrow < 0 && tid == 0) atomicOr(p.status, DEV_BAD_NEIGHBOUR);
    };
    auto freq_table = [&](int tile) {
        for (int i = tid; i < c.F; i += nt) {
            const size_t ix = (size_t)tile * c.F + i;
            sF[(tile & 1) * c.F + i] = ix < p.fm.count ? (long long)freq_of(p.fm, ix) : -1ll;
        }
    };
    auto issue = [&](int tile, int ib) {
        int xrow, kidx;
        bond(ib, xrow, kidx);
        const long long* fq = sF + (tile & 1) * c.F;
        for (int i = tid; i < c.F * Cp::ITEMS; i += nt) {
            const int f = i / Cp::ITEMS, e = i - f * Cp::ITEMS;
            const long long g = fq[f];
            const bool ok = g >= 0 && xrow >= 0;
            Cp::run(sX + (size_t)f * S::XS, ok ? p.X + ((size_t)g * nX + xrow) * nel : p.X, e, ok);
        }
        for (int i = tid; i < c.F * 9; i += nt) {
            const int f = i / 9, e = i - f * 9;
            const long long g = fq[f];
            const bool ok = g >= 0 && xrow >= 0;
            tile_cp_async<8>(reinterpret_cast<float*>(sK + i), ok ? p.K + ((size_t)g * nK + kidx) * 9 + e : p.K, ok);
        }
        tile_cp_commit();
    };

    if (ODD)  // padding rows and columns of X stay zero (the copies never write them)
        for (int i = tid; i < c.F * S::XS; i += nt) sX[i] = 0.f;
    freq_table(tile0);
    if (resident)
        for (int ib = 0; ib < nb; ++ib) stage_T(ib, ib);
    __syncthreads();
    if (nb > 0 && tile0 < tile1) issue(tile0, 0);

    for (int tile = tile0; tile < tile1; ++tile) {
        if (tile + 1 < tile1) freq_table(tile + 1);  // read after the barriers below
        float2 ar[NF][RH], ai[NF][RH];
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
            for (int r = 0; r < RH; ++r) ar[f][r] = ai[f][r] = make_float2(0.f, 0.f);
        for (int ib = 0; ib < nb; ++ib) {
            const int slot = resident ? ib : 0;
            tile_cp_wait();
            __syncthreads();  // X and K have landed; the previous bond's reads of U (and of T) are done
            if (!resident) {
                stage_T(ib, 0);
                __syncthreads();
            }
            if (lane) {
                const float* R = sR + (size_t)slot * S::RB + cp * S::RSTR;
                const float* X = sX + (size_t)fs * S::XS + m0 * NP * 2;
                float2 pr[NF][3][RH], pi[NF][3][RH];
#pragma unroll
                for (int f = 0; f < NF; ++f)
#pragma unroll
                    for (int j = 0; j < 3; ++j)
#pragma unroll
                        for (int r = 0; r < RH; ++r) pr[f][j][r] = pi[f][j][r] = make_float2(0.f, 0.f);
#pragma unroll
                for (int l = 0; l < NP; l += 2) {
                    float4 g[NF][RH];  // X[m0 + r][l], X[m0 + r][l + 1]
#pragma unroll
                    for (int f = 0; f < NF; ++f)
#pragma unroll
                        for (int r = 0; r < RH; ++r) g[f][r] = lds4(X + (size_t)f * c.fg * S::XS + (r * NP + l) * 2);
#pragma unroll
                    for (int dl = 0; dl < 2; ++dl)
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            if (l + dl >= N) continue;  // the padding column of an odd block
                            const float4 b = lds4(R + j * CP * S::RSTR + (l + dl) * 4);
                            const float2 br = lo2(b), bi = hi2(b), nbi = f2neg(b.z, b.w);
#pragma unroll
                            for (int f = 0; f < NF; ++f)
#pragma unroll
                                for (int r = 0; r < RH; ++r) {
                                    const float x = dl ? g[f][r].z : g[f][r].x, y = dl ? g[f][r].w : g[f][r].y;
                                    pr[f][j][r] = fma2(f2dup(x), br, pr[f][j][r]);
                                    pi[f][j][r] = fma2(f2dup(x), bi, pi[f][j][r]);
                                    pr[f][j][r] = fma2(f2dup(y), nbi, pr[f][j][r]);
                                    pi[f][j][r] = fma2(f2dup(y), br, pi[f][j][r]);
                                }
                        }
                }
                // U_i = sum_j k_ij P_j, element by element
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const float2* K = sK + (fs + f * c.fg) * 9;
                    float2 k[9];
#pragma unroll
                    for (int ij = 0; ij < 9; ++ij) {
                        k[ij] = K[ij];
                        if (GRADG) k[ij].y = -k[ij].y;
                    }
                    float* U = sU + (size_t)(fs + f * c.fg) * S::US + (m0 * CP + cp) * 4;
#pragma unroll
                    for (int r = 0; r < RH; ++r)
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            float2 ur = make_float2(0.f, 0.f), ui = ur;
#pragma unroll
                            for (int j = 0; j < 3; ++j) {
                                const float2 kk = k[i * 3 + j];
                                ur = fma2(f2dup(kk.x), pr[f][j][r], ur);
                                ui = fma2(f2dup(kk.x), pi[f][j][r], ui);
                                ur = fma2(f2dup(-kk.y), pi[f][j][r], ur);
                                ui = fma2(f2dup(kk.y), pr[f][j][r], ui);
                            }
                            *reinterpret_cast<float4*>(U + (i * NP + r) * CP * 4) = make_float4(ur.x, ur.y, ui.x, ui.y);
                        }
                }
            }
            __syncthreads();  // U is complete, X and K are free
            {
                const bool last = ib + 1 == nb;
                if (!last) issue(tile, ib + 1);
                else if (tile + 1 < tile1) issue(tile + 1, 0);
            }
            if (lane) {
                const float* L = sL + (size_t)slot * S::LB + m0 * NP * 2;
                const float* U = sU + (size_t)fs * S::US + cp * 4;
#pragma unroll 1
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int m = 0; m < NP; m += 2) {
                        float4 t[RH];
#pragma unroll
                        for (int r = 0; r < RH; ++r) t[r] = lds4(L + (i * NP * NP + r * NP + m) * 2);
#pragma unroll
                        for (int dm = 0; dm < 2; ++dm)
#pragma unroll
                            for (int f = 0; f < NF; ++f) {
                                if (m + dm >= N) continue;
                                const float4 u = lds4(U + (size_t)f * c.fg * S::US + (i * NP + m + dm) * CP * 4);
                                const float2 ur = lo2(u), ui = hi2(u), nui = f2neg(u.z, u.w);
#pragma unroll
                                for (int r = 0; r < RH; ++r) {
                                    const float x = dm ? t[r].z : t[r].x, y = dm ? t[r].w : t[r].y;
                                    ar[f][r] = fma2(f2dup(x), ur, ar[f][r]);
                                    ai[f][r] = fma2(f2dup(x), ui, ai[f][r]);
                                    ar[f][r] = fma2(f2dup(y), nui, ar[f][r]);
                                    ai[f][r] = fma2(f2dup(y), ur, ai[f][r]);
                                }
                            }
                    }
            }
        }
        if (lane) {
            const float sc = GRADG ? -(float)p.scale : (float)p.scale;  // times i*sc
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const size_t ix = (size_t)tile * c.F + fs + f * c.fg;
                if (ix >= p.fm.count) continue;
                float2* o = p.out + (freq_of(p.fm, ix) * nO + tgt) * nel;
#pragma unroll
                for (int r = 0; r < RH; ++r) {
                    const int m = m0 + r, n = 2 * cp;
                    const float2 v0 = make_float2(-sc * ai[f][r].x, sc * ar[f][r].x);
                    const float2 v1 = make_float2(-sc * ai[f][r].y, sc * ar[f][r].y);
                    if (!ODD) {
                        *reinterpret_cast<float4*>(o + m * N + n) = make_float4(v0.x, v0.y, v1.x, v1.y);
                    } else if (m < N) {
                        o[m * N + n] = v0;
                        if (n + 1 < N) o[m * N + n + 1] = v1;
                    }
                }
            }
        }
    }
    tile_cp_wait();
}

template <int NP, int ODD, bool GRADG>
cudaError_t launch_prod32_t(const TileArgs& p, size_t ntgt, cudaStream_t st) {
    const TileCfg c = make_tile_cfg<NP>(p.d.NB, ntgt, p.fm.count);
    auto kern = spec_prod32_kernel<NP, ODD, GRADG>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, c.smem);
    if (e != cudaSuccess) return e;
    if (ntgt == 0 || c.nchunks == 0) return cudaSuccess;
    if (c.nchunks > 65535) return cudaErrorInvalidValue;
    SSE_TIMED(GRADG ? "spec_gradg_kernel" : "spec_prod32_kernel", st,
              kern<<<dim3((unsigned)ntgt, (unsigned)c.nchunks), c.threads, c.smem, st>>>(c, p));
    return cudaGetLastError();
}

template <bool GRADG>
cudaError_t launch_prod32(const TileArgs& p, size_t ntgt, cudaStream_t st) {
    switch (p.d.Norb) {
        case 1: return launch_prod32_t<2, 1, GRADG>(p, ntgt, st);
        case 2: return launch_prod32_t<2, 0, GRADG>(p, ntgt, st);
        case 3: return launch_prod32_t<4, 1, GRADG>(p, ntgt, st);
        case 4: return launch_prod32_t<4, 0, GRADG>(p, ntgt, st);
        case 5: return launch_prod32_t<6, 1, GRADG>(p, ntgt, st);
        case 6: return launch_prod32_t<6, 0, GRADG>(p, ntgt, st);
        case 7: return launch_prod32_t<8, 1, GRADG>(p, ntgt, st);
        case 8: return launch_prod32_t<8, 0, GRADG>(p, ntgt, st);
        case 9: return launch_prod32_t<10, 1, GRADG>(p, ntgt, st);
        case 10: return launch_prod32_t<10, 0, GRADG>(p, ntgt, st);
        case 11: return launch_prod32_t<12, 1, GRADG>(p, ntgt, st);
        case 12: return launch_prod32_t<12, 0, GRADG>(p, ntgt, st);
        case 13: return launch_prod32_t<14, 1, GRADG>(p, ntgt, st);
        case 14: return launch_prod32_t<14, 0, GRADG>(p, ntgt, st);
        case 15: return launch_prod32_t<16, 1, GRADG>(p, ntgt, st);
        case 16: return launch_prod32_t<16, 0, GRADG>(p, ntgt, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace
}  // namespace sse
