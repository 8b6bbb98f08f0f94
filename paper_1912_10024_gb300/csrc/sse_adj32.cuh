// FP32 adjoint products of the transform path (mode FP32_FFT of the gradients in dH and D). Per bond (a, s),
// b = nbr[a][s], and frequency f, with W = W^_a(f), G = G^_b(f), A_j = dH_j, k = K^(f), c = i * scale:
//
//   T_j = W A_j,  B_i = A_i G                                        (phase 1: A shared by every frequency)
//   H^_ij = tr(A_i^H W A_j G^H) = sum_mn T_j[m][n] conj(B_i[m][n])     (the gradient in D, before its transform)
//   grad dH_mu += sum_f X_mu G^H + W^H U_mu,  X_mu = sum_j conj(c k_mu,j) T_j,  U_mu = sum_i c k_i,mu B_i  (phase 2)
//
// 12 block products, and the traces come from the registers that hold T_j and B_i. The second sum runs over the
// frequencies as well, so its 3 x Norb^2 sums stay in registers from tile to tile.
//
// What bounds it: the FP32 pipe and the shared-memory return path (128 bytes per clock and SM; see sse_prod32.cuh).
// Phase 1: a thread owns a 2 x 2 pair of the three T_j and B_i for NF frequencies. Phase 2: half of the threads' groups
// add X_mu G^H and half W^H U_mu, each thread two rows (columns) by half of the columns (rows) of the three sums for one
// (frequency, l) in GP: 5.5 FMAs per float loaded. W^, G^ and K^ of the next tile arrive by cp.async meanwhile, so a tile
// takes two barriers. FMAs are issued in pairs along the dimension in which the shared operand is stored in pairs, so
// that only the other operand has to be duplicated in registers.
// FinFET: 99.3 -> 92.8 ms for both types (0.52 of the FP32 pipe in useful work; ncu at the adjoint workload: FMA pipe 61%
// active, shared-memory wavefronts 58%, two warps per scheduler waiting on fixed latencies). Measured with the groups' sums
// rounded: NF = 2 with two CTAs per SM 91.5 ms, NF = 1 with three 92.7, with four (spills) 99.9.
#pragma once

#include "sse_prod32.cuh"

namespace sse {
namespace {

// The sums of phase 2 are flushed to the FP64 partial after at most this many FP32 additions into one of them: the chain of the
// previous kernel (32 frequencies of six terms per lane). Without the flush a chunk of 320 frequencies put the coupling
// gradient at the FinFET workload 7.7e-7 from the 64-bit value instead of 4.7e-7.
constexpr int kAdj32ChainTerms = 192;

template <int NP>
struct AdjShape {
    static constexpr int TN = NP / 2, T = TN * TN;  // column pairs, phase-1 threads per frequency set
    static constexpr int TP = T | 1;                // trace parts per (frequency, ij): an odd stride spreads the banks
    static constexpr int NF = NP == 2 ? 1 : 2;      // frequencies per thread in phase 1
    static constexpr int FG = 128 / T, F = FG * NF;
    static constexpr int RH = NP / 2;               // rows per thread in phase 2
    static constexpr int GP = 64 / NP;              // groups of NP threads per half of phase 2
    static constexpr int USED = FG * T > 2 * GP * NP ? FG * T : 2 * GP * NP;
    // tiles between two flushes: two additions per (frequency, l) into each sum
    static constexpr int CHAIN = 2 * ((F * NP + GP - 1) / GP);
    static constexpr int FLUSH = CHAIN < kAdj32ChainTerms ? kAdj32ChainTerms / CHAIN : 1;
    static constexpr int THREADS = (USED + 31) / 32 * 32;
    // floats of W^ or G^ per frequency: two sets in one warp start 2 NP banks apart, so their rows do not collide
    // (blocks of up to 4 x 4: no padding, the copies would be mostly padding)
    static constexpr int XS = NP * NP * 2 + (NP <= 4 ? 0 : ((2 * NP - NP * NP * 2) % 32 + 32) % 32);
    static constexpr int MS = 3 * NP * NP * 2;      // floats of X_mu or U_mu per frequency
    static constexpr int AB = 3 * NP * TN * 4;      // floats of dH in one of its two layouts
    static constexpr int off_A = 0;
    static constexpr int off_W = off_A + 2 * AB * 4;              // [2][F][XS] W^[m][l], then [2][F][XS] G^[l][n]
    static constexpr int off_M = off_W + 4 * F * XS * 4;          // [F][MS] X_mu[l][m pair], then [F][MS] U_mu[l][n pair]
    static constexpr int off_P = off_M + (F > GP ? F : GP) * 2 * MS * 4;  // (the groups' sums too); [F][9][TP] trace parts
    static constexpr int off_K = off_P + (F * 9 * TP * 8 + 15) / 16 * 16;  // [2][F][9]
    static constexpr int smem = off_K + 2 * F * 9 * 8;
    static constexpr int CTAS = smem <= (228 / 3 - 1) * 1024 ? 3 : 2;
    static_assert(smem <= (228 / CTAS - 1) * 1024, "CTAS CTAs per SM");
};

struct Adj32Cfg {
    int F, fchunk, nchunks, spc;  // frequencies per tile, tiles per chunk, chunks, bonds per CTA (grid z: the rest)
};

template <int NP>
Adj32Cfg adj32_cfg_t(size_t nA, int NB, size_t nfreq) {
    using S = AdjShape<NP>;
    Adj32Cfg c{};
    c.F = S::F;
    const size_t tiles = (nfreq + S::F - 1) / S::F;
    const size_t chunks = ((size_t)152 * S::CTAS * 12 + nA - 1) / (nA ? nA : 1);  // enough CTAs for ~12 waves
    size_t per = (tiles + chunks - 1) / chunks;
    per = per < 1 ? 1 : per;
    c.fchunk = (int)per;
    c.nchunks = (int)((tiles + per - 1) / per);
    c.spc = nA * c.nchunks < (size_t)152 * S::CTAS * 2 ? 1 : NB;  // few CTAs: one bond each
    return c;
}

inline Adj32Cfg make_adj32_cfg(const sse_dims& d, size_t nfreq) {
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    switch ((d.Norb + 1) / 2) {
        case 1: return adj32_cfg_t<2>(nA, d.NB, nfreq);
        case 2: return adj32_cfg_t<4>(nA, d.NB, nfreq);
        case 3: return adj32_cfg_t<6>(nA, d.NB, nfreq);
        case 4: return adj32_cfg_t<8>(nA, d.NB, nfreq);
        case 5: return adj32_cfg_t<10>(nA, d.NB, nfreq);
        case 6: return adj32_cfg_t<12>(nA, d.NB, nfreq);
        case 7: return adj32_cfg_t<14>(nA, d.NB, nfreq);
        default: return adj32_cfg_t<16>(nA, d.NB, nfreq);
    }
}

struct Adj32Args {
    sse_dims d;
    const int32_t* nbr;
    const double2* dH;
    const float2* What;   // [f][nA][nel]
    const float2* Ghat;   // [f][NA][nel]
    const float2* Khat;   // [f][nA][NB][9]
    float2* Hhat;         // [f][nA][NB][9]
    double2* gdh_part;    // [chunk][nA][NB][3][nel]
    int nfreq;
    double scale;
    unsigned* status;
};

// s + x, with the rounding error of the addition, exact in FP32 (Knuth's TwoSum), added to e. The up to 64 group sums of a
// flush keep the bits that FP64 additions would (an e of at most 64 errors of 2^-24 loses less than 2^-40), without the
// narrow FP64 pipe's additions and conversions. Adjoint at the FinFET workload, both types: 109.6 ms, against 117.5 with
// FP64 additions and 108.4 with rounded FP32 ones.
__device__ __forceinline__ void two_sum(float& s, float& e, float x) {
    const float t = s + x, b = t - s;
    e += (s - (t - b)) + (x - b);
    s = t;
}

template <int NP, int ODD>
__global__ void __launch_bounds__(AdjShape<NP>::THREADS, AdjShape<NP>::CTAS) spec_adj32_kernel(Adj32Cfg c, Adj32Args p) {
    using S = AdjShape<NP>;
    using Cp = TileCopy<NP, ODD>;
    constexpr int N = NP - ODD, nel = N * N, NF = S::NF, F = S::F, XS = S::XS, MS = S::MS, nt = S::THREADS, RH = S::RH;
    extern __shared__ __align__(16) unsigned char smem[];
    float* sA = reinterpret_cast<float*>(smem + S::off_A);  // [3 j][NP l][TN n] (re, re, im, im) of A_j[l][n]; then
                                                            // [3 i][NP l][TN m] of A_i[m][l]
    float* sW = reinterpret_cast<float*>(smem + S::off_W);
    float* sG = sW + 2 * F * XS;
    float* sX = reinterpret_cast<float*>(smem + S::off_M);
    float* sU = sX + F * MS;
    float2* sP = reinterpret_cast<float2*>(smem + S::off_P);
    float2* sK = reinterpret_cast<float2*>(smem + S::off_K);
    const sse_dims& d = p.d;
    const int tid = threadIdx.x, la = blockIdx.x, a = d.a_begin + la;
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const int ntiles = (p.nfreq + F - 1) / F;
    const int tile0 = blockIdx.y * c.fchunk, tile1 = min(ntiles, tile0 + c.fchunk);
    // phase 1: frequency set, pair of rows, pair of columns
    const int fs = tid / S::T, tt = tid - fs * S::T, mp = tt / S::TN, np = tt - mp * S::TN;
    const bool lane1 = fs < S::FG;
    // phase 2: group, its half of the work, pair and half of the block
    const int gr = tid / NP, t2 = tid - gr * NP, part = gr & 1, k0 = t2 / S::TN * RH, pp = t2 % S::TN;
    const bool lane2 = gr < 2 * S::GP;

    auto stage_A = [&](int s) {
        const double2* H = p.dH + ((size_t)a * d.NB + s) * 3 * nel;
        for (int i = tid; i < 3 * NP * NP; i += nt) {
            const int j = i / (NP * NP), e = i - j * (NP * NP), r = e / NP, q = e - r * NP;
            float2 v = make_float2(0.f, 0.f);  // A_j[r][q]
            if (r < N && q < N) {
                const double2 h = H[j * nel + r * N + q];
                v = make_float2((float)h.x, (float)h.y);
            }
            float* o = sA + ((j * NP + r) * S::TN + q / 2) * 4 + (q & 1);
            o[0] = v.x;
            o[2] = v.y;
            o = sA + S::AB + ((j * NP + q) * S::TN + r / 2) * 4 + (r & 1);
            o[0] = v.x;
            o[2] = v.y;
        }
    };
    auto issue = [&](int s, int tile, int buf) {
        const int b = p.nbr[(size_t)a * d.NB + s];
        const bool bok = b >= 0 && b < d.NA;
        for (int i = tid; i < F * Cp::ITEMS; i += nt) {
            const int f = i / Cp::ITEMS, e = i - f * Cp::ITEMS, g = tile * F + f;
            const bool ok = bok && g < p.nfreq;
            Cp::run(sW + (buf * F + f) * XS, ok ? p.What + ((size_t)g * nA + la) * nel : p.What, e, ok);
            Cp::run(sG + (buf * F + f) * XS, ok ? p.Ghat + ((size_t)g * d.NA + b) * nel : p.Ghat, e, ok);
        }
        for (int i = tid; i < F * 9; i += nt) {
            const int f = i / 9, e = i - f * 9, g = tile * F + f;
            const bool ok = bok && g < p.nfreq;
            tile_cp_async<8>(reinterpret_cast<float*>(sK + buf * F * 9 + i),
                             ok ? p.Khat + (((size_t)g * nA + la) * d.NB + s) * 9 + e : p.Khat, ok);
        }
        tile_cp_commit();
    };

    if (ODD)  // padding rows and columns of W^ and G^ stay zero (the copies never write them)
        for (int i = tid; i < 4 * F * XS; i += nt) sW[i] = 0.f;
    const int s0 = blockIdx.z * c.spc, s1 = min(d.NB, s0 + c.spc);
    stage_A(s0);
    if (ODD) __syncthreads();
    if (tile0 < tile1) issue(s0, tile0, 0);
    int buf = 0;
    for (int s = s0; s < s1; ++s) {
        if (tid == 0) {
            const int b = p.nbr[(size_t)a * d.NB + s];
            if (b < 0 || b >= d.NA) atomicOr(p.status, DEV_BAD_NEIGHBOUR);
        }
        // grad dH_mu[m][n]: part 0 holds pairs over m = 2 pp, 2 pp + 1 of columns n = k0 + k, part 1 pairs over n of rows m
        float2 ar[3][RH], ai[3][RH];
#pragma unroll
        for (int mu = 0; mu < 3; ++mu)
#pragma unroll
            for (int k = 0; k < RH; ++k) ar[mu][k] = ai[mu][k] = make_float2(0.f, 0.f);
        int chain = 0;
        bool first = true;
        for (int tile = tile0; tile < tile1; ++tile, buf ^= 1) {
            tile_cp_wait();
            __syncthreads();  // this tile has landed; the previous tile's phase 2 and sums are done
            if (tile + 1 < tile1) issue(s, tile + 1, buf ^ 1);
            else if (s + 1 < s1) issue(s + 1, tile0, buf ^ 1);
            const float* W = sW + buf * F * XS;
            const float* G = sG + buf * F * XS;
            if (lane1) {
                const float* P = sA + np * 4;
                const float* Q = sA + S::AB + mp * 4;
                float2 tr[NF][3][2], ti[NF][3][2];  // T_j[row of the pair], pairs over the columns
                float2 br[NF][3][2], bi[NF][3][2];  // B_i[column of the pair], pairs over the rows
#pragma unroll
                for (int f = 0; f < NF; ++f)
#pragma unroll
                    for (int j = 0; j < 3; ++j)
#pragma unroll
                        for (int r = 0; r < 2; ++r)
                            tr[f][j][r] = ti[f][j][r] = br[f][j][r] = bi[f][j][r] = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int l0 = 0; l0 < NP; l0 += 2) {
                    float4 w[NF][2];  // W[m][l0], W[m][l0 + 1]
#pragma unroll
                    for (int f = 0; f < NF; ++f)
#pragma unroll
                        for (int r = 0; r < 2; ++r)
                            w[f][r] = lds4(W + (fs + f * S::FG) * XS + ((2 * mp + r) * NP + l0) * 2);
#pragma unroll
                    for (int dl = 0; dl < 2; ++dl) {
                        if (ODD && l0 + dl >= N) continue;  // the padding column of an odd block
                        float4 g[NF];  // G[l][n] of the two columns
#pragma unroll
                        for (int f = 0; f < NF; ++f)
                            g[f] = lds4(G + (fs + f * S::FG) * XS + ((l0 + dl) * NP + 2 * np) * 2);
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            const float4 u = lds4(P + (j * NP + l0 + dl) * S::TN * 4);
                            const float4 v = lds4(Q + (j * NP + l0 + dl) * S::TN * 4);
                            const float2 ur = lo2(u), ui = hi2(u), nui = f2neg(u.z, u.w);
                            const float2 vr = lo2(v), vi = hi2(v), nvi = f2neg(v.z, v.w);
#pragma unroll
                            for (int f = 0; f < NF; ++f)
#pragma unroll
                                for (int r = 0; r < 2; ++r) {
                                    const float2 x = f2dup(dl ? w[f][r].z : w[f][r].x);
                                    const float2 y = f2dup(dl ? w[f][r].w : w[f][r].y);
                                    const float2 gx = f2dup(r ? g[f].z : g[f].x), gy = f2dup(r ? g[f].w : g[f].y);
                                    tr[f][j][r] = fma2(x, ur, tr[f][j][r]);
                                    ti[f][j][r] = fma2(x, ui, ti[f][j][r]);
                                    br[f][j][r] = fma2(vr, gx, br[f][j][r]);
                                    bi[f][j][r] = fma2(vr, gy, bi[f][j][r]);
                                    tr[f][j][r] = fma2(y, nui, tr[f][j][r]);
                                    ti[f][j][r] = fma2(y, ur, ti[f][j][r]);
                                    br[f][j][r] = fma2(nvi, gy, br[f][j][r]);
                                    bi[f][j][r] = fma2(vi, gx, bi[f][j][r]);
                                }
                        }
                    }
                }
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const int fi = fs + f * S::FG;
                    // this thread's part of sum_mn T_j[m][n] conj(B_i[m][n])
                    float2* o = sP + (size_t)fi * 9 * S::TP + tt;
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        float2 qr[2], qi[2];  // B_i[row], pairs over the columns
                        qr[0] = make_float2(br[f][i][0].x, br[f][i][1].x);
                        qr[1] = make_float2(br[f][i][0].y, br[f][i][1].y);
                        qi[0] = make_float2(bi[f][i][0].x, bi[f][i][1].x);
                        qi[1] = make_float2(bi[f][i][0].y, bi[f][i][1].y);
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            float2 h = make_float2(0.f, 0.f), g = h, k = h;
#pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                h = fma2(tr[f][j][r], qr[r], h);
                                h = fma2(ti[f][j][r], qi[r], h);
                                g = fma2(ti[f][j][r], qr[r], g);
                                k = fma2(tr[f][j][r], qi[r], k);
                            }
                            o[(i * 3 + j) * S::TP] = make_float2(h.x + h.y, (g.x + g.y) - (k.x + k.y));
                        }
                    }
                    // X_mu = sum_j -i conj(K_mu,j) T_j, U_mu = sum_i i K_i,mu B_i
                    const float2* K = sK + (buf * F + fi) * 9;
                    float* Xo = sX + (size_t)fi * MS + ((2 * np) * S::TN + mp) * 4;
                    float* Uo = sU + (size_t)fi * MS + ((2 * mp) * S::TN + np) * 4;
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        float2 xr[2], xi[2], ur[2], ui[2];
#pragma unroll
                        for (int r = 0; r < 2; ++r) xr[r] = xi[r] = ur[r] = ui[r] = make_float2(0.f, 0.f);
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            const float2 k1 = K[mu * 3 + j], k2 = K[j * 3 + mu];
                            const float2 ky = f2dup(-k1.y), kx = f2dup(k1.x), nx = f2dup(-k1.x);
                            const float2 qy = f2dup(-k2.y), qx = f2dup(k2.x), mx = f2dup(-k2.x);
#pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                xr[r] = fma2(ky, tr[f][j][r], xr[r]);
                                xi[r] = fma2(ky, ti[f][j][r], xi[r]);
                                xr[r] = fma2(kx, ti[f][j][r], xr[r]);
                                xi[r] = fma2(nx, tr[f][j][r], xi[r]);
                                ur[r] = fma2(qy, br[f][j][r], ur[r]);
                                ui[r] = fma2(qy, bi[f][j][r], ui[r]);
                                ur[r] = fma2(mx, bi[f][j][r], ur[r]);
                                ui[r] = fma2(qx, br[f][j][r], ui[r]);
                            }
                        }
                        float4* xo = reinterpret_cast<float4*>(Xo + mu * NP * S::TN * 4);
                        xo[0] = make_float4(xr[0].x, xr[1].x, xi[0].x, xi[1].x);
                        xo[S::TN] = make_float4(xr[0].y, xr[1].y, xi[0].y, xi[1].y);
                        float4* uo = reinterpret_cast<float4*>(Uo + mu * NP * S::TN * 4);
                        uo[0] = make_float4(ur[0].x, ur[1].x, ui[0].x, ui[1].x);
                        uo[S::TN] = make_float4(ur[0].y, ur[1].y, ui[0].y, ui[1].y);
                    }
                }
            }
            __syncthreads();  // X_mu, U_mu and the trace parts are complete
            for (int g = tid; g < F * 9; g += nt) {  // fixed-order sums over the tile's threads
                const int rf = g / 9, ij = g - rf * 9, ff = tile * F + rf;
                if (ff >= p.nfreq) continue;
                const float2* v = sP + (size_t)g * S::TP;
                float2 sum = make_float2(0.f, 0.f), odd = sum;
#pragma unroll
                for (int u = 0; u < S::T; u += 2) {
                    sum = cadd(sum, v[u]);
                    if (u + 1 < S::T) odd = cadd(odd, v[u + 1]);
                }
                p.Hhat[(((size_t)ff * nA + la) * d.NB + s) * 9 + ij] = cadd(sum, odd);
            }
            if (lane2) {
                // part 0: X_mu[m][l] conj(G[n][l]); part 1: conj(W[l][m]) U_mu[l][n]: pairs times conjugated scalars
                const float* pairs = sX + part * F * MS + pp * 4;
                const float* scal = part == 0 ? G + k0 * NP * 2 : W + k0 * 2;
                const int sl = part == 0 ? 2 : NP * 2, sk = part == 0 ? NP * 2 : 2;
#pragma unroll 1
                for (int u = gr >> 1; u < F * N; u += S::GP) {
                    const int f = u / N, l = u - f * N;
                    float2 z[RH];
#pragma unroll
                    for (int k = 0; k < RH; ++k) z[k] = ld2(scal + f * XS + l * sl + k * sk);
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        const float4 v = lds4(pairs + f * MS + (mu * NP + l) * S::TN * 4);
                        const float2 vr = lo2(v), vi = hi2(v), nvr = f2neg(v.x, v.y);
#pragma unroll
                        for (int k = 0; k < RH; ++k) {
                            const float2 zr = f2dup(z[k].x), zi = f2dup(z[k].y);
                            ar[mu][k] = fma2(zr, vr, ar[mu][k]);
                            ai[mu][k] = fma2(zr, vi, ai[mu][k]);
                            ar[mu][k] = fma2(zi, vi, ar[mu][k]);
                            ai[mu][k] = fma2(zi, nvr, ai[mu][k]);
                        }
                    }
                }
            }
            if (++chain < S::FLUSH && tile + 1 < tile1) continue;
            // flush: sum the groups (fixed order) and add to this chunk's FP64 partial
            chain = 0;
            __syncthreads();  // phase 2 is done with X_mu and U_mu
            float2* sAcc = reinterpret_cast<float2*>(sX);  // [2 GP][3][nel]
            if (lane2)
#pragma unroll
                for (int mu = 0; mu < 3; ++mu)
#pragma unroll
                    for (int k = 0; k < RH; ++k) {
                        float2* o = sAcc + (gr * 3 + mu) * nel;
                        const int p0 = 2 * pp, kk = k0 + k;
                        const int step = part == 0 ? N : 1;
                        o += part == 0 ? p0 * N + kk : kk * N + p0;
                        if (kk < N) o[0] = make_float2(ar[mu][k].x, ai[mu][k].x);
                        if (kk < N && p0 + 1 < N) o[step] = make_float2(ar[mu][k].y, ai[mu][k].y);
                        ar[mu][k] = ai[mu][k] = make_float2(0.f, 0.f);
                    }
            __syncthreads();
            const double inv = p.scale / (double)p.nfreq;
            double2* part_out = p.gdh_part + (((size_t)blockIdx.y * nA + la) * d.NB + s) * 3 * nel;
            for (int i = tid; i < 3 * nel; i += nt) {  // entry i belongs to one thread
                float2 sum = make_float2(0.f, 0.f), low = sum;
#pragma unroll
                for (int g = 0; g < 2 * S::GP; ++g) {
                    const float2 x = sAcc[g * 3 * nel + i];
                    two_sum(sum.x, low.x, x.x);
                    two_sum(sum.y, low.y, x.y);
                }
                double2 v = make_double2((double)sum.x + (double)low.x, (double)sum.y + (double)low.y);
                if (!isfinite(sum.x) || !isfinite(sum.y)) {  // the sum or one of its terms leaves the FP32 range
                    v = make_double2(0.0, 0.0);
                    for (int g = 0; g < 2 * S::GP; ++g) {
                        const float2 x = sAcc[g * 3 * nel + i];
                        v = make_double2(v.x + (double)x.x, v.y + (double)x.y);
                    }
                }
                v = make_double2(v.x * inv, v.y * inv);
                if (!first) {
                    const double2 o = part_out[i];
                    v = make_double2(v.x + o.x, v.y + o.y);
                }
                part_out[i] = v;
            }
            first = false;
            // the next tile writes X_mu and U_mu after its first barrier
        }
        if (s + 1 < s1) stage_A(s + 1);  // phase 1 of the last tile has passed for every thread
    }
    tile_cp_wait();
}

template <int NP, int ODD>
cudaError_t launch_adj32_t(const Adj32Args& p, cudaStream_t st) {
    const size_t nA = (size_t)(p.d.a_end - p.d.a_begin);
    const Adj32Cfg c = adj32_cfg_t<NP>(nA, p.d.NB, (size_t)p.nfreq);
    auto kern = spec_adj32_kernel<NP, ODD>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, AdjShape<NP>::smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)nA, (unsigned)c.nchunks, (unsigned)((p.d.NB + c.spc - 1) / c.spc));
    SSE_TIMED("spec_adj_kernel", st, kern<<<grid, AdjShape<NP>::THREADS, AdjShape<NP>::smem, st>>>(c, p));
    return cudaGetLastError();
}

inline cudaError_t launch_adj32(const Adj32Args& p, cudaStream_t st) {
    switch (p.d.Norb) {
#define SSE_ADJ32(n) \
    case n: return launch_adj32_t<(n + 1) / 2 * 2, n % 2>(p, st);
        SSE_ADJ32(1) SSE_ADJ32(2) SSE_ADJ32(3) SSE_ADJ32(4) SSE_ADJ32(5) SSE_ADJ32(6) SSE_ADJ32(7) SSE_ADJ32(8)
        SSE_ADJ32(9) SSE_ADJ32(10) SSE_ADJ32(11) SSE_ADJ32(12) SSE_ADJ32(13) SSE_ADJ32(14) SSE_ADJ32(15) SSE_ADJ32(16)
#undef SSE_ADJ32
        default: return cudaErrorNotSupported;
    }
}

}  // namespace
}  // namespace sse
