// Pi of Eq. (4) through the transforms: the per-frequency half products and traces in FP64 (spec_pi_kernel) and
// FP32 (spec_pi32_kernel), the store of the inverse transform, the 3x3 symmetrisation and the driver.
#include "sse_prod32.cuh"
#include "sse_tri.cuh"

namespace sse {
namespace {

// ---------------------------------------------------------------------------
struct PiCfg {
    int nel, F, threads, fchunk;
    int off_A, off_X, off_Y, off_P, off_R, off_D, off_self, smem;
};

PiCfg make_pi_cfg(const sse_dims& d, size_t nfreq) {
    PiCfg c{};
    c.nel = d.Norb * d.Norb;
    const int pl = c.nel * 8;
    auto a16 = [](int x) { return (x + 15) & ~15; };
    c.F = pick_frequencies(c.nel, [&](int F) {
        return (long)d.NB * 3 * 4 * pl + F * 3 * pl * 2 + F * 6 * pl * 2 + F * 9 * d.Norb * 16 + F * 9 * 16 + 96;
    });
    c.F = spread_frequencies(c.F, c.nel, 2 * (size_t)(d.a_end - d.a_begin), nfreq);
    c.threads = ((c.F * c.nel + 31) / 32) * 32;
    c.off_A = 0;                                     // [NB][3][4 planes: re, im, re+im, re-im]
    c.off_X = a16(c.off_A + d.NB * 3 * 4 * pl);      // [F][3 planes]
    c.off_Y = a16(c.off_X + c.F * 3 * pl);           // [F][3 planes]
    c.off_P = a16(c.off_Y + c.F * 3 * pl);           // [F][3 i][2 planes]
    c.off_R = a16(c.off_P + c.F * 6 * pl);           // [F][3 j][2 planes]
    c.off_D = a16(c.off_R + c.F * 6 * pl);           // [F][9][Norb] complex: diagonal terms
    c.off_self = a16(c.off_D + c.F * 9 * d.Norb * 16);  // [F][9] complex: diagonal-block sums
    c.smem = a16(c.off_self + c.F * 9 * 16);
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    size_t want = (size_t)152 * 2 * 8;
    size_t chunks = (want + 2 * nA - 1) / (nA ? 2 * nA : 1);
    if (chunks < 1) chunks = 1;
    size_t fc = (nfreq + chunks - 1) / chunks;
    fc = ((fc + c.F - 1) / c.F) * c.F;
    c.fchunk = (int)(fc < 1 ? 1 : fc);
    return c;
}

__global__ void __launch_bounds__(kProdMaxThreads, 2)
spec_pi_kernel(PiCfg c, sse_dims d, FreqMap fm, const int32_t* __restrict__ nbr, const double2* __restrict__ dH,
               const double2* __restrict__ Gl_hat, const double2* __restrict__ Gg_hat, double2* __restrict__ Cl_hat,
               double2* __restrict__ Cg_hat, unsigned* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int Norb = d.Norb, nel = c.nel;
    const int la = blockIdx.x;
    const int a = d.a_begin + la;
    const int t = blockIdx.z;
    const double2* X_hat = t == 0 ? Gl_hat : Gg_hat;  // G^t of atom a
    const double2* Y_hat = t == 0 ? Gg_hat : Gl_hat;  // G^t' of the neighbour
    double2* C_hat = t == 0 ? Cl_hat : Cg_hat;
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const size_t i_begin = (size_t)blockIdx.y * c.fchunk;  // frequency indices of the map
    const size_t i_end = min(fm.count, i_begin + c.fchunk);
    double* sA = reinterpret_cast<double*>(smem + c.off_A);
    double* sX = reinterpret_cast<double*>(smem + c.off_X);
    double* sY = reinterpret_cast<double*>(smem + c.off_Y);
    double* sP = reinterpret_cast<double*>(smem + c.off_P);
    double* sR = reinterpret_cast<double*>(smem + c.off_R);
    double2* sD = reinterpret_cast<double2*>(smem + c.off_D);
    double2* sSelf = reinterpret_cast<double2*>(smem + c.off_self);
    const int tid = threadIdx.x;
    const int fl = tid / nel, e = tid - fl * nel;
    const int m = e / Norb, n = e - m * Norb;
    const bool lane = fl < c.F;
    const int slots = d.NB + 1;
    const int ndiag = c.F * 9 * Norb;

    for (int i = tid; i < d.NB * 3 * nel; i += blockDim.x) {
        const int si = i / nel, ee = i - si * nel;
        const double2 v = dH[((size_t)a * d.NB) * 3 * nel + i];
        double* P = sA + (size_t)si * 4 * nel;
        P[ee] = v.x;
        P[nel + ee] = v.y;
        P[2 * nel + ee] = v.x + v.y;
        P[3 * nel + ee] = v.x - v.y;
    }
    if (tid == 0 && t == 0)
        for (int s = 0; s < d.NB; ++s) {
            const int b = nbr[(size_t)a * d.NB + s];
            if (b < 0 || b >= d.NA) atomicOr(status, DEV_BAD_NEIGHBOUR);
        }
    __syncthreads();

    for (size_t i0 = i_begin; i0 < i_end; i0 += c.F) {
        const bool act = lane && i0 + fl < i_end;
        const size_t f = act ? freq_of(fm, i0 + fl) : 0;
        const size_t fneg = act ? freq_neg(fm, f) : 0;
        if (lane) {
            double2 x = make_double2(0.0, 0.0);
            if (act) x = X_hat[(f * d.NA + a) * nel + e];
            put3(sX + (size_t)fl * 3 * nel, nel, e, x);
        }
        // diagonal-block sums: entry g = (frequency, ij) belongs to thread g mod blockDim for the whole batch
        for (int g = tid; g < c.F * 9; g += blockDim.x) sSelf[g] = make_double2(0.0, 0.0);
        for (int s = 0; s < d.NB; ++s) {
            const int b = nbr[(size_t)a * d.NB + s];
            const bool bok = b >= 0 && b < d.NA;
            if (lane) {
                double2 y = make_double2(0.0, 0.0);
                if (act && bok) y = Y_hat[(fneg * d.NA + b) * nel + e];
                put3(sY + (size_t)fl * 3 * nel, nel, e, y);
            }
            __syncthreads();
            // half products P_i = dH_i^H X, R_j = dH_j Y (Gauss 3-multiply MACs)
            if (lane) {
                const double* A = sA + (size_t)s * 12 * nel;
                const double* Xp = sX + (size_t)fl * 3 * nel;
                const double* Yp = sY + (size_t)fl * 3 * nel;
#pragma unroll 1
                for (int i = 0; i < 3; ++i) {
                    const double* Ai = A + (size_t)i * 4 * nel;
                    double t1 = 0.0, u2 = 0.0, t3 = 0.0, r1 = 0.0, r2 = 0.0, r3 = 0.0;
                    for (int l = 0; l < Norb; ++l) {
                        const int lm = l * Norb + m, ml = m * Norb + l, ln = l * Norb + n;
                        t1 = fma(Ai[lm], Xp[ln], t1);                  // conj(A_i[l][m]) X[l][n]
                        u2 = fma(Ai[nel + lm], Xp[nel + ln], u2);
                        t3 = fma(Ai[3 * nel + lm], Xp[2 * nel + ln], t3);
                        r1 = fma(Ai[ml], Yp[ln], r1);                  // A_i[m][l] Y[l][n]
                        r2 = fma(Ai[nel + ml], Yp[nel + ln], r2);
                        r3 = fma(Ai[2 * nel + ml], Yp[2 * nel + ln], r3);
                    }
                    double* P = sP + ((size_t)fl * 3 + i) * 2 * nel;
                    P[e] = t1 + u2;
                    P[nel + e] = t3 - t1 + u2;
                    double* R = sR + ((size_t)fl * 3 + i) * 2 * nel;
                    R[e] = r1 - r2;
                    R[nel + e] = r3 - r1 - r2;
                }
            }
            __syncthreads();
            // diagonal terms D_ij[m] = sum_n P_i[m][n] R_j[n][m]
            for (int g = tid; g < ndiag; g += blockDim.x) {
                const int fi = g / (9 * Norb), rem = g - fi * 9 * Norb;
                const int ij = rem / Norb, mm = rem - ij * Norb;
                const int i = ij / 3, j = ij - 3 * i;
                const double* P = sP + ((size_t)fi * 3 + i) * 2 * nel;
                const double* R = sR + ((size_t)fi * 3 + j) * 2 * nel;
                double re = 0.0, im = 0.0;
                for (int nn = 0; nn < Norb; ++nn) {
                    const double pr = P[mm * Norb + nn], pi = P[nel + mm * Norb + nn];
                    const double rr = R[nn * Norb + mm], ri = R[nel + nn * Norb + mm];
                    re = fma(pr, rr, re);
                    re = fma(-pi, ri, re);
                    im = fma(pr, ri, im);
                    im = fma(pi, rr, im);
                }
                sD[g] = make_double2(re, im);
            }
            __syncthreads();
            for (int g = tid; g < c.F * 9; g += blockDim.x) {  // fixed-order sums over the rows m
                const int rf = g / 9, ij = g - rf * 9;
                const double2* v = sD + (size_t)g * Norb;
                double2 sum = v[0];
                for (int mm = 1; mm < Norb; ++mm) sum = cadd(sum, v[mm]);
                const double2 self = cadd(sSelf[g], sum);
                sSelf[g] = self;
                if (i0 + rf < i_end) {
                    const size_t ff = freq_of(fm, i0 + rf);
                    C_hat[((ff * nA + la) * slots + s) * 9 + ij] = sum;
                    if (s == d.NB - 1) C_hat[((ff * nA + la) * slots + d.NB) * 9 + ij] = self;
                }
            }
            // the next bond rewrites sY before its first barrier; sP, sR and sD only after it
        }
        __syncthreads();  // sX of the next frequency batch
    }
}

// ---------------------------------------------------------------------------
// FP32 phonon self-energy (mode FP32_FFT). A thread owns the 2 x 2 pairs (m, n) of P_i[m][n] (P_i = dH_i^H X^) and of
// R_j[n][m] (R_j = dH_j Y^) for the three i and j and for NF frequencies, so its part of every trace
// tr(P_i R_j) = sum_mn P_i[m][n] R_j[n][m] is formed from its own registers; the parts are summed over the tile's
// threads in a fixed order.
//
// What bounds it: the FP32 pipe and the shared-memory return path (128 bytes per clock and SM; see sse_prod32.cuh). The
// coupling blocks are the same for every frequency, so NF frequencies per thread raise the FMAs per float loaded from 3
// (one frequency, with R_j exchanged through shared memory) to 4.8 (NF = 2) and 6 (NF = 3). FMAs are issued in
// pairs: over m for P, over n for R, with X^ and Y^ duplicated. FinFET workload: 55.1 -> 38.7 ms for Pi^< and Pi^>
// (0.58 of the FP32 pipe); NF = 2 with three CTAs per SM (168 registers) is taken since it measured 38.7 ms against
// 42.0 for NF = 2 with two CTAs and 40.7 for NF = 3 with two: warps to cover the latencies count for more than loads.
// ---------------------------------------------------------------------------
template <int NP>
struct PiShape {
    static constexpr int TN = NP / 2, T = TN * TN;  // pairs per block edge, threads per frequency set
    static constexpr int TP = T | 1;                // trace parts per (frequency, ij): an odd stride spreads the banks
    static constexpr int NF = 2;                    // frequencies per thread (see above)
    static constexpr int FG = 128 / T;              // frequency sets per CTA
    static constexpr int F = FG * NF;
    static constexpr int THREADS = (FG * T + 31) / 32 * 32;
    static constexpr int CTAS = 3;
    // floats of X^ or Y^ per frequency: two sets in one warp start 2 NP banks apart, so their rows do not collide
    // (blocks of up to 4 x 4: no padding, the copies would be mostly padding)
    static constexpr int XS = NP * NP * 2 + (NP <= 4 ? 0 : ((2 * NP - NP * NP * 2) % 32 + 32) % 32);
    static constexpr int AB = 3 * NP * TN * 4;      // floats of one bond's dH in one of its two layouts
};

struct PiTileCfg {
    int fchunk, nchunks, nres;
    int off_X, off_Y, off_P, off_self, off_F, smem;
};

template <int NP>
PiTileCfg make_pi_tile_cfg(const sse_dims& d, size_t nfreq) {
    using S = PiShape<NP>;
    auto a16 = [](int x) { return (x + 15) & ~15; };
    PiTileCfg c{};
    auto place = [&](int nres) {
        c.nres = nres;
        c.off_X = nres * 2 * S::AB * 4;
        c.off_Y = c.off_X + S::F * S::XS * 4;
        c.off_P = c.off_Y + S::F * S::XS * 4;
        c.off_self = a16(c.off_P + S::F * 9 * S::TP * 8);
        c.off_F = c.off_self + S::F * 9 * 8;
        c.smem = a16(c.off_F + 4 * S::F * 4);
        return c.smem;
    };
    // every bond's dH stays resident where it fits beside the buffers of CTAS CTAs
    if (place(d.NB) > (227 / S::CTAS - 1) * 1024) place(1);
    // tiles per CTA: enough CTAs for ~8 waves, at most 8 tiles (dH is staged per CTA)
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const size_t tiles = (nfreq + S::F - 1) / S::F;
    size_t per = tiles * 2 * nA / ((size_t)152 * S::CTAS * 8);
    per = per < 1 ? 1 : per > 8 ? 8 : per;
    c.fchunk = (int)per;
    c.nchunks = (int)((tiles + per - 1) / per);
    return c;
}

template <int NP, int ODD>
__global__ void __launch_bounds__(PiShape<NP>::THREADS, PiShape<NP>::CTAS)
spec_pi32_kernel(PiTileCfg c, sse_dims d, FreqMap fm, const int32_t* __restrict__ nbr, const double2* __restrict__ dH,
                 const float2* __restrict__ Gl_hat, const float2* __restrict__ Gg_hat, float2* __restrict__ Cl_hat,
                 float2* __restrict__ Cg_hat, unsigned* __restrict__ status) {
    using S = PiShape<NP>;
    using Cp = TileCopy<NP, ODD>;
    constexpr int N = NP - ODD, nel = N * N, NF = S::NF, F = S::F, XS = S::XS, nt = S::THREADS;
    extern __shared__ __align__(16) unsigned char smem[];
    // [res][P: [3 i][NP l][TN m] (re, re, im, im) of dH_i[l][m]; R: [3 j][NP l][TN n] of dH_j[n][l]]
    float* sA = reinterpret_cast<float*>(smem);
    float* sX = reinterpret_cast<float*>(smem + c.off_X);  // [F][NP l][NP n]
    float* sY = reinterpret_cast<float*>(smem + c.off_Y);  // [F][NP l][NP m]
    float2* sP = reinterpret_cast<float2*>(smem + c.off_P);      // [F][9][TP] trace parts
    float2* sSelf = reinterpret_cast<float2*>(smem + c.off_self);  // [F][9] diagonal-block sums
    int* sF = reinterpret_cast<int*>(smem + c.off_F);            // [2 tiles][f, -f][F], -1: none
    const int tid = threadIdx.x, la = blockIdx.x, a = d.a_begin + la, t = blockIdx.z, slots = d.NB + 1;
    const float2* X_hat = t == 0 ? Gl_hat : Gg_hat;  // G^t of atom a
    const float2* Y_hat = t == 0 ? Gg_hat : Gl_hat;  // G^t' of the neighbour
    float2* C_hat = t == 0 ? Cl_hat : Cg_hat;
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const int ntiles = (int)((fm.count + F - 1) / F);
    const int tile0 = blockIdx.y * c.fchunk, tile1 = min(ntiles, tile0 + c.fchunk);
    const bool resident = c.nres >= d.NB;
    const int fs = tid / S::T, tt = tid - fs * S::T;
    const int mp = tt / S::TN, np = tt - mp * S::TN;
    const bool lane = fs < S::FG;

    auto stage_A = [&](int s, int slot) {
        const double2* H = dH + ((size_t)a * d.NB + s) * 3 * nel;
        float* P = sA + (size_t)slot * 2 * S::AB;
        float* R = P + S::AB;
        for (int i = tid; i < 3 * NP * NP; i += nt) {
            const int j = i / (NP * NP), e = i - j * (NP * NP), r = e / NP, q = e - r * NP;
            float2 v = make_float2(0.f, 0.f);  // dH_j[r][q]
            if (r < N && q < N) {
                const double2 h = H[j * nel + r * N + q];
                v = make_float2((float)h.x, (float)h.y);
            }
            float* o = P + ((j * NP + r) * S::TN + q / 2) * 4 + (q & 1);
            o[0] = v.x;
            o[2] = v.y;
            o = R + ((j * NP + q) * S::TN + r / 2) * 4 + (r & 1);
            o[0] = v.x;
            o[2] = v.y;
        }
    };
    auto freq_table = [&](int tile) {
        int* f = sF + (tile & 1) * 2 * F;
        for (int i = tid; i < F; i += nt) {
            const size_t ix = (size_t)tile * F + i;
            const bool ok = ix < fm.count;
            const size_t g = ok ? freq_of(fm, ix) : 0;
            f[i] = ok ? (int)g : -1;
            f[F + i] = ok ? (int)freq_neg(fm, g) : -1;
        }
    };
    auto issue_one = [&](float* dst, const int* fq, const float2* src, int atom, bool aok) {
        for (int i = tid; i < F * Cp::ITEMS; i += nt) {
            const int f = i / Cp::ITEMS, e = i - f * Cp::ITEMS;
            const int g = fq[f];
            const bool ok = g >= 0 && aok;
            Cp::run(dst + f * XS, ok ? src + ((size_t)g * d.NA + atom) * nel : src, e, ok);
        }
    };
    auto issue_Y = [&](int tile, int s) {
        const int b = nbr[(size_t)a * d.NB + s];
        issue_one(sY, sF + (tile & 1) * 2 * F + F, Y_hat, b, b >= 0 && b < d.NA);
        tile_cp_commit();
    };

    if (ODD)  // padding rows and columns stay zero (the copies never write them)
        for (int i = tid; i < F * XS; i += nt) sX[i] = sY[i] = 0.f;
    if (tid == 0 && t == 0)
        for (int s = 0; s < d.NB; ++s) {
            const int b = nbr[(size_t)a * d.NB + s];
            if (b < 0 || b >= d.NA) atomicOr(status, DEV_BAD_NEIGHBOUR);
        }
    freq_table(tile0);
    if (resident)
        for (int s = 0; s < d.NB; ++s) stage_A(s, s);
    __syncthreads();
    if (tile0 < tile1) {
        issue_one(sX, sF + (tile0 & 1) * 2 * F, X_hat, a, true);
        issue_Y(tile0, 0);
    }

    for (int tile = tile0; tile < tile1; ++tile) {
        for (int s = 0; s < d.NB; ++s) {
            tile_cp_wait();
            __syncthreads();  // X and Y have landed; the previous bond's sums over sP are done
            if (s == 0 && tile + 1 < tile1) freq_table(tile + 1);  // read after the next barrier
            if (!resident) {
                stage_A(s, 0);
                __syncthreads();
            }
            if (lane) {
                const float* P = sA + (size_t)(resident ? s : 0) * 2 * S::AB + mp * 4;
                const float* R = sA + (size_t)(resident ? s : 0) * 2 * S::AB + S::AB + np * 4;
                const float* X = sX + fs * XS + np * 4;
                const float* Y = sY + fs * XS + mp * 4;
                float2 pr[NF][3][2], pi[NF][3][2];  // (P[m0][n], P[m0 + 1][n])
                float2 rr[NF][3][2], ri[NF][3][2];  // (R[n0][m], R[n0 + 1][m])
#pragma unroll
                for (int f = 0; f < NF; ++f)
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int n = 0; n < 2; ++n)
                            pr[f][i][n] = pi[f][i][n] = rr[f][i][n] = ri[f][i][n] = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int l = 0; l < N; ++l) {
                    float4 x[NF], y[NF];
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        x[f] = lds4(X + f * S::FG * XS + l * NP * 2);
                        y[f] = lds4(Y + f * S::FG * XS + l * NP * 2);
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const float4 u = lds4(P + (i * NP + l) * S::TN * 4), v = lds4(R + (i * NP + l) * S::TN * 4);
                        const float2 ar = lo2(u), ai = hi2(u), na = f2neg(u.z, u.w);
                        const float2 br = lo2(v), bi = hi2(v), nb = f2neg(v.z, v.w);
#pragma unroll
                        for (int f = 0; f < NF; ++f)
#pragma unroll
                            for (int n = 0; n < 2; ++n) {
                                const float2 xr = f2dup(n ? x[f].z : x[f].x), xi = f2dup(n ? x[f].w : x[f].y);
                                const float2 yr = f2dup(n ? y[f].z : y[f].x), yi = f2dup(n ? y[f].w : y[f].y);
                                pr[f][i][n] = fma2(ar, xr, pr[f][i][n]);  // conj(dH_i[l][m]) X[l][n]
                                pi[f][i][n] = fma2(ar, xi, pi[f][i][n]);
                                rr[f][i][n] = fma2(br, yr, rr[f][i][n]);  // dH_j[n][l] Y[l][m]
                                ri[f][i][n] = fma2(br, yi, ri[f][i][n]);
                                pr[f][i][n] = fma2(ai, xi, pr[f][i][n]);
                                pi[f][i][n] = fma2(na, xr, pi[f][i][n]);
                                rr[f][i][n] = fma2(nb, yi, rr[f][i][n]);
                                ri[f][i][n] = fma2(bi, yr, ri[f][i][n]);
                            }
                    }
                }
                // this thread's part of tr(P_i R_j)
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    float2* o = sP + (size_t)(fs + f * S::FG) * 9 * S::TP + tt;
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        float2 qr[2], qi[2];  // (R[n][m0], R[n][m0 + 1])
                        qr[0] = make_float2(rr[f][j][0].x, rr[f][j][1].x);
                        qr[1] = make_float2(rr[f][j][0].y, rr[f][j][1].y);
                        qi[0] = make_float2(ri[f][j][0].x, ri[f][j][1].x);
                        qi[1] = make_float2(ri[f][j][0].y, ri[f][j][1].y);
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            float2 h = make_float2(0.f, 0.f), g = h, k = h;
#pragma unroll
                            for (int n = 0; n < 2; ++n) {
                                h = fma2(pr[f][i][n], qr[n], h);
                                g = fma2(pi[f][i][n], qi[n], g);
                                k = fma2(pr[f][i][n], qi[n], k);
                                k = fma2(pi[f][i][n], qr[n], k);
                            }
                            o[(i * 3 + j) * S::TP] = make_float2((h.x + h.y) - (g.x + g.y), k.x + k.y);
                        }
                    }
                }
            }
            __syncthreads();  // the trace parts are complete; X and Y are free
            if (s + 1 < d.NB) {
                issue_Y(tile, s + 1);
            } else if (tile + 1 < tile1) {
                issue_one(sX, sF + ((tile + 1) & 1) * 2 * F, X_hat, a, true);
                issue_Y(tile + 1, 0);
            }
            for (int g = tid; g < F * 9; g += nt) {  // fixed-order sums over the tile's threads
                const int rf = g / 9, ij = g - rf * 9;
                const int ff = sF[(tile & 1) * 2 * F + rf];
                if (ff < 0) continue;
                const float2* v = sP + (size_t)g * S::TP;
                float2 sum = make_float2(0.f, 0.f), odd = sum;
#pragma unroll
                for (int u = 0; u < S::T; u += 2) {
                    sum = cadd(sum, v[u]);
                    if (u + 1 < S::T) odd = cadd(odd, v[u + 1]);
                }
                sum = cadd(sum, odd);
                const float2 self = s == 0 ? sum : cadd(sSelf[g], sum);
                sSelf[g] = self;  // entry g belongs to one thread for the whole tile
                C_hat[(((size_t)ff * nA + la) * slots + s) * 9 + ij] = sum;
                if (s == d.NB - 1) C_hat[(((size_t)ff * nA + la) * slots + d.NB) * 9 + ij] = self;
            }
        }
    }
}

template <int NP, int ODD>
cudaError_t launch_pi32_t(const sse_dims& d, const FreqMap& fm, const int32_t* nbr, const double2* dH,
                          const float2* const* Gh, float2* const* Ch, unsigned* status, cudaStream_t st) {
    const PiTileCfg c = make_pi_tile_cfg<NP>(d, fm.count);
    auto kern = spec_pi32_kernel<NP, ODD>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, c.smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(d.a_end - d.a_begin), (unsigned)c.nchunks, 2);
    SSE_TIMED("spec_pi_kernel", st,
              kern<<<grid, PiShape<NP>::THREADS, c.smem, st>>>(c, d, fm, nbr, dH, Gh[0], Gh[1], Ch[0], Ch[1], status));
    return cudaGetLastError();
}

cudaError_t launch_pi32(const sse_dims& d, const FreqMap& fm, const int32_t* nbr, const double2* dH,
                        const float2* const* Gh, float2* const* Ch, unsigned* status, cudaStream_t st) {
    switch (d.Norb) {
#define SSE_PI32(n) \
    case n: return launch_pi32_t<(n + 1) / 2 * 2, n % 2>(d, fm, nbr, dH, Gh, Ch, status, st);
        SSE_PI32(1) SSE_PI32(2) SSE_PI32(3) SSE_PI32(4) SSE_PI32(5) SSE_PI32(6) SSE_PI32(7) SSE_PI32(8)
        SSE_PI32(9) SSE_PI32(10) SSE_PI32(11) SSE_PI32(12) SSE_PI32(13) SSE_PI32(14) SSE_PI32(15) SSE_PI32(16)
#undef SSE_PI32
        default: return cudaErrorNotSupported;
    }
}

// Pi^t[q][w][a][slot][ij] = -i*scale * conj(v) * inv for rows l = w+1 in [1, Nw]
template <class C>
struct StorePiT {
    double2* P;
    int Nw, NA, slots;
    size_t col0;
    double inv_scale;  // scale / (Nkz L)
    int rows;
    __device__ void operator()(int q, int r, size_t col, C v) const {
        if (r < 1 || r > Nw) return;
        const size_t rowlen = (size_t)NA * slots * 9;
        // C = conj(v) * inv; Pi = -i * scale * C, in FP64
        P[((size_t)q * Nw + (r - 1)) * rowlen + col0 + col] =
            make_double2(-(double)v.y * inv_scale, -(double)v.x * inv_scale);
    }
};

// (P - P^H)/2 on every 3x3 block of the atoms in range
__global__ void symmetrize3_kernel(sse_dims d, double2* __restrict__ P) {
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const int slots = d.NB + 1;
    const size_t nblk = (size_t)d.Nqz * d.Nw * nA * slots;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nblk; i += (size_t)gridDim.x * blockDim.x) {
        const size_t qw = i / (nA * slots), rem = i - qw * nA * slots;
        double2* B = P + ((qw * d.NA + d.a_begin) * slots + rem) * 9;
        for (int r = 0; r < 3; ++r)
            for (int c2 = r; c2 < 3; ++c2) {
                const double2 x = B[r * 3 + c2], y = B[c2 * 3 + r];
                B[r * 3 + c2] = make_double2(0.5 * (x.x - y.x), 0.5 * (x.y + y.y));
                if (r != c2) B[c2 * 3 + r] = make_double2(0.5 * (y.x - x.x), 0.5 * (y.y + x.y));
            }
    }
}

}  // namespace

struct PiLayout {
    int L;
    size_t off_tw, off_G[2], off_C[2], total;
};

PiLayout pi_layout(const sse_dims& d, size_t csz = 16) {  // csz: bytes per complex spectrum entry
    PiLayout l{};
    l.L = spectral_length(d);
    const size_t nA = (size_t)(d.a_end - d.a_begin), nel = (size_t)d.Norb * d.Norb;
    const size_t spec = (size_t)d.Nkz * l.L;
    l.off_tw = 0;
    l.off_G[0] = align256((size_t)l.L * 16);
    l.off_G[1] = align256(l.off_G[0] + spec * d.NA * nel * csz);
    l.off_C[0] = align256(l.off_G[1] + spec * d.NA * nel * csz);
    l.off_C[1] = align256(l.off_C[0] + spec * nA * (d.NB + 1) * 9 * csz);
    l.total = align256(l.off_C[1] + spec * nA * (d.NB + 1) * 9 * csz);
    return l;
}

size_t spectral_pi_workspace(const sse_dims& d) { return pi_layout(d).total; }
size_t spectral_pi32_workspace(const sse_dims& d) { return pi_layout(d, 8).total; }

bool spectral_pi_supported(const sse_dims& d) {
    const int L = spectral_length(d);
    return d.Nkz <= kMaxNk && L < kFftMaxLength && make_plan(L).smem <= 227 * 1024 && d.NB <= 16 &&
           make_pi_cfg(d, (size_t)d.Nkz * L).smem <= 227 * 1024;  // the FP32 kernel's limits are wider
}

namespace {
// Pi in the real type T: double (FP64) or float (FP32_FFT: FP32 transforms and products, FP64 inputs and outputs).
template <class T>
cudaError_t spectral_pi_t(const sse_dims& d, const int32_t* nbr, const double2* dH, const double2* G_less,
                          const double2* G_greater, double scale, uint32_t flags, double2* P_less,
                          double2* P_greater, unsigned* status, void* ws, size_t ws_bytes, cudaStream_t st) {
    using C = typename CX<T>::C;
    constexpr bool fp32 = sizeof(T) == 4;
    if (!spectral_pi_supported(d)) return cudaErrorNotSupported;
    const PiLayout lay = pi_layout(d, sizeof(C));
    if (ws_bytes < lay.total) return cudaErrorInvalidValue;
    unsigned char* base = static_cast<unsigned char*>(ws);
    C* tw = reinterpret_cast<C*>(base + lay.off_tw);
    C* Gh[2] = {reinterpret_cast<C*>(base + lay.off_G[0]), reinterpret_cast<C*>(base + lay.off_G[1])};
    C* Ch[2] = {reinterpret_cast<C*>(base + lay.off_C[0]), reinterpret_cast<C*>(base + lay.off_C[1])};
    const int L = lay.L;
    const FftPlan plan = make_plan(L, (int)sizeof(C));
    const size_t nA = (size_t)(d.a_end - d.a_begin), nel = (size_t)d.Norb * d.Norb;
    const size_t gcols = (size_t)d.NA * nel, ccols = nA * (d.NB + 1) * 9;
    if (nA == 0) return cudaSuccess;
    cudaError_t e;
    SSE_TIMED("twiddle_kernel", st, twiddle_kernel<<<grid_for(L, 256), 256, 0, st>>>(L, tw));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const double2* G[2] = {G_less, G_greater};
    const bool half = (flags & SSE_FLAG_ANTIHERMITIAN) != 0;
    const FreqMap fm = make_freq_map(d.Nkz, L, half);
    // anti-Hermitian blocks: transforms of the upper triangle's columns (sse_tri.cuh), one type at a time in the region of
    // both C^ spectra, which the products write later
    const TriMap tri = make_tri_map(d.Norb);
    const size_t tg = (size_t)d.NA * tri.nt;
    const bool use_tri = half && tri_applies(d, L, (lay.total - lay.off_C[0]) / sizeof(C));
    for (int t = 0; t < 2; ++t) {
        if (use_tri) {
            e = launch_fft32("fft_e_kernel(G)", plan, tw, LoadGTri<C>{G[t], d.NE, gcols, tri},
                             StoreSpecT<C>{Ch[0], L, tg, L}, tg, d.Nkz, st);
            if (e != cudaSuccess) return e;
            e = launch_kz_expand("dft_kz_expand_kernel(G)", Ch[0], Gh[t], tri, d.Nkz, d.Nkz, L, tg, true, st);
            if (e != cudaSuccess) return e;
            continue;
        }
        e = launch_fft32("fft_e_kernel(G)", plan, tw, LoadGT<C>{G[t], d.NE, gcols}, StoreSpecT<C>{Gh[t], L, gcols, L},
                       gcols, d.Nkz, st);
        if (e != cudaSuccess) return e;
        if ((e = launch_dft_k("dft_kz_kernel(G)", Gh[t], d.Nkz, d.Nkz, (size_t)L * gcols, 0, st)) != cudaSuccess) return e;
    }
    if (half && (flags & SSE_FLAG_CHECK))
        for (int t = 0; t < 2; ++t) {
            SSE_TIMED("check_antiherm_kernel", st,
                      check_antiherm_kernel<<<grid_for((size_t)d.Nkz * d.NE * d.NA * nel, 256), 256, 0, st>>>(
                          G[t], (size_t)d.Nkz * d.NE * d.NA, d.Norb, status));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    if constexpr (fp32) {
        const float2* Gc[2] = {Gh[0], Gh[1]};
        if ((e = launch_pi32(d, fm, nbr, dH, Gc, Ch, status, st)) != cudaSuccess) return e;
    } else {
        const PiCfg pc = make_pi_cfg(d, fm.count);
        if ((e = cudaFuncSetAttribute(spec_pi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, pc.smem)) !=
            cudaSuccess)
            return e;
        const size_t gy = (fm.count + pc.fchunk - 1) / pc.fchunk;
        SSE_TIMED("spec_pi_kernel", st,
                  spec_pi_kernel<<<dim3((unsigned)nA, (unsigned)gy, 2), pc.threads, pc.smem, st>>>(
                      pc, d, fm, nbr, dH, Gh[0], Gh[1], Ch[0], Ch[1], status));
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (half)
        for (int t = 0; t < 2; ++t) {
            SSE_TIMED("mirror_pi_kernel", st,
                      mirror_pi_kernel<<<grid_for(fm.count * nA * (d.NB + 1) * 9, 256), 256, 0, st>>>(
                          fm, nA * (d.NB + 1), Ch[t]));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    double2* P[2] = {P_less, P_greater};
    const double inv_scale = scale / ((double)d.Nkz * (double)L);
    for (int t = 0; t < 2; ++t) {
        if ((e = launch_dft_k("dft_kz_kernel(C)", Ch[t], d.Nkz, d.Nkz, (size_t)L * ccols, 1, st)) != cudaSuccess) return e;
        e = launch_fft32("fft_e_kernel(C)", plan, tw, LoadSpecConjT<C>{Ch[t], L, ccols},
                       StorePiT<C>{P[t], d.Nw, d.NA, d.NB + 1, (size_t)d.a_begin * (d.NB + 1) * 9, inv_scale,
                                   d.Nw + 1},
                       ccols, d.Nqz, st);
        if (e != cudaSuccess) return e;
        if (flags & SSE_FLAG_SYMMETRIZE) {
            SSE_TIMED("symmetrize3_kernel", st,
                      symmetrize3_kernel<<<grid_for((size_t)d.Nqz * d.Nw * nA * (d.NB + 1), 256), 256, 0, st>>>(
                          d, P[t]));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}
}  // namespace

cudaError_t spectral_pi(const sse_dims& d, const int32_t* nbr, const double2* dH, const double2* G_less,
                        const double2* G_greater, double scale, uint32_t flags, double2* P_less, double2* P_greater,
                        unsigned* status, void* ws, size_t ws_bytes, cudaStream_t st) {
    return spectral_pi_t<double>(d, nbr, dH, G_less, G_greater, scale, flags, P_less, P_greater, status, ws,
                                 ws_bytes, st);
}

cudaError_t spectral_pi32(const sse_dims& d, const int32_t* nbr, const double2* dH, const double2* G_less,
                          const double2* G_greater, double scale, uint32_t flags, double2* P_less,
                          double2* P_greater, unsigned* status, void* ws, size_t ws_bytes, cudaStream_t st) {
    return spectral_pi_t<float>(d, nbr, dH, G_less, G_greater, scale, flags, P_less, P_greater, status, ws,
                                ws_bytes, st);
}

}  // namespace sse
