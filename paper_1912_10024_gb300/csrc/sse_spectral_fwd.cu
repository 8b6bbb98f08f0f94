// Sigma of Eq. (3) through the transforms: the per-frequency block products in FP64 (spec_prod_kernel, mode
// FP64_FFT) and FP32 (spec_prod32_kernel, mode FP32_FFT), the symmetrisation, the workspace layout and the
// drivers (device buffers, and the pipelined variant behind the host-buffer entry point). Mode F16X3_FFT runs the
// same FP32 transforms with the block products of sse_spectral_tc.cu on the tensor cores.
#include "sse_prod32.cuh"
#include "sse_tri.cuh"

namespace sse {
namespace {

template <class T>
__global__ void spec_prod_kernel(ProdCfg c, sse_dims d, FreqMap fm, const int32_t* __restrict__ nbr,
                                 const double2* __restrict__ dH, const typename CX<T>::C* __restrict__ Ghat,
                                 const typename CX<T>::C* __restrict__ Khat, typename CX<T>::C* __restrict__ Shat,
                                 double scale, unsigned* __restrict__ status) {
    using C = typename CX<T>::C;
    extern __shared__ __align__(16) unsigned char smem[];
    const int Norb = d.Norb, nel = c.nel;
    const int la = blockIdx.x;
    const int a = d.a_begin + la;
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const size_t i_begin = (size_t)blockIdx.y * c.fchunk;  // frequency indices of the map
    const size_t i_end = min(fm.count, i_begin + c.fchunk);
    T* sA = reinterpret_cast<T*>(smem + c.off_A);
    T* sG = reinterpret_cast<T*>(smem + c.off_G);
    C* sK = reinterpret_cast<C*>(smem + c.off_K);
    T* sW = reinterpret_cast<T*>(smem + c.off_W);
    T* sU = reinterpret_cast<T*>(smem + c.off_U);
    const int tid = threadIdx.x;
    const int fl = tid / nel, e = tid - fl * nel;
    const int m = e / Norb, n = e - m * Norb;
    const bool lane = fl < c.F;

    for (int i = tid; i < d.NB * 3 * nel; i += blockDim.x) {
        const int si = i / nel, ee = i - si * nel;
        const double2 v = dH[((size_t)a * d.NB) * 3 * nel + i];
        put3(sA + (size_t)si * 3 * nel, nel, ee, CT<C>::mk((T)v.x, (T)v.y));
    }
    int bnb[16];
    for (int s = 0; s < d.NB && s < 16; ++s) {
        const int b = nbr[(size_t)a * d.NB + s];
        bnb[s] = (b >= 0 && b < d.NA) ? b : -1;
        if (bnb[s] < 0 && tid == 0) atomicOr(status, DEV_BAD_NEIGHBOUR);
    }
    __syncthreads();

    for (size_t i0 = i_begin; i0 < i_end; i0 += c.F) {
        const bool act = lane && i0 + fl < i_end;
        const size_t f = act ? freq_of(fm, i0 + fl) : 0;
        T T1 = 0, T2 = 0, T3 = 0;
        for (int s = 0; s < d.NB; ++s) {
            const int b = s < 16 ? bnb[s] : -1;
            // stage G^_b(f) and K^_(a,s)(f)
            if (lane) {
                C g = CT<C>::mk(0, 0);
                if (act && b >= 0) g = Ghat[(f * d.NA + b) * nel + e];
                put3(sG + (size_t)fl * 3 * nel, nel, e, g);
            }
            for (int i = tid; i < c.F * 9; i += blockDim.x) {
                const int fk = i / 9, ij = i - fk * 9;
                C k = CT<C>::mk(0, 0);
                if (i0 + fk < i_end && b >= 0) k = Khat[((freq_of(fm, i0 + fk) * nA + la) * d.NB + s) * 9 + ij];
                sK[i] = k;
            }
            __syncthreads();
            // W_i[m][n] = sum_j K_ij conj(dH_j[n][m])
            if (lane) {
                const T* A = sA + (size_t)s * 9 * nel;
                const int et = n * Norb + m;
                T ar[3], ai[3];  // conj(dH_j[n][m]) = (ar, -ai)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    ar[j] = A[(size_t)j * 3 * nel + et];
                    ai[j] = A[(size_t)j * 3 * nel + nel + et];
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    C acc = CT<C>::mk(0, 0);  // plain FMA chains: no separate multiplies or adds
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const C k = sK[fl * 9 + i * 3 + j];
                        acc.x = fma(k.x, ar[j], acc.x);
                        acc.x = fma(k.y, ai[j], acc.x);
                        acc.y = fma(k.y, ar[j], acc.y);
                        acc.y = fma(-k.x, ai[j], acc.y);
                    }
                    put3(sW + ((size_t)fl * 3 + i) * 3 * nel, nel, e, acc);
                }
            }
            __syncthreads();
            // U_i = G^ W_i
            if (lane) {
                const T* Gp = sG + (size_t)fl * 3 * nel;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const T* Wp = sW + ((size_t)fl * 3 + i) * 3 * nel;
                    T t1 = 0, t2 = 0, t3 = 0;
                    for (int l = 0; l < Norb; ++l) {
                        const int ga = m * Norb + l, wb = l * Norb + n;
                        t1 = fma(Gp[ga], Wp[wb], t1);
                        t2 = fma(Gp[nel + ga], Wp[nel + wb], t2);
                        t3 = fma(Gp[2 * nel + ga], Wp[2 * nel + wb], t3);
                    }
                    put3(sU + ((size_t)fl * 3 + i) * 3 * nel, nel, e, CT<C>::mk(t1 - t2, t3 - t1 - t2));
                }
            }
            __syncthreads();
            // acc += sum_i dH_i U_i
            if (lane) {
                const T* A = sA + (size_t)s * 9 * nel;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const T* Ap = A + (size_t)i * 3 * nel;
                    const T* Up = sU + ((size_t)fl * 3 + i) * 3 * nel;
                    for (int l = 0; l < Norb; ++l) {
                        const int aa = m * Norb + l, ub = l * Norb + n;
                        T1 = fma(Ap[aa], Up[ub], T1);
                        T2 = fma(Ap[nel + aa], Up[nel + ub], T2);
                        T3 = fma(Ap[2 * nel + aa], Up[2 * nel + ub], T3);
                    }
                }
            }
        }
        if (act) {
            const T re = T1 - T2, im = T3 - T1 - T2;
            Shat[(f * nA + la) * nel + e] = CT<C>::mk((T)(-scale * (double)im), (T)(scale * (double)re));  // i*scale*(re+i im)
        }
    }
}

// (S - S^H)/2 on the blocks of atoms in range: FP32 spectra, and FP64 ones where the inverse kz DFT does not project
// (Nkz > 8). A CTA takes about 1024 elements of whole blocks through shared memory, so that the accesses are contiguous
// although every element meets its transposed one, and divides 64-bit indices once per block. NA = 90, Norb = 7, NE = 301,
// Nkz = 4, both types: 131 -> 96 us (340 MB, 50 us; the FP64 operations 35 us). Forming each pair of elements once halves
// those but adds a pass over shared memory: 120 us.
constexpr int kSymElems = 1024, kSymThreads = 256;

__global__ void __launch_bounds__(kSymThreads) symmetrize_kernel(sse_dims d, double2* __restrict__ S) {
    __shared__ double2 tile[kSymElems];
    __shared__ double2* base[kSymElems];
    const int Norb = d.Norb, nel = Norb * Norb, per = kSymElems / nel;  // nel <= 256
    const size_t nA = (size_t)(d.a_end - d.a_begin);
    const size_t nblk = (size_t)d.Nkz * d.NE * nA;
    for (size_t b0 = (size_t)blockIdx.x * per; b0 < nblk; b0 += (size_t)gridDim.x * per) {
        const int nb = (int)min((size_t)per, nblk - b0);
        for (int i = threadIdx.x; i < nb; i += kSymThreads) {
            const size_t ke = (b0 + i) / nA, la = b0 + i - ke * nA;
            base[i] = S + (ke * d.NA + d.a_begin + la) * nel;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb * nel; i += kSymThreads) {
            const int blk = i / nel;
            tile[i] = base[blk][i - blk * nel];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb * nel; i += kSymThreads) {
            const int blk = i / nel, e = i - blk * nel, m = e / Norb, n = e - m * Norb;
            const double2 x = tile[i], y = tile[blk * nel + n * Norb + m];
            base[blk][e] = make_double2(0.5 * (x.x - y.x), 0.5 * (x.y + y.y));
        }
        __syncthreads();  // tile and base are rewritten
    }
}

inline unsigned symmetrize_grid(const sse_dims& d, int Nkz) {
    const size_t nblk = (size_t)Nkz * d.NE * (size_t)(d.a_end - d.a_begin);
    const size_t per = kSymElems / (d.Norb * d.Norb), g = (nblk + per - 1) / per;
    return (unsigned)(g < 1 ? 1 : g > 0x7fffffff ? 0x7fffffff : g);
}

struct SpecLayout {
    int L;
    size_t off_tw, off_G, off_K, off_S, total;
};

SpecLayout spec_layout(const sse_dims& d, size_t csz = 16) {  // csz: bytes per complex spectrum entry
    SpecLayout l{};
    l.L = spectral_length(d);
    const size_t nA = (size_t)(d.a_end - d.a_begin), nel = (size_t)d.Norb * d.Norb;
    const size_t spec = (size_t)d.Nkz * l.L;
    l.off_tw = 0;
    l.off_G = align256(l.off_tw + (size_t)l.L * 16);
    l.off_K = align256(l.off_G + spec * d.NA * nel * csz);
    l.off_S = align256(l.off_K + spec * nA * d.NB * 9 * csz);
    l.total = align256(l.off_S + spec * nA * nel * csz);
    return l;
}

}  // namespace

int spectral_length(const sse_dims& d) {
    for (int L = d.NE + d.Nw;; ++L) {  // smallest 2^a 3^b: radix-4/2/3 stages only
        int m = L;
        while (m % 2 == 0) m /= 2;
        while (m % 3 == 0) m /= 3;
        if (m == 1) return L;
    }
}

bool spectral_supported(const sse_dims& d) {
    const int L = spectral_length(d);
    return d.Nkz <= kMaxNk && L < kFftMaxLength && make_plan(L).smem <= 227 * 1024 && d.NB <= 16 &&
           make_prod_cfg(d, (size_t)d.Nkz * L).smem <= 227 * 1024;
}

// The FP32 product kernel takes every block size and bond count of spectral_supported.
bool spectral_fwd_supported(const sse_dims& d) { return spectral_supported(d); }

size_t spectral_fwd_workspace(const sse_dims& d) { return spec_layout(d).total; }
size_t spectral_fwd32_workspace(const sse_dims& d) { return spec_layout(d, 8).total; }

namespace {
// The forward in the real type T: double (FP64_FFT) or float (FP32_FFT: FP32 transforms and block
// products on the FP32 pipe, FP64 inputs and outputs).
template <class T>
cudaError_t spectral_fwd_t(const Problem& p, double2* S_less, double2* S_greater, unsigned* status, void* ws,
                           size_t ws_bytes, cudaStream_t st, const FwdPipe* pipe = nullptr, bool tc = false) {
    // With `pipe` (inputs arriving from the host): the lag kernel is transformed first, G^t slice by slice as its
    // kz slices arrive, and the inverse E-transform of Sigma^t runs slice by slice so that each slice's download
    // can start; without it every transform is one launch over all slices.
    using C = typename CX<T>::C;
    const sse_dims& d = p.d;
    // tc: mode F16X3_FFT, the FP32 transforms with the block products on the tensor cores where those are faster
    if (tc && sizeof(T) != 4) return cudaErrorNotSupported;
    if (!(tc ? spectral_fwd_tc_supported(d) : spectral_fwd_supported(d))) return cudaErrorNotSupported;
    const SpecLayout lay = spec_layout(d, sizeof(C));
    if (ws_bytes < lay.total) return cudaErrorInvalidValue;
    unsigned char* base = static_cast<unsigned char*>(ws);
    C* tw = reinterpret_cast<C*>(base + lay.off_tw);
    C* Gh = reinterpret_cast<C*>(base + lay.off_G);
    C* Kh = reinterpret_cast<C*>(base + lay.off_K);
    C* Sh = reinterpret_cast<C*>(base + lay.off_S);
    const int L = lay.L;
    const FftPlan plan = make_plan(L, (int)sizeof(C));
    const size_t nA = (size_t)(d.a_end - d.a_begin), nel = (size_t)d.Norb * d.Norb;
    const size_t gcols = (size_t)d.NA * nel, kcols = nA * d.NB * 9, scols = nA * nel;
    cudaError_t e;
    if (nA == 0) return cudaSuccess;

    SSE_TIMED("twiddle_kernel", st, twiddle_kernel<<<grid_for(L, 256), 256, 0, st>>>(L, tw));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const bool half = (p.flags & SSE_FLAG_ANTIHERMITIAN) != 0;
    const FreqMap fm = make_freq_map(d.Nkz, L, half);
    if (half && (p.flags & SSE_FLAG_CHECK)) {
        if (pipe)  // every input (the copies are issued in order on one stream)
            if ((e = cudaStreamWaitEvent(st, pipe->g[1][d.Nkz - 1], 0)) != cudaSuccess) return e;
        for (int t = 0; t < 2; ++t) {
            SSE_TIMED("check_antiherm_kernel", st,
                      check_antiherm_kernel<<<grid_for((size_t)d.Nkz * d.NE * d.NA * nel, 256), 256, 0, st>>>(
                          p.G[t], (size_t)d.Nkz * d.NE * d.NA, d.Norb, status));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            SSE_TIMED("check_antiherm_kernel", st,
                      check_antiherm_kernel<<<grid_for((size_t)d.Nqz * d.Nw * d.NA * d.NB * 9, 256), 256, 0, st>>>(
                          p.D[t], (size_t)d.Nqz * d.Nw * d.NA * d.NB, 3, status));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    // anti-Hermitian blocks: transforms of the upper triangle's columns (sse_tri.cuh). The triangle of G^ sits in S^'s
    // region until the products write there, that of S^ in G^'s after them.
    const TriMap tri = make_tri_map(d.Norb);
    const bool use_tri = half && tri_applies(d, L, (size_t)d.Nkz * L * scols);
    const size_t tg = (size_t)d.NA * tri.nt, ts = nA * tri.nt;  // columns
    // Symmetrised Sigma of general inputs: projected in the inverse kz DFT, then likewise by its triangle. FP64 spectra only:
    // the symmetrisation is FP64 arithmetic in every mode, so FP32 spectra are transformed back in full and
    // symmetrize_kernel averages each pair of elements, anti-Hermitian inputs included.
    const bool sym = (p.flags & SSE_FLAG_SYMMETRIZE) != 0;
    const bool use_project = sizeof(T) == 8 && sym && !half && tri_applies(d, L, (size_t)-1);
    const bool s_tri = use_project || (use_tri && (sizeof(T) == 8 || !sym));
    // the same for the 3 x 3 blocks of the lag kernel, whose triangle comes before that of G^ in S^'s region
    const TriMap tri3 = make_tri_map(3);
    const size_t tk = nA * d.NB * tri3.nt;
    const bool use_tri3 = use_tri && tk <= scols && tk <= 0x7fffffffu;
    C* Kc = Sh;
    C* Gc = Sh;
    C* Sc = Gh;
    const ProdCfg pc = make_prod_cfg(d, fm.count, (int)sizeof(T));
    constexpr bool tiled = sizeof(T) == 4;  // FP32: register-tiled kernel
    if constexpr (!tiled)
        if ((e = cudaFuncSetAttribute(spec_prod_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, pc.smem)) !=
            cudaSuccess)
            return e;
    double2* S[2] = {S_less, S_greater};
    if (pipe && (e = cudaStreamWaitEvent(st, pipe->inputs, 0)) != cudaSuccess) return e;
    for (int t = 0; t < 2; ++t) {
        // 1. lag kernel -> K^ (needs only D; with `pipe` it runs while G^t is still arriving)
        const size_t rowlen = (size_t)d.NA * d.NB * 9, kcol0 = (size_t)d.a_begin * d.NB * 9;
        if (use_tri3) {
            e = launch_fft32("fft_e_kernel(K)", plan, tw,
                             LoadLagTri<C>{p.D[t], p.D[1 - t], d.Nw, L, rowlen, kcol0, tri3},
                             StoreSpecT<C>{Kc, L, tk, L}, tk, d.Nqz, st);
            if (e != cudaSuccess) return e;
            e = launch_kz_expand("dft_kz_expand_kernel(K)", Kc, Kh, tri3, d.Nkz, d.Nqz, L, tk, false, st);
        } else {
            e = launch_fft32("fft_e_kernel(K)", plan, tw, LoadLagT<C>{p.D[t], p.D[1 - t], d.Nw, L, rowlen, kcol0},
                             StoreSpecT<C>{Kh, L, kcols, L}, kcols, d.Nqz, st);
            if (e != cudaSuccess) return e;
            e = launch_dft_k("dft_kz_kernel(K)", Kh, d.Nkz, d.Nqz, (size_t)L * kcols, 0, st);
        }
        if (e != cudaSuccess) return e;
        // 2. G^t -> G^ (E-transform per kz slice as the slices arrive, then the kz DFT)
        const int gslices = pipe ? d.Nkz : 1, gper = pipe ? 1 : d.Nkz;
        for (int k = 0; k < gslices; ++k) {
            if (pipe && (e = cudaStreamWaitEvent(st, pipe->g[t][k], 0)) != cudaSuccess) return e;
            const double2* Gk = p.G[t] + (size_t)k * d.NE * gcols;
            if (use_tri)
                e = launch_fft32("fft_e_kernel(G)", plan, tw, LoadGTri<C>{Gk, d.NE, gcols, tri},
                                 StoreSpecT<C>{Gc + (size_t)k * L * tg, L, tg, L}, tg, gper, st);
            else
                e = launch_fft32("fft_e_kernel(G)", plan, tw, LoadGT<C>{Gk, d.NE, gcols},
                                 StoreSpecT<C>{Gh + (size_t)k * L * gcols, L, gcols, L}, gcols, gper, st);
            if (e != cudaSuccess) return e;
        }
        e = use_tri ? launch_kz_expand("dft_kz_expand_kernel(G)", Gc, Gh, tri, d.Nkz, d.Nkz, L, tg, false, st)
                    : launch_dft_k("dft_kz_kernel(G)", Gh, d.Nkz, d.Nkz, (size_t)L * gcols, 0, st);
        if (e != cudaSuccess) return e;
        // 3. block products (one frequency of each (f, -f) pair with anti-Hermitian inputs, then the mirror)
        if (tc && spectral_prod_tc_pays(d)) {
            e = spectral_prod_tc(d, fm, p.nbr, p.dH, reinterpret_cast<const float2*>(Gh),
                                 reinterpret_cast<const float2*>(Kh), reinterpret_cast<float2*>(Sh), p.scale, status,
                                 st);
            if (e != cudaSuccess) return e;
        } else if constexpr (tiled) {
            e = launch_prod32<false>(TileArgs{d, fm, p.nbr, nullptr, nullptr, p.dH, Gh, Kh, Sh, p.scale, status}, nA, st);
            if (e != cudaSuccess) return e;
        } else {
            const size_t gy = (fm.count + pc.fchunk - 1) / pc.fchunk;
            SSE_TIMED("spec_prod_kernel", st,
                      spec_prod_kernel<T><<<dim3((unsigned)nA, (unsigned)gy), pc.threads, pc.smem, st>>>(
                          pc, d, fm, p.nbr, p.dH, Gh, Kh, Sh, p.scale, status));
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (half && !s_tri) {
            SSE_TIMED("mirror_sigma_kernel", st,
                      mirror_sigma_kernel<<<grid_for(fm.count * nA * nel, 256), 256, 0, st>>>(fm, nA, d.Norb, Sh));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        // 4. inverse transforms into Sigma^t
        if (use_project) {
            if constexpr (sizeof(T) == 8)
                e = launch_kz_project("dft_kz_project_kernel(S)", Sh, Sc, tri, d.Nkz, L, ts, st);
        } else if (s_tri) {
            e = launch_kz_compress("dft_kz_compress_kernel(S)", Sh, Sc, tri, d.Nkz, L, ts, st);
        } else {
            e = launch_dft_k("dft_kz_kernel(S)", Sh, d.Nkz, d.Nkz, (size_t)L * scols, 1, st);
        }
        if (e != cudaSuccess) return e;
        const double inv = (use_project ? 0.5 : 1.0) / ((double)d.Nkz * (double)L);
        // with `pipe` slice by slice, each handed to its download as soon as it is written
        const int sslices = pipe ? d.Nkz : 1, sper = pipe ? 1 : d.Nkz;
        sse_dims dk = d;
        dk.Nkz = sper;
        for (int k = 0; k < sslices; ++k) {
            double2* Sk = S[t] + (size_t)k * d.NE * d.NA * nel;
            if (s_tri)
                e = launch_fft32("fft_e_kernel(S)", plan, tw, LoadSpecConjT<C>{Sc + (size_t)k * L * ts, L, ts},
                                 StoreSigmaTri<C>{Sk, d.NE, gcols, (size_t)d.a_begin * nel, inv, d.NE, sym ? 1 : 0, tri},
                                 ts, sper, st);
            else
                e = launch_fft32("fft_e_kernel(S)", plan, tw, LoadSpecConjT<C>{Sh + (size_t)k * L * scols, L, scols},
                                 StoreSigmaT<C>{Sk, d.NE, gcols, (size_t)d.a_begin * nel, inv, d.NE}, scols, sper, st);
            if (e != cudaSuccess) return e;
            if (sym && !s_tri) {
                SSE_TIMED("symmetrize_kernel", st,
                          symmetrize_kernel<<<symmetrize_grid(d, sper), kSymThreads, 0, st>>>(dk, Sk));
                if ((e = cudaGetLastError()) != cudaSuccess) return e;
            }
            if (pipe && (e = cudaEventRecord(pipe->s[t][k], st)) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}
}  // namespace

cudaError_t spectral_fwd_pipelined(const Problem& p, int mode, double2* S_less, double2* S_greater, unsigned* status,
                                   void* ws, size_t ws_bytes, cudaStream_t st, const FwdPipe& pipe) {
    if (mode == SSE_MODE_FP64_FFT) return spectral_fwd_t<double>(p, S_less, S_greater, status, ws, ws_bytes, st, &pipe);
    return spectral_fwd_t<float>(p, S_less, S_greater, status, ws, ws_bytes, st, &pipe, mode == SSE_MODE_F16X3_FFT);
}

cudaError_t spectral_fwd(const Problem& p, double2* S_less, double2* S_greater, unsigned* status, void* ws,
                         size_t ws_bytes, cudaStream_t st) {
    return spectral_fwd_t<double>(p, S_less, S_greater, status, ws, ws_bytes, st);
}

cudaError_t spectral_fwd32(const Problem& p, double2* S_less, double2* S_greater, unsigned* status, void* ws,
                           size_t ws_bytes, cudaStream_t st) {
    return spectral_fwd_t<float>(p, S_less, S_greater, status, ws, ws_bytes, st);
}

bool spectral_fwd_tc_supported(const sse_dims& d) {
    return spectral_fwd_supported(d) && spectral_prod_tc_supported(d);
}

cudaError_t spectral_fwd_tc(const Problem& p, double2* S_less, double2* S_greater, unsigned* status, void* ws,
                            size_t ws_bytes, cudaStream_t st) {
    return spectral_fwd_t<float>(p, S_less, S_greater, status, ws, ws_bytes, st, nullptr, true);
}

}  // namespace sse
