// Transform kernels with compile-time sizes. (1) FP32 E-direction transforms with the DFT codelets in registers: each CTA
// transforms 8 adjacent columns of one batch, of length L = L1 * L2, in two passes (the four-step factorisation of the
// DFT: L2 DFTs of length L1 down the stride-L2 rows, the twiddles exp(-2 pi i n2 k1 / L), then L1 DFTs of length L2 along
// contiguous rows) with one exchange through shared memory. Every index inside a codelet is a constant; the radix-4/2/3
// Stockham kernel fft_e_kernel keeps the lengths without two codelet factors and the FP64 transforms. Same loader and
// store interface. (2) The kz DFT of FP32 and FP64 spectra with the grid size as a template parameter.
//
// Included at the end of sse_spectral.cuh (it uses that file's loaders, stores, CT, launch_fft and SSE_TIMED).
#pragma once

#include <string.h>

#include <algorithm>
#include <type_traits>

namespace sse {
namespace {

// cos(2 pi k / n) and sin(2 pi k / n), evaluated at compile time: the angle is reduced exactly on the integers to a
// quadrant and phi in [0, pi/2), then Taylor series of 16 terms (truncation below 1e-20).
struct CxCis {
    double c, s;
};
__host__ __device__ constexpr double cx_series(double x, bool sine) {
    double term = sine ? x : 1.0, sum = term;
    for (int i = 1; i < 16; ++i) {
        const double a = sine ? 2.0 * i : 2.0 * i - 1.0;
        term *= -x * x / (a * (a + 1.0));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr CxCis cx_cis(long k, long n) {
    k %= n;
    if (k < 0) k += n;
    const long q = (4 * k) / n, r = 4 * k - q * n;  // 2 pi k / n = (pi / 2) (q + r / n)
    const double phi = 1.5707963267948966 * (double)r / (double)n;
    const double c = cx_series(phi, false), s = cx_series(phi, true);
    return q == 0 ? CxCis{c, s} : q == 1 ? CxCis{-s, c} : q == 2 ? CxCis{-c, -s} : CxCis{s, -c};
}

template <int I, int End, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < End) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, End>(f);
    }
}

// v * exp(-2 pi i E / N) with the angle known at compile time (multiples of pi/2 without multiplies)
template <int E, int N>
__device__ __forceinline__ float2 tw_const(float2 v) {
    constexpr int e = ((E % N) + N) % N;
    if constexpr (e == 0) {
        return v;
    } else if constexpr (4 * e == N) {
        return make_float2(v.y, -v.x);
    } else if constexpr (2 * e == N) {
        return make_float2(-v.x, -v.y);
    } else if constexpr (4 * e == 3 * N) {
        return make_float2(-v.y, v.x);
    } else {
        constexpr CxCis w = cx_cis(e, N);
        constexpr float c = (float)w.c, s = (float)-w.s;  // exp(-2 pi i e / N) = c + i s
        return make_float2(fmaf(v.x, c, -v.y * s), fmaf(v.x, s, v.y * c));
    }
}

// In-place DFT of N values held in registers, X[k] = sum_n x[n] exp(-2 pi i n k / N), N = 2^a 3^b: direct forms for
// N <= 4, otherwise decimation in time N = R * M (R = 4, 2 or 3): the R DFTs of length M of the stride-R
// subsequences, the twiddles exp(-2 pi i r k' / N), and the M DFTs of length R that give X[k' + M q].
template <int N>
struct RegDft;
template <>
struct RegDft<1> {
    __device__ __forceinline__ static void run(float2 (&)[1]) {}
};
template <>
struct RegDft<2> {
    __device__ __forceinline__ static void run(float2 (&x)[2]) {
        const float2 a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    }
};
template <>
struct RegDft<3> {
    __device__ __forceinline__ static void run(float2 (&x)[3]) {
        constexpr float h = 0.86602540378443865f;  // sin(pi / 3)
        const float2 t = cadd(x[1], x[2]), d = csub(x[1], x[2]);
        const float2 m = make_float2(fmaf(-0.5f, t.x, x[0].x), fmaf(-0.5f, t.y, x[0].y));
        const float2 r = make_float2(h * d.y, -h * d.x);  // -i sin(pi/3) (x1 - x2)
        x[0] = cadd(x[0], t);
        x[1] = cadd(m, r);
        x[2] = csub(m, r);
    }
};
template <>
struct RegDft<4> {
    __device__ __forceinline__ static void run(float2 (&x)[4]) {
        const float2 s02 = cadd(x[0], x[2]), d02 = csub(x[0], x[2]);
        const float2 s13 = cadd(x[1], x[3]), d13 = csub(x[1], x[3]);
        const float2 md = make_float2(d13.y, -d13.x);  // -i (x1 - x3)
        x[0] = cadd(s02, s13);
        x[2] = csub(s02, s13);
        x[1] = cadd(d02, md);
        x[3] = csub(d02, md);
    }
};

template <int N>
struct RegDft {
    static constexpr int R = (N % 4 == 0) ? 4 : (N % 2 == 0) ? 2 : 3;
    static constexpr int M = N / R;
    static_assert(M * R == N && M > 1, "N = 2^a 3^b above 4");
    __device__ __forceinline__ static void run(float2 (&x)[N]) {
        float2 y[R][M];
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int m = 0; m < M; ++m) y[r][m] = x[R * m + r];
            RegDft<M>::run(y[r]);
        }
        static_for<0, M>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            float2 z[R];
            static_for<0, R>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                z[r] = tw_const<r * k, N>(y[r][k]);
            });
            RegDft<R>::run(z);
#pragma unroll
            for (int q = 0; q < R; ++q) x[k + M * q] = z[q];
        });
    }
};

// Columns per CTA: rows of 128 bytes, 8 columns of FP64 input or 16 of an FP32 spectrum (FinFET, inverse transform of S^,
// both types: 8 columns 3.84 ms, 16 columns 3.18, 4 columns 5.41; G with 4 columns 6.42, with 8 4.70). The large codelets
// keep 8, since two CTAs of 16 do not fit an SM.
constexpr int kE4Cols = 8, kE4ColsWide = 16;

// codelet lengths: the small set keeps two 24-point columns' worth of registers free for occupancy, the large one reaches
// L = 36^2
constexpr int kE4Small = 24, kE4Large = 36;
inline bool e4_codelet(int n, int most) {
    for (int c : {4, 6, 8, 9, 12, 16, 18, 24, 27, 32, 36})
        if (n == c) return n <= most;
    return false;
}

// f(std::integral_constant<int, n>) for a codelet length n known at run time
template <int MOST, class F>
__device__ __forceinline__ void e4_with(int n, F&& f) {
    switch (n) {
        case 4: f(std::integral_constant<int, 4>{}); break;
        case 6: f(std::integral_constant<int, 6>{}); break;
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 9: f(std::integral_constant<int, 9>{}); break;
        case 12: f(std::integral_constant<int, 12>{}); break;
        case 16: f(std::integral_constant<int, 16>{}); break;
        case 18: f(std::integral_constant<int, 18>{}); break;
        case 24: f(std::integral_constant<int, 24>{}); break;
        default:
            if constexpr (MOST > kE4Small) {
                if (n == 27) f(std::integral_constant<int, 27>{});
                else if (n == 32) f(std::integral_constant<int, 32>{});
                else f(std::integral_constant<int, 36>{});
            }
    }
}

struct E4Plan {
    int L, L1, L2, LP;  // L = L1 * L2; blocks of L2 rows padded to LP, an odd count (banks)
    int cols, threads, smem;  // one thread per column and codelet; tile + twiddle table
    bool ok, large;
};

// the most balanced factorisation into two codelet lengths, the larger at most twice the smaller (in the pass of the shorter
// DFTs a CTA's threads are idle in the ratio of the two: L = 243 = 9 * 27 lost, S^ 711 -> 939 us at NA = 1024, Norb = 6)
inline E4Plan make_e4_plan(int L, bool wide) {
    E4Plan p{};
    p.L = L;
    for (int a = 4; a * a <= L; ++a)
        if (L % a == 0 && L / a <= 2 * a && e4_codelet(a, kE4Large) && e4_codelet(L / a, kE4Large))
            p.L1 = a, p.L2 = L / a, p.ok = true;
    if (!p.ok) return p;
    p.LP = p.L2 | 1;
    p.large = p.L2 > kE4Small;
    p.cols = wide && !p.large ? kE4ColsWide : kE4Cols;
    p.threads = (p.cols * p.L2 + 31) / 32 * 32;
    p.smem = p.L1 * p.LP * p.cols * 8 + L * 8;
    return p;
}

// CTA: CC adjacent columns of one batch (blockIdx.y). ld(batch, r, col) gives row r < L (zero where the loader
// pads), sv(batch, e, col, v) takes frequency rows e < sv.rows, as for fft_e_kernel. Pass 1 reads its rows from global
// memory (all rows of a codelet in flight) and pass 2 writes its frequencies there: the tile crosses shared memory once,
// with one barrier. The codelet lengths are run-time
// choices inside one kernel, so every L = 2^a 3^b with two factors among them (all from 36 to 576 but a few) is served.
// FinFET, two types: inverse transform of S^ 4.64 -> 3.18 ms (8 columns, four barriers and four passes over shared memory
// before); L = 324 (NA = 90, Norb = 7): 97 -> 74 us against the Stockham kernel.
template <int MOST, int CC>
struct E4Bounds {  // 192 threads with four CTAs per SM or 384 with two (85 registers), 288 with two (112)
    static constexpr int THREADS = (CC * MOST + 31) / 32 * 32, CTAS = MOST <= kE4Small && CC == kE4Cols ? 4 : 2;
};

template <int MOST, int CC, class Load, class Store>
__global__ void __launch_bounds__(E4Bounds<MOST, CC>::THREADS, E4Bounds<MOST, CC>::CTAS)
    fft_e4_kernel(E4Plan p, const float2* __restrict__ tw_g, Load ld, Store sv, size_t ncols) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* X = reinterpret_cast<float2*>(smem_raw);  // [L1][LP][CC]
    float2* tw = X + p.L1 * p.LP * CC;               // [L] exp(-2 pi i m / L)
    const int tid = threadIdx.x, batch = blockIdx.y, c = tid % CC, q = tid / CC;
    const size_t col = (size_t)blockIdx.x * CC + c;
    const bool in = col < ncols;
    for (int m = tid; m < p.L; m += blockDim.x) tw[m] = tw_g[m];
    // 1. DFTs of length L1 (rows L2 n1 + n2, n2 = q), twiddled by w_L^(n2 k1)
    e4_with<MOST>(p.L1, [&](auto nc) {
        constexpr int N = decltype(nc)::value;
        float2 x[N];
#pragma unroll
        for (int n1 = 0; n1 < N; ++n1)
            x[n1] = in && q < p.L2 ? ld(batch, p.L2 * n1 + q, col) : make_float2(0.f, 0.f);
        RegDft<N>::run(x);
        __syncthreads();  // the twiddle table
        if (q < p.L2) {
#pragma unroll
            for (int k1 = 0; k1 < N; ++k1) X[(k1 * p.LP + q) * CC + c] = k1 ? cmul(x[k1], tw[q * k1]) : x[k1];
        }
    });
    __syncthreads();
    // 2. DFTs of length L2 along each block of contiguous rows (k1 = q): frequency k1 + L1 k2
    if (q >= p.L1) return;
    e4_with<MOST>(p.L2, [&](auto nc) {
        constexpr int N = decltype(nc)::value;
        float2 x[N];
#pragma unroll
        for (int n2 = 0; n2 < N; ++n2) x[n2] = X[(q * p.LP + n2) * CC + c];
        RegDft<N>::run(x);
#pragma unroll
        for (int k2 = 0; k2 < N; ++k2) {
            const int e = q + p.L1 * k2;
            if (in && e < sv.rows) sv(batch, e, col, x[k2]);
        }
    });
}

template <int MOST, int CC, class Load, class Store>
cudaError_t launch_e4_t(const char* name, const E4Plan& p, const float2* tw, Load ld, Store sv, size_t ncols, int batches,
                        cudaStream_t st) {
    auto kern = fft_e4_kernel<MOST, CC, Load, Store>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, p.smem);
    if (e != cudaSuccess) return e;
    const size_t gx = (ncols + CC - 1) / CC;
    if (gx == 0 || batches == 0) return cudaSuccess;
    if (gx > 0x7fffffffu || batches > 65535) return cudaErrorInvalidValue;
    SSE_TIMED(name, st, kern<<<dim3((unsigned)gx, (unsigned)batches), p.threads, p.smem, st>>>(p, tw, ld, sv, ncols));
    return cudaGetLastError();
}

// profile labels of the register-codelet kernels (plain, and prefetching for the FP64 inputs that it takes) for a transform
// the drivers name "fft_e_kernel(X)"
inline const char* e4_label(const char* name, bool prefetch) {
    static const char* const labels[][3] = {
        {"fft_e_kernel(G)", "fft_e4_kernel(G)", "fft_e4p_kernel(G)"},
        {"fft_e_kernel(W)", "fft_e4_kernel(W)", "fft_e4p_kernel(W)"},
        {"fft_e_kernel(K)", "fft_e4_kernel(K)"},
        {"fft_e_kernel(S)", "fft_e4_kernel(S)"},
        {"fft_e_kernel(H)", "fft_e4_kernel(H)"},
        {"fft_e_kernel(R)", "fft_e4_kernel(R)"},
        {"fft_e_kernel(C)", "fft_e4_kernel(C)"}};
    for (const auto& l : labels)
        if (strcmp(l[0], name) == 0 && l[prefetch ? 2 : 1]) return l[prefetch ? 2 : 1];
    return name;
}

// The same transform in a persistent CTA that copies the next tile into a raw staging buffer (cp.async, the
// loader's own element type) while it transforms the current one, for loaders that read one global element per
// (batch, row, column): the tile's loads are no longer a wait between the CTA's compute phases.
constexpr int kE4pSmemMax = 113 * 1024;

template <class T, class = void>
struct HasRawSrc : std::false_type {};
template <class T>
struct HasRawSrc<T, std::void_t<typename T::Raw>> : std::true_type {};
template <class T, bool = HasRawSrc<T>::value>
struct HasRawSrcType {
    using type = char;
};
template <class T>
struct HasRawSrcType<T, true> {
    using type = typename T::Raw;
};

// asynchronous copy of one 8- or 16-byte element global -> shared; with ok false the destination is zero-filled and
// nothing is read
template <int B>
__device__ __forceinline__ void cp_async_elem(uint32_t dst, const void* src, bool ok) {
    static_assert(B == 8 || B == 16, "8- or 16-byte elements");
    if constexpr (B == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(ok ? 8 : 0) : "memory");
}

template <class Load>
size_t e4p_smem(const E4Plan& p, const Load& ld) {
    return (size_t)p.smem + (size_t)ld.src_rows() * kE4Cols * sizeof(typename Load::Raw);
}

template <int MOST, class Load, class Store>
__global__ void __launch_bounds__(E4Bounds<MOST, kE4Cols>::THREADS, MOST <= kE4Small ? 3 : 2)
    fft_e4p_kernel(E4Plan p, const float2* __restrict__ tw_g, Load ld, Store sv, size_t ncols, int gx, int ntiles) {
    using Raw = typename Load::Raw;
    constexpr int CC = kE4Cols;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int rows = ld.src_rows();
    Raw* raw = reinterpret_cast<Raw*>(smem_raw);                       // [rows][CC]: the next tile as stored
    float2* X = reinterpret_cast<float2*>(raw + (size_t)rows * CC);  // [L1][LP][CC]
    float2* tw = X + p.L1 * p.LP * CC;                               // [L]
    const int tid = threadIdx.x, nt = blockDim.x, c = tid % CC;
    int q = tid / CC;
    const uint32_t raw_s = (uint32_t)__cvta_generic_to_shared(raw);
    auto issue = [&](int tile) {
        const int batch = tile / gx;
        const size_t col = (size_t)(tile % gx) * CC + c;
        const bool ok = col < ncols;
        for (int r = q; r < rows; r += nt / CC)
            cp_async_elem<(int)sizeof(Raw)>(raw_s + (uint32_t)((r * CC + c) * (int)sizeof(Raw)),
                                           ld.src(ok ? batch : 0, ok ? r : 0, ok ? col : 0), ok);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int m = tid; m < p.L; m += nt) tw[m] = tw_g[m];
    if ((int)blockIdx.x < ntiles) issue(blockIdx.x);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int batch = tile / gx;
        const size_t col = (size_t)(tile % gx) * CC + c;
        asm volatile("" : "+r"(q));  // or the addresses of every codelet length are kept across tiles (and spilled)
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the raw tile has landed for every thread; the previous tile's second pass has read X
        e4_with<MOST>(p.L1, [&](auto nc) {
            constexpr int N = decltype(nc)::value;
            if (q >= p.L2) return;
            float2 x[N];
#pragma unroll
            for (int n1 = 0; n1 < N; ++n1) {
                const int r = p.L2 * n1 + q;
                x[n1] = r < rows ? Load::cvt(raw[r * CC + c]) : make_float2(0.f, 0.f);
            }
            RegDft<N>::run(x);
#pragma unroll
            for (int k1 = 0; k1 < N; ++k1) X[(k1 * p.LP + q) * CC + c] = k1 ? cmul(x[k1], tw[q * k1]) : x[k1];
        });
        __syncthreads();  // X is complete, the raw buffer is free
        if (tile + (int)gridDim.x < ntiles) issue(tile + gridDim.x);
        if (q >= p.L1) continue;
        e4_with<MOST>(p.L2, [&](auto nc) {
            constexpr int N = decltype(nc)::value;
            float2 x[N];
#pragma unroll
            for (int n2 = 0; n2 < N; ++n2) x[n2] = X[(q * p.LP + n2) * CC + c];
            RegDft<N>::run(x);
#pragma unroll
            for (int k2 = 0; k2 < N; ++k2) {
                const int e = q + p.L1 * k2;
                if (col < ncols && e < sv.rows) sv(batch, e, col, x[k2]);
            }
        });
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int MOST, class Load, class Store>
cudaError_t launch_e4p_t(const char* name, const E4Plan& p, const float2* tw, Load ld, Store sv, size_t ncols,
                         int batches, cudaStream_t st) {
    const size_t smem = e4p_smem(p, ld);
    auto kern = fft_e4p_kernel<MOST, Load, Store>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const size_t gx = (ncols + kE4Cols - 1) / kE4Cols;
    if (gx == 0 || batches == 0) return cudaSuccess;
    if (gx * (size_t)batches > 0x7fffffffu) return cudaErrorInvalidValue;
    const int ntiles = (int)(gx * (size_t)batches);
    int dev = 0, nsm = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, p.threads, smem)) != cudaSuccess) return e;
    const int grid = std::min(ntiles, std::max(1, per_sm) * nsm);
    SSE_TIMED(name, st, kern<<<grid, p.threads, smem, st>>>(p, tw, ld, sv, ncols, (int)gx, ntiles));
    return cudaGetLastError();
}

// loaders of an FP32 spectrum
template <class Load>
constexpr bool e4_wide = HasRawSrc<Load>::value && sizeof(typename HasRawSrcType<Load>::type) == 8;

// The prefetching kernel for FP64 input tiles where the staging buffer fits: FinFET, transform of G, both types 4.70 ms
// against 6.22 with fft_e4_kernel (the conversions hold up its loads); fft_e4_kernel for FP32 input, which needs none.
template <int MOST, class Load, class Store>
cudaError_t launch_e4_any(const char* name, const E4Plan& p, const float2* tw, Load ld, Store sv, size_t ncols,
                          int batches, cudaStream_t st) {
    if constexpr (HasRawSrc<Load>::value && sizeof(typename HasRawSrcType<Load>::type) == 16) {
        if (e4p_smem(p, ld) <= (size_t)kE4pSmemMax)
            return launch_e4p_t<MOST>(e4_label(name, true), p, tw, ld, sv, ncols, batches, st);
    }
    if constexpr (e4_wide<Load> && MOST <= kE4Small)
        return launch_e4_t<MOST, kE4ColsWide>(e4_label(name, false), p, tw, ld, sv, ncols, batches, st);
    else
        return launch_e4_t<MOST, kE4Cols>(e4_label(name, false), p, tw, ld, sv, ncols, batches, st);
}

// FP64 tiles that are read in full but do not fit the staging buffer: the 27-point codelets (radix 3 only) lose to the
// Stockham kernel there (G at NA = 512, Norb = 6: L = 729 1687 against 1290 us, L = 972 1760 against 1557; the 32 x 36
// codelets of L = 1152 do not). The pairs without 27 of two such lengths lose as well: 18 x 36 of L = 648 557 against 515 us,
// 24 x 36 of L = 864 729 against 576 (the same sizes, Nkz = 2).
template <class Load>
bool e4_loses(const E4Plan& p, const Load& ld) {
    if constexpr (HasRawSrc<Load>::value && sizeof(typename HasRawSrcType<Load>::type) == 16)
        return (p.L1 == 27 || p.L2 == 27) && e4p_smem(p, ld) > (size_t)kE4pSmemMax;
    else
        return false;
}

// FP32 E-transforms of the lengths with two codelet factors; every other length, and the FP64 transforms, take
// fft_e_kernel.
template <class Load, class Store>
cudaError_t launch_fft32(const char* name, const FftPlan& p, const typename Load::C* tw, Load ld, Store sv, size_t ncols,
                         int batches, cudaStream_t st) {
    if constexpr (std::is_same<typename Load::C, float2>::value) {
        const E4Plan e4 = make_e4_plan(p.L, e4_wide<Load>);
        if (e4.ok && !e4_loses(e4, ld))
            return e4.large ? launch_e4_any<kE4Large>(name, e4, tw, ld, sv, ncols, batches, st)
                            : launch_e4_any<kE4Small>(name, e4, tw, ld, sv, ncols, batches, st);
    }
    return launch_fft(name, p, tw, ld, sv, ncols, batches, st);
}

// kz-direction DFT with the grid size Nk as a template parameter (FP32 and FP64 spectra), in place on X[Nk][M]:
// out[kappa] = sum_{k < n_in} x_k exp(-+2 pi i k kappa / Nk), one column m per thread, the column in registers and
// the cosines and sines compile-time constants. Inputs k and Nk - k are paired (p = x_k + x_{Nk-k},
// q = x_k - x_{Nk-k}) and so are outputs kappa and Nk - kappa: out[kappa] = C -+ i S, out[Nk - kappa] = C +- i S
// with C = x_0 (+ (-1)^kappa x_{Nk/2}) + sum_k p_k cos(2 pi k kappa / Nk), S = sum_k q_k sin(2 pi k kappa / Nk).
// out(kappa, value) takes each result once.
template <class C, int NK, class Out>
__device__ __forceinline__ void kz_dft(const C (&x)[NK], int inverse, Out&& out) {
    using R = typename CT<C>::R;
    constexpr int H = (NK - 1) / 2;  // (k, NK - k) pairs
    constexpr bool EVEN = NK % 2 == 0;
    const R sgn = inverse ? (R)1 : (R)-1;
    C p[H + 1], q[H + 1];
    C c0 = x[0];
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        p[k] = cadd(x[k], x[NK - k]);
        q[k] = csub(x[k], x[NK - k]);
        c0 = cadd(c0, p[k]);
    }
    const C xh = EVEN ? x[NK / 2] : CT<C>::mk(0, 0);
    out(0, cadd(c0, xh));
    static_for<1, H + 1>([&](auto kc) {
        constexpr int kap = decltype(kc)::value;
        C Cs = x[0], Sn = CT<C>::mk(0, 0);
        static_for<1, H + 1>([&](auto jc) {
            constexpr int k = decltype(jc)::value;
            constexpr CxCis w = cx_cis((long)k * kap, NK);
            Cs.x = fma(p[k].x, (R)w.c, Cs.x);
            Cs.y = fma(p[k].y, (R)w.c, Cs.y);
            Sn.x = fma(q[k].x, (R)w.s, Sn.x);
            Sn.y = fma(q[k].y, (R)w.s, Sn.y);
        });
        if constexpr (EVEN) {
            constexpr R e = (kap & 1) ? (R)-1 : (R)1;
            Cs.x = fma(e, xh.x, Cs.x);
            Cs.y = fma(e, xh.y, Cs.y);
        }
        out(kap, CT<C>::mk(Cs.x - sgn * Sn.y, Cs.y + sgn * Sn.x));
        out(NK - kap, CT<C>::mk(Cs.x + sgn * Sn.y, Cs.y - sgn * Sn.x));
    });
    if constexpr (EVEN && NK > 1) {  // kappa = NK/2: cos(pi k) = (-1)^k, sin = 0
        C Cs = x[0];
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            const R e = (k & 1) ? (R)-1 : (R)1;
            Cs.x = fma(e, p[k].x, Cs.x);
            Cs.y = fma(e, p[k].y, Cs.y);
        }
        constexpr R e = ((NK / 2) & 1) ? (R)-1 : (R)1;
        out(NK / 2, CT<C>::mk(fma(e, xh.x, Cs.x), fma(e, xh.y, Cs.y)));
    }
}

template <class C, int NK>
__global__ void __launch_bounds__(256) dft_kz_kernel(C* __restrict__ X, int n_in, size_t M, int inverse) {
    for (size_t m = blockIdx.x * (size_t)blockDim.x + threadIdx.x; m < M; m += (size_t)gridDim.x * blockDim.x) {
        C x[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) x[k] = k < n_in ? X[(size_t)k * M + m] : CT<C>::mk(0, 0);
        kz_dft<C, NK>(x, inverse, [&](int kap, C v) { X[(size_t)kap * M + m] = v; });
    }
}

template <class C, int NK>
cudaError_t launch_dft_kz_t(const char* name, C* X, int n_in, size_t M, int inverse, cudaStream_t st) {
    SSE_TIMED(name, st, dft_kz_kernel<C, NK><<<grid_for(M, 256), 256, 0, st>>>(X, n_in, M, inverse));
    return cudaGetLastError();
}

// the kz DFT of a spectrum: the compile-time kernel for Nk = 1 .. kMaxNk
template <class C>
cudaError_t launch_dft_k(const char* name, C* X, int Nk, int n_in, size_t M, int inverse, cudaStream_t st) {
    if (M == 0) return cudaSuccess;
    switch (Nk) {
        case 1: return launch_dft_kz_t<C, 1>(name, X, n_in, M, inverse, st);
        case 2: return launch_dft_kz_t<C, 2>(name, X, n_in, M, inverse, st);
        case 3: return launch_dft_kz_t<C, 3>(name, X, n_in, M, inverse, st);
        case 4: return launch_dft_kz_t<C, 4>(name, X, n_in, M, inverse, st);
        case 5: return launch_dft_kz_t<C, 5>(name, X, n_in, M, inverse, st);
        case 6: return launch_dft_kz_t<C, 6>(name, X, n_in, M, inverse, st);
        case 7: return launch_dft_kz_t<C, 7>(name, X, n_in, M, inverse, st);
        case 8: return launch_dft_kz_t<C, 8>(name, X, n_in, M, inverse, st);
        case 9: return launch_dft_kz_t<C, 9>(name, X, n_in, M, inverse, st);
        case 10: return launch_dft_kz_t<C, 10>(name, X, n_in, M, inverse, st);
        case 11: return launch_dft_kz_t<C, 11>(name, X, n_in, M, inverse, st);
        case 12: return launch_dft_kz_t<C, 12>(name, X, n_in, M, inverse, st);
        case 13: return launch_dft_kz_t<C, 13>(name, X, n_in, M, inverse, st);
        case 14: return launch_dft_kz_t<C, 14>(name, X, n_in, M, inverse, st);
        case 15: return launch_dft_kz_t<C, 15>(name, X, n_in, M, inverse, st);
        case 16: return launch_dft_kz_t<C, 16>(name, X, n_in, M, inverse, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace sse
