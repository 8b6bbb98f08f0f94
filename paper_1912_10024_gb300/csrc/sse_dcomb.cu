// Bond weights of Eq. (3): Dc_ab = D_ba - D_bb - D_aa + D_ab (Sec. 2), and their adjoint.
//
// Raw phonon Green's functions: [Nqz][Nw][NA][NB+1][3][3], slot s < NB = D_ab for
// b = nbr[a][s], slot NB = the self block D_aa. D_ba is the block atom b stores in
// the slot s' with nbr[b][s'] = a (symmetric neighbour lists). No atomics, so the results are deterministic.
//
// Both kernels are gathers. A thread keeps its column (the same for every (qz, w)) and walks down the
// rows: consecutive threads read and write consecutive 16-byte words, and the neighbour lookup (dependent loads) and the
// index arithmetic are paid once per thread. The forward takes a row at a time, eight independent loads, with four CTAs
// per SM: with two rows and two CTAs it took 204 us at the FinFET workload, but 60 us instead of 34 for one row of
// NA = 32000, NB = 4 (a thread per block: 40) and 131 instead of 78 for one row of NA = 16384, NB = 16.
// What bounds them is not only HBM: six (forward) and four (adjoint) FP64 additions per complex entry take 163 and 108 us
// on the FP64 pipe at the FinFET workload, against 87 us for the bytes of each. Measured there: forward 207 us, adjoint
// 144 us (one thread per 144-byte block, nine strided words each: 214 and 279 us; one short-lived thread per entry and
// four rows, which repeats the lookups: about 600 us each).
#include <cuda_runtime.h>
#include <stdint.h>

#include "sse_internal.h"

namespace sse {
namespace {

__device__ __forceinline__ int reverse_slot(const int32_t* nbr, int NB, int a, int b) {
    for (int s = 0; s < NB; ++s)
        if (nbr[(size_t)b * NB + s] == a) return s;
    return -1;
}

constexpr int kDcombThreads = 256;
constexpr int kDcombTableBonds = 64;  // bonds per atom up to which the adjoint keeps its reverse bonds in shared memory

// Dc[q][w][a][s] for atoms in range; bonds without a reverse slot (or an out-of-range
// neighbour) get zero and raise the status bit. One thread per output entry of a row, both types of a row at a time.
__global__ void __launch_bounds__(kDcombThreads, 4)
dcomb_fwd_kernel(sse_dims d, const int32_t* __restrict__ nbr, const double2* __restrict__ raw_l,
                 const double2* __restrict__ raw_g, double2* __restrict__ Dl, double2* __restrict__ Dg,
                 unsigned* __restrict__ status) {
    const size_t col = blockIdx.x * (size_t)blockDim.x + threadIdx.x;  // (atom in range, slot, entry)
    if (col >= (size_t)(d.a_end - d.a_begin) * d.NB * 9) return;
    const size_t la = col / 9 / d.NB;
    const int bond = (int)(col / 9 - la * d.NB), e = (int)(col % 9);
    const int a = d.a_begin + (int)la;
    const int b = nbr[(size_t)a * d.NB + bond];
    const int sr = (b >= 0 && b < d.NA) ? reverse_slot(nbr, d.NB, a, b) : -1;
    const bool ok = sr >= 0;
    if (!ok && e == 0 && blockIdx.y == 0) atomicOr(status, DEV_BAD_NEIGHBOUR);
    const size_t bw = (size_t)d.NB * 9, rw = bw + 9;  // entries per atom
    const size_t aa = a * rw + bw + e, ab = a * rw + (size_t)bond * 9 + e;
    const size_t ba = ok ? b * rw + (size_t)sr * 9 + e : ab, bb = ok ? b * rw + bw + e : aa;
    const size_t o = a * bw + (size_t)bond * 9 + e;
    const int rows = d.Nqz * d.Nw;
    const size_t rp = d.NA * rw, op = d.NA * bw;  // row pitches
    for (int r = blockIdx.y; r < rows; r += gridDim.y) {
        const double2 *l = raw_l + r * rp, *g = raw_g + r * rp;
        const double2 x[2] = {l[ba], g[ba]}, y[2] = {l[bb], g[bb]}, z[2] = {l[aa], g[aa]}, u[2] = {l[ab], g[ab]};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            double2 v = make_double2(0.0, 0.0);
            if (ok)  // left to right
                v = make_double2(x[k].x - y[k].x - z[k].x + u[k].x, x[k].y - y[k].y - z[k].y + u[k].y);
            (k ? Dg : Dl)[r * op + o] = v;
        }
    }
}

// Adjoint: raw slot s < NB of atom a receives +g(a, s) (its D_ab term) and +g(b, s') (the D_ba term
// of the reverse bond); the self slot receives minus the sum of both over all of a's bonds. One thread per (atom,
// entry), four bonds of both types at a time.
__global__ void __launch_bounds__(kDcombThreads, 2)
dcomb_bwd_kernel(sse_dims d, const int32_t* __restrict__ nbr, const double2* __restrict__ g_l,
                 const double2* __restrict__ g_g, double2* __restrict__ r_l, double2* __restrict__ r_g,
                 unsigned* __restrict__ status) {
    extern __shared__ int sRev[];  // [atoms of this block][NB] reverse bond b * NB + s', -1: none
    const int nA = d.a_end - d.a_begin;
    const size_t c0 = blockIdx.x * (size_t)blockDim.x;
    const int la0 = (int)(c0 / 9), natoms = min(nA, (int)((c0 + blockDim.x - 1) / 9) + 1) - la0;
    const bool table = d.NB <= kDcombTableBonds;
    auto reverse = [&](int a, int s) {
        const int b = nbr[(size_t)a * d.NB + s];
        const int sr = (b >= 0 && b < d.NA) ? reverse_slot(nbr, d.NB, a, b) : -1;
        return sr < 0 ? (long long)-1 : (long long)b * d.NB + sr;
    };
    if (table) {
        for (int i = threadIdx.x; i < natoms * d.NB; i += blockDim.x)
            sRev[i] = (int)reverse(d.a_begin + la0 + i / d.NB, i % d.NB);
        __syncthreads();
    }
    const size_t col = c0 + threadIdx.x;
    if (col >= (size_t)nA * 9) return;
    const int la = (int)(col / 9), e = (int)(col % 9), a = d.a_begin + la;
    const size_t bw = (size_t)d.NB * 9, rw = bw + 9;
    const size_t go = a * bw + e, ro = a * rw + e;
    const int rows = d.Nqz * d.Nw;
    for (int r = blockIdx.y; r < rows; r += gridDim.y) {
        const double2* G[2] = {g_l + (size_t)r * d.NA * bw, g_g + (size_t)r * d.NA * bw};
        double2* R[2] = {r_l + (size_t)r * d.NA * rw + ro, r_g + (size_t)r * d.NA * rw + ro};
        double2 self[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
        for (int s0 = 0; s0 < d.NB; s0 += 4) {
            long long rev[4];
            double2 u[4][2], v[4][2];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int s = s0 + k;
                rev[k] = s >= d.NB ? -1 : table ? sRev[(la - la0) * d.NB + s] : reverse(a, s);
                if (s < d.NB && rev[k] < 0 && e == 0 && r == 0) atomicOr(status, DEV_BAD_NEIGHBOUR);
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (rev[k] < 0) continue;
                    u[k][t] = G[t][go + (size_t)s * 9];
                    v[k][t] = G[t][rev[k] * 9 + e];
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (s0 + k >= d.NB) continue;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    double2 sum = make_double2(0.0, 0.0);
                    if (rev[k] >= 0) {
                        sum = make_double2(u[k][t].x + v[k][t].x, u[k][t].y + v[k][t].y);
                        self[t].x -= sum.x;
                        self[t].y -= sum.y;
                    }
                    R[t][(size_t)(s0 + k) * 9] = sum;
                }
            }
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) R[t][bw] = self[t];
    }
}

// cols threads across, and as many blocks down the `steps` row steps as make eight per SM, rounded down: the adjoint's 1188
// blocks at FinFET are four full waves of two per SM (144 us), 1224 begin a fifth (152 us)
dim3 dcomb_grid(size_t cols, int steps) {
    const size_t gx = (cols + kDcombThreads - 1) / kDcombThreads;
    size_t gy = gx < 152 * 8 ? (size_t)152 * 8 / gx : 1;
    gy = gy < (size_t)steps ? gy : (size_t)steps;
    return dim3((unsigned)gx, (unsigned)(gy < 65535 ? gy : 65535));
}

}  // namespace

cudaError_t dcomb_fwd(const sse_dims& d, const int32_t* nbr, const double2* raw_l, const double2* raw_g,
                      double2* Dl, double2* Dg, unsigned* status, cudaStream_t st) {
    const dim3 grid = dcomb_grid((size_t)(d.a_end - d.a_begin) * d.NB * 9, d.Nqz * d.Nw);
    SSE_TIMED("dcomb_fwd_kernel", st,
              dcomb_fwd_kernel<<<grid, kDcombThreads, 0, st>>>(d, nbr, raw_l, raw_g, Dl, Dg, status));
    return cudaGetLastError();
}

cudaError_t dcomb_bwd(const sse_dims& d, const int32_t* nbr, const double2* g_l, const double2* g_g, double2* r_l,
                      double2* r_g, unsigned* status, cudaStream_t st) {
    const dim3 grid = dcomb_grid((size_t)(d.a_end - d.a_begin) * 9, d.Nqz * d.Nw);
    const int smem = d.NB <= kDcombTableBonds ? (kDcombThreads / 9 + 2) * d.NB * 4 : 0;
    SSE_TIMED("dcomb_bwd_kernel", st,
              dcomb_bwd_kernel<<<grid, kDcombThreads, smem, st>>>(d, nbr, g_l, g_g, r_l, r_g, status));
    return cudaGetLastError();
}

}  // namespace sse
