// Diagonal-resolved trispectrum: the closed quadruples of a quadruplet
// (a, b, c, d) split by the shell D of their diagonal q = k1 + k2.
//
// With F_ab(q) = sum_{m1 + m2 = q} D(m1) D(m2) over S_a x S_b, the closed
// quadruples with k1 + k2 = q in S_D sum to
//   num_D = sum_{q in S_D} F_ab(q) F_cd(-q) = sum_{q in S_D} Re[F_ab(q) conj F_cd(q)]
// (a real field has F_cd(-q) = conj F_cd(q)).  F_ab is the forward DFT of the
// product of two shell fields of Eq. delta_nr on the evaluation grid M (the
// Kronecker-delta identity of Sec. 2 applied to the pair): DFT_M[I_a I_b] =
// M^3 F_ab on every q that can close (M is above R_a + R_b + R_c + R_d).  So
// one forward transform per distinct pair (a, b) and one shell-restricted
// Gram product per (quadruplet, D) over the half spectrum box (weight 2 off
// the planes q_z = 0 and M/2, whose conjugate points are stored themselves).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "fbs_internal.h"

namespace fbs {

namespace {

// Block (task, quadruplet group): partial sums part[task][q] = w sum_e
// Re[F_u conj F_v] over the task's half-box modes, F rows u, v of quadruplet q
// (rows of FA, then of FB).  The modes' values of every row are staged as FP64
// in shared memory, [mode][row], so each is converted once for all the
// quadruplets, and a thread spends two FP64 FMAs per mode and quadruplet:
// what bounds it (two FP64 lanes a cycle per SM: 90 us of FMAs for 123
// quadruplets at 96^3 and 8 shells).  One block per (shell, quadruplet),
// converting both rows and multiplying by the weight for every mode, took
// 1,313 us there, most of it in the blocks of the largest shells; now 155 us.
constexpr int kDiagThreads = 128;

template <int kDiagQuads>  // quadruplets per thread
__global__ void __launch_bounds__(kDiagThreads) diag_gram_kernel(
    const float2 *__restrict__ FA, int na, const float2 *__restrict__ FB, int rows, long long per,
    const int2 *__restrict__ uv, int nq, const int *__restrict__ idx, const DiagTask *__restrict__ tasks, int chunk,
    double *__restrict__ part) {
    extern __shared__ double2 sF[];  // [chunk][rows]
    const DiagTask t = tasks[blockIdx.x];
    int2 me[kDiagQuads];
    double s[kDiagQuads];
#pragma unroll
    for (int j = 0; j < kDiagQuads; ++j) {
        const int q = (blockIdx.y * kDiagQuads + j) * kDiagThreads + threadIdx.x;
        me[j] = q < nq ? uv[q] : make_int2(0, 0);
        s[j] = 0.0;
    }
    for (int e0 = t.e0; e0 < t.e1; e0 += chunk) {
        const int n = min(chunk, t.e1 - e0);
        __syncthreads();
        for (int i = threadIdx.x; i < rows * n; i += kDiagThreads) {
            const int r = i / n, k = i - r * n;
            const float2 v = (r < na ? FA + r * per : FB + (r - na) * per)[idx[e0 + k]];
            sF[k * rows + r] = make_double2((double)v.x, (double)v.y);
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < n; ++k) {
#pragma unroll
            for (int j = 0; j < kDiagQuads; ++j) {
                const double2 x = sF[k * rows + me[j].x], y = sF[k * rows + me[j].y];
                s[j] = fma(x.y, y.y, fma(x.x, y.x, s[j]));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < kDiagQuads; ++j) {
        const int q = (blockIdx.y * kDiagQuads + j) * kDiagThreads + threadIdx.x;
        if (q < nq) part[(long long)blockIdx.x * nq + q] = (double)t.w * s[j];
    }
}

// out[qout[q] * nd + D] = scale * sum of the shell's task partials: eight
// threads to a quadruplet, in a fixed order.
__global__ void __launch_bounds__(256) diag_reduce_kernel(const double *__restrict__ part, int nq,
                                                          const int *__restrict__ tstart, int nd,
                                                          const int *__restrict__ qout, double scale,
                                                          double *__restrict__ out) {
    __shared__ double red[256];
    const int q = 32 * blockIdx.x + (threadIdx.x & 31), ty = threadIdx.x >> 5, D = blockIdx.y;
    double s = 0.0;
    if (q < nq) {
#pragma unroll 4
        for (int t = tstart[D] + ty; t < tstart[D + 1]; t += 8) s += part[(long long)t * nq + q];
    }
    red[threadIdx.x] = s;
    __syncthreads();
    if (ty || q >= nq) return;
    for (int k = 1; k < 8; ++k) s += red[threadIdx.x + 32 * k];
    out[(long long)qout[q] * nd + D] = scale * s;
}

// T_D = cT num_D / N_D (NaN where no closed quadruple has its diagonal in D).
__global__ void diag_normalise_kernel(const double *__restrict__ num, const double *__restrict__ cnt, long long n,
                                      double cT, double *__restrict__ TD) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) TD[i] = cnt[i] > 0.0 ? cT * num[i] / cnt[i] : nan("");
}

}  // namespace

// Quadruplets uv (rows of FA, then of FB: FB == FA's continuation has nb = 0)
// over the tasks of every shell; part: ntasks x nq doubles.
void launch_diag_gram(Plan &p, const float2 *FA, int na, const float2 *FB, int nb, long long per, const int2 *d_uv,
                      int nq, const int *d_idx, const DiagTask *d_tasks, int ntasks, const int *d_tstart, int nd,
                      const int *d_qout, double scale, double *part, double *out) {
    if (nq == 0 || nd == 0) return;
    const int rows = na + nb;
    // about 64 KB of staged modes (three CTAs per SM), one mode at least
    const int chunk = std::max(1, std::min(64, (64 * 1024) / (rows * (int)sizeof(double2))));
    const size_t sm = (size_t)chunk * rows * sizeof(double2);
    if (sm > 220 * 1024) throw Failure{FBS_ERR_ARG, "too many pair spectra in a group"};
    if (ntasks > 0) {
        const int per_block = kDiagThreads * (nq > kDiagThreads ? 2 : 1);
        const auto kernel = nq > kDiagThreads ? diag_gram_kernel<2> : diag_gram_kernel<1>;
        allow_smem(kernel);
        dim3 grid(ntasks, (nq + per_block - 1) / per_block);
        kernel<<<grid, kDiagThreads, sm, p.stream>>>(FA, na, FB, rows, per, d_uv, nq, d_idx, d_tasks, chunk,
                                                               part);
        FBS_CUDA(cudaGetLastError());
    }
    diag_reduce_kernel<<<dim3((nq + 31) / 32, nd), 256, 0, p.stream>>>(part, nq, d_tstart, nd, d_qout, scale, out);
    FBS_CUDA(cudaGetLastError());
}

void launch_diag_normalise(Plan &p, const double *num, const double *cnt, long long n, double cT, double *TD) {
    if (n == 0) return;
    diag_normalise_kernel<<<(unsigned)((n + 255) / 256), 256, 0, p.stream>>>(num, cnt, n, cT, TD);
    FBS_CUDA(cudaGetLastError());
}

}  // namespace fbs
