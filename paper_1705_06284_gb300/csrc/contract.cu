// Real-space product sums of the FFT estimator (Sec. 2, Eqs. Jeong_gen,
// Jeong_BI) on CUDA cores, the FP64 count sums that give the exact triangle
// counts, and the FP64 normalisation epilogue (Eqs. Jeong_PS, Jeong_BI).
//
// Work is grouped by "outer pairs": for a bispectrum one of a triplet's three
// pairs, with the third bin as the inner row; for a trispectrum the pair
// (c, d) with the product of the pair (a, b).  A pair's product is formed once
// per point and reused for all its inner rows.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <array>
#include <map>
#include <utility>
#include <vector>

#include "fbs_internal.h"
#include "pair_cover.h"

namespace fbs {

static constexpr int kCThreads = 512;     // 16 warps, one CTA per SM
static constexpr int kGroupItems = 4096;  // items per CTA at most (12 bytes of shared memory each)

__device__ __forceinline__ void lds_points(const float *row, int lane, int k, float2 &u, float2 &w) {
    const float4 v = reinterpret_cast<const float4 *>(row)[lane + 32 * k];
    u = make_float2(v.x, v.y);
    w = make_float2(v.z, v.w);
}

// Stage I[b][q0 .. q0 + chunk) of every bin (asynchronous copies; the ragged
// tail zero-padded by plain stores), one copy group.
template <int chunk>
__device__ __forceinline__ void stage_chunk(const float *I, long long bin_stride, long long npts, int nbins,
                                            long long q0, float *dst) {
    constexpr int n4 = chunk / 4;
    for (int i = threadIdx.x; i < nbins * n4; i += kCThreads) {
        const int b = i / n4, k = i % n4;
        const long long q = q0 + 4LL * k;
        const float *src = I + b * bin_stride + q;
        if (q + 3 < npts) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(dst + 4 * i)),
                         "l"(src)
                         : "memory");
        } else {
            float4 v;
            v.x = q + 0 < npts ? src[0] : 0.f;
            v.y = q + 1 < npts ? src[1] : 0.f;
            v.z = q + 2 < npts ? src[2] : 0.f;
            v.w = 0.f;
            reinterpret_cast<float4 *>(dst)[i] = v;
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// ------------------------------------------------------------------ FP32
// grid.x: point-range blocks; grid.y: blocks of pair groups; grid.z: fields.
// A warp holds the products of four outer pairs (one group) at PPL points per
// lane and runs over the group's inner rows (single bins, or products of two
// for quadruplets) two at a time: a row's values are loaded once and
// multiplied into up to four items, and the lane sums of eight items are
// reduced together (nine shuffles).  A chunk's FP32 sums go to shared memory,
// one word per item, and are added to the FP64 totals by all threads: FP64
// adds are scarce here (two a cycle per SM), and one lane's add per item, as
// the one-pair form had it, costs as much as the products.  The next chunk's
// fields are copied while this one's are used, and groups go to free warps,
// the longest first.
// What bounds it: shared-memory loads (69% of the cycles at 256^3, 32 linear
// bins: 16 wavefronts per row and 16 per factor of a pair, for 512 points).
// Measured against one pair at a time with one FP64 add per item: 256^3, 32
// linear bins 4.89 -> 1.57 ms, 16 fields of 96^3, 24 bins 2.97 -> 0.96 ms,
// 108^3, 10 log bins, triplets and quadruplets 460 -> 181 us.
// bin_stride and the fields' base are multiples of 16 bytes (even grids).
template <int PPL, bool QUAD>
__global__ void __launch_bounds__(kCThreads, 1) contract_fp32_kernel(
    const float *__restrict__ I, long long bin_stride, long long npts, int nbins, const FpGroup *__restrict__ groups,
    const FpRow *__restrict__ rows, const int *__restrict__ iout, const int4 *__restrict__ blocks, int nitems_total,
    double *__restrict__ part, int part_rows, int first) {
    constexpr int chunk = 32 * PPL;
    extern __shared__ __align__(16) unsigned char smraw[];
    // field blockIdx.z of a batch: its bins follow the previous fields' in I
    I += (long long)blockIdx.z * nbins * bin_stride;
    const int4 blk = blocks[blockIdx.y];  // groups [x, y), first item z, items w
    const int nloc = blk.w;
    float *const sI = reinterpret_cast<float *>(smraw);  // two stages of nbins x chunk
    double *const acc = reinterpret_cast<double *>(sI + 2 * nbins * chunk);
    float *const tmp = reinterpret_cast<float *>(acc + nloc);
    for (int i = threadIdx.x; i < nloc; i += kCThreads) acc[i] = 0.0;

    // contiguous point range of this CTA, in whole chunks
    const long long nchunks = (npts + chunk - 1) / chunk;
    const long long c0 = nchunks * blockIdx.x / gridDim.x;
    const long long c1 = nchunks * (blockIdx.x + 1) / gridDim.x;
    const int lane = threadIdx.x & 31;
    __shared__ int next_group;
    if (threadIdx.x == 0) next_group = 0;

    if (c0 < c1) stage_chunk<chunk>(I, bin_stride, npts, nbins, c0 * chunk, sI);
    for (long long ch = c0; ch < c1; ++ch) {
        const float *const st = sI + ((ch - c0) & 1) * nbins * chunk;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // this chunk is staged; the other stage's readers and tmp's are done
        if (ch + 1 < c1)
            stage_chunk<chunk>(I, bin_stride, npts, nbins, (ch + 1) * chunk, sI + ((ch + 1 - c0) & 1) * nbins * chunk);
        // groups, longest first, to the warps that are free
        for (;;) {
            int g = lane == 0 ? atomicAdd(&next_group, 1) : 0;
            g = blk.x + __shfl_sync(0xffffffffu, g, 0);
            if (g >= blk.y) break;
            const FpGroup *G = groups + g;
            float2 pp[4][PPL / 2];
            const float *const rb = st + G->b[0] * chunk;
#pragma unroll
            for (int k = 0; k < PPL / 4; ++k) {
                float2 u0, u1;
                lds_points(rb, lane, k, u0, u1);
#pragma unroll
                for (int j = 0; j < 4; ++j) {  // pairs of a group mostly share their first bin
                    float2 x0 = u0, x1 = u1, w0, w1;
                    if (j > 0 && G->b[j] != G->b[0]) lds_points(st + G->b[j] * chunk, lane, k, x0, x1);
                    lds_points(st + G->c[j] * chunk, lane, k, w0, w1);
                    pp[j][2 * k] = __fmul2_rn(x0, w0);
                    pp[j][2 * k + 1] = __fmul2_rn(x1, w1);
                }
            }
            const int4 *const rp = reinterpret_cast<const int4 *>(rows);
            const int e1 = G->row1;
            int4 n0 = rp[G->row0], n1 = rp[G->row0 + 1];
            for (int e = G->row0; e < e1; e += 2) {  // a group has an even number of rows
                const int4 r[2] = {n0, n1};
                n0 = rp[min(e + 2, e1 - 2)];
                n1 = rp[min(e + 3, e1 - 1)];
                float s[2][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 v[PPL / 2];
#pragma unroll
                    for (int k = 0; k < PPL / 4; ++k) lds_points(st + r[h].x * chunk, lane, k, v[2 * k], v[2 * k + 1]);
                    if (QUAD) {
#pragma unroll
                        for (int k = 0; k < PPL / 4; ++k) {
                            float2 w0, w1;
                            lds_points(st + r[h].y * chunk, lane, k, w0, w1);
                            v[2 * k] = __fmul2_rn(v[2 * k], w0);
                            v[2 * k + 1] = __fmul2_rn(v[2 * k + 1], w1);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {  // items that do not exist are formed too: no branches
                        float2 t = __fmul2_rn(pp[j][0], v[0]);
#pragma unroll
                        for (int k = 1; k < PPL / 2; ++k) t = __ffma2_rn(pp[j][k], v[k], t);
                        s[h][j] = t.x + t.y;
                    }
                }
                // eight sums over 32 lanes: row (lane bit 4), pair (bits 3, 2)
                const bool hi = lane & 16, p1 = lane & 8, p0 = lane & 4;
                float a[4], b[2];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    a[j] = (hi ? s[1][j] : s[0][j]) + __shfl_xor_sync(0xffffffffu, hi ? s[0][j] : s[1][j], 16);
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    b[j] = (p1 ? a[2 + j] : a[j]) + __shfl_xor_sync(0xffffffffu, p1 ? a[j] : a[2 + j], 8);
                float t = (p0 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, p0 ? b[0] : b[1], 4);
                t += __shfl_xor_sync(0xffffffffu, t, 2);
                t += __shfl_xor_sync(0xffffffffu, t, 1);
                const int mask = hi ? r[1].z : r[0].z, first = hi ? r[1].w : r[0].w, j = (lane >> 2) & 3;
                if ((lane & 3) == 0 && (mask >> j & 1)) tmp[first + __popc(mask & ((1 << j) - 1))] = t;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) next_group = 0;  // read again past the next barrier
        for (int i = threadIdx.x; i < nloc; i += kCThreads) acc[i] += (double)tmp[i];  // the same thread every time
    }
    double *row = part + ((long long)blockIdx.z * part_rows + blockIdx.x) * nitems_total;
    for (int i = threadIdx.x; i < nloc; i += kCThreads) {
        double &d = row[iout[blk.z + i]];
        d = first ? acc[i] : d + acc[i];
    }
}

// ------------------------------------------------------------------ reduce
// Sums of a level's partials, one launch: blocks [0, nblk[0]) and [nblk[0],
// nblk[0] + nblk[1]) take 32 items each of the two segments, out[map[i]] =
// scale * sum_r part[r * ld + i] over the rows the contraction wrote; the rest
// take one bin each, sumsq[pbin[b]] = scale * sum_r sq[b][r].  Eight threads
// share an item's rows (one thread per item and 304 rows, most of them zero,
// took 40 to 50 us of dependent loads for any size).  Every sum has a fixed
// order.  Field blockIdx.y of a batch: partials sfs, outputs ofs further on.
// NORM (a plan of one level, whose items are the plan's): the estimates too,
// which saves a launch of 6 us that waits for this one.
struct ReduceSeg {
    const double *part;
    const int *map;
    double *out;
    int n, ld, rows;
    long long sfs, ofs;
};
// The estimates of a sum over the whole plan (NormArgs):
// B = V^2/N_pix^3 num/(N_pix N_tri), P = V/N_pix^2 sumsq/(N_pix |S_b|)
// (NaN for empty shells), T = V^3/N_pix^4 qnum/(N_pix N_quad).
struct NormArgs {
    const int64_t *ntri;
    const double *nq;
    const long long *shell;
    double *B, *P, *T;  // outputs (any may be null)
    double L;
    int N, ntrip, nquad, nbins;
    const int *err;       // this evaluation's wait-timeout code (or null)
    int *sticky, *h_err;  // kept until the host reports it, and its pinned host copy
};
__device__ __forceinline__ double norm_B(const NormArgs &a, double num, int i) {
    const double V = a.L * a.L * a.L, npix = (double)a.N * a.N * a.N, cB = V * V / (npix * npix * npix);
    return cB * num / (npix * (double)a.ntri[i]);
}
__device__ __forceinline__ double norm_P(const NormArgs &a, double sumsq, int b) {
    const double V = a.L * a.L * a.L, npix = (double)a.N * a.N * a.N, cP = V / (npix * npix);
    return a.shell[b] > 0 ? cP * sumsq / (npix * (double)a.shell[b]) : nan("");
}
__device__ __forceinline__ double norm_T(const NormArgs &a, double num, int i) {
    const double V = a.L * a.L * a.L, npix = (double)a.N * a.N * a.N;
    const double cT = V * V * V / (npix * npix * npix * npix);
    return cT * num / (npix * a.nq[i]);
}
// A tensor-core wait gave up: the sums are incomplete.  One thread of the
// grid (`one`) keeps the code and copies it to the host.
__device__ __forceinline__ bool norm_bad(const NormArgs &a, bool one) {
    const bool bad = a.err && *a.err;
    if (one && a.sticky) {
        const int v = bad ? *a.err : *a.sticky;
        if (bad) *a.sticky = v;
        if (a.h_err) *(volatile int *)a.h_err = v;
    }
    return bad;
}

struct ReduceArgs {
    ReduceSeg seg[2];
    int nblk[2];
    const double *sq;
    const int *pbin;
    double *sumsq;
    int sqrows;
    long long sfs, ofs;
    double scale;
    NormArgs norm;
};

template <bool NORM>
__global__ void __launch_bounds__(256) level_reduce_kernel(const __grid_constant__ ReduceArgs a) {
    __shared__ double red[256];
    const int tid = threadIdx.x;
    int blk = blockIdx.x;
    const long long f = blockIdx.y;
    bool bad = false;
    if (NORM) {
        bad = norm_bad(a.norm, blk == 0 && f == 0 && tid == 0);
        if (blk == 0 && a.norm.P)
            for (int b = tid; b < a.norm.nbins; b += 256)
                if (a.norm.shell[b] <= 0) a.norm.P[f * a.norm.nbins + b] = nan("");
    }
    const int which = blk < a.nblk[0] ? 0 : blk < a.nblk[0] + a.nblk[1] ? 1 : 2;
    if (which < 2) {
        const ReduceSeg &g = a.seg[which];
        if (which) blk -= a.nblk[0];
        const int i = 32 * blk + (tid & 31), ty = tid >> 5;
        const double *part = g.part + blockIdx.y * g.sfs;
        double s = 0.0;
        if (i < g.n) {
#pragma unroll 4
            for (int r = ty; r < g.rows; r += 8) s += part[(long long)r * g.ld + i];
        }
        red[tid] = s;
        __syncthreads();
        if (ty == 0 && i < g.n) {
            for (int k = 1; k < 8; ++k) s += red[tid + 32 * k];
            const int o = g.map ? g.map[i] : i;
            s *= a.scale;
            g.out[blockIdx.y * g.ofs + o] = s;
            if (NORM && !which && a.norm.B) a.norm.B[f * a.norm.ntrip + o] = bad ? nan("") : norm_B(a.norm, s, o);
            if (NORM && which && a.norm.T) a.norm.T[o] = bad ? nan("") : norm_T(a.norm, s, o);
        }
        return;
    }
    blk -= a.nblk[0] + a.nblk[1];
    if (a.pbin[blk] < 0) return;
    const double *sq = a.sq + blockIdx.y * a.sfs + (long long)blk * a.sqrows;
    double s = 0.0;
#pragma unroll 4
    for (int r = tid; r < a.sqrows; r += 256) s += sq[r];
    red[tid] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (tid < w) red[tid] += red[tid + w];
        __syncthreads();
    }
    if (tid == 0) {
        const int b = a.pbin[blk];
        s = a.scale * red[0];
        a.sumsq[blockIdx.y * a.ofs + b] = s;
        if (NORM && a.norm.P) a.norm.P[f * a.norm.nbins + b] = norm_P(a.norm, s, b);
    }
}

// ------------------------------------------------------------------ normalise
// Estimates of a plan of several levels, after the last level's reduction.
// Field blockIdx.y of a batch: its sums and outputs follow the previous fields'.
__global__ void normalise_kernel(const __grid_constant__ NormArgs a, const double *__restrict__ tnum,
                                 const double *__restrict__ qnum, const double *__restrict__ sumsq) {
    const long long f = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool bad = norm_bad(a, i == 0 && f == 0);
    if (a.B && i < a.ntrip) a.B[f * a.ntrip + i] = bad ? nan("") : norm_B(a, tnum[f * a.ntrip + i], i);
    if (a.P && i < a.nbins) a.P[f * a.nbins + i] = norm_P(a, sumsq[f * a.nbins + i], i);
    if (a.T && i < a.nquad) a.T[i] = bad ? nan("") : norm_T(a, qnum[i], i);
}

// ------------------------------------------------------------------ connected trispectrum
// Per-shell moments of the spectrum box (the forward output): for bin b
// (blockIdx.y), over the rows (m_x, m_y) of its sub-box |m_j| <= R_b that
// this one of gridDim.x chunks takes,
//   S2 = sum |D|^2, S4 = sum |D|^4 over the shell's modes,
//   Z4 = sum D^4 over its self-conjugate modes (m = -m mod N, D real there).
// The box holds mz >= 0 only: a mode with 0 < mz < N/2 stands for itself and
// its conjugate at -mz (weight 2); the planes mz = 0 and mz = N/2 hold both.
// One partial per (bin, chunk, moment), from a fixed-shape block reduction.
// A warp takes a row, rows are dealt out round robin (the widest shell holds
// most of the modes) and rows outside the shell cost one test.  Measured at
// 162, 9 logarithmic bins: 65 -> 22 us against 16 chunks of modes, each
// found by 64-bit divisions.
__global__ void __launch_bounds__(256) shell_moments_kernel(const float2 *__restrict__ box, BoxGeom bg,
                                                            const BinGeom *__restrict__ gb,
                                                            double *__restrict__ part) {
    __shared__ double red[3][256];
    const int b = blockIdx.y, N = bg.N;
    const BinGeom g = gb[b];
    double s2 = 0.0, s4 = 0.0, z4 = 0.0;
    if (!g.empty) {
        const int lane = threadIdx.x & 31, rows = g.Db * g.Db, step = gridDim.x * 8;
        for (int r0 = blockIdx.x * 8 + (threadIdx.x >> 5); r0 < rows; r0 += 4 * step) {
            const float2 *row[4];  // four rows in flight
            int r2[4];             // at most N^2 / 2; -1: no row
            bool sc[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * step, jx = r / g.Db, jy = r - jx * g.Db;
                const int mx = box_freq(jx, g.Db, N), my = box_freq(jy, g.Db, N);
                r2[q] = r < rows ? mx * mx + my * my : -1;
                row[q] = box + ((long long)box_index(mx, bg.D) * bg.D + box_index(my, bg.D)) * bg.Dz;
                sc[q] = (mx == 0 || 2 * mx == -N) && (my == 0 || 2 * my == -N);
            }
            for (int mz = lane; mz < g.Dzb; mz += 32) {
                const bool plane = mz == 0 || 2 * mz == N;
                const double w = plane ? 1.0 : 2.0;
                float2 d[4];
                bool on[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const long long s = (long long)r2[q] + mz * mz;
                    d[q] = make_float2(0.f, 0.f);
                    on[q] = r2[q] >= 0 && s >= g.thr_lo && s < g.thr_hi;
                    if (on[q]) d[q] = row[q][mz];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (!on[q]) continue;
                    const double a2 = (double)d[q].x * d[q].x + (double)d[q].y * d[q].y;
                    s2 += w * a2;
                    s4 += w * a2 * a2;
                    if (sc[q] && plane) z4 += (double)d[q].x * d[q].x * d[q].x * d[q].x;
                }
            }
        }
    }
    red[0][threadIdx.x] = s2;
    red[1][threadIdx.x] = s4;
    red[2][threadIdx.x] = z4;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 3) part[((long long)b * gridDim.x + blockIdx.x) * 3 + threadIdx.x] = red[threadIdx.x][0];
}

// Connected trispectrum of each closed quadruplet (a <= b <= c <= d): the sum
// over its closed quadruples with the paired ones (m_i + m_j = 0 mod N for
// two of the modes) left out, by inclusion-exclusion over the three pairings:
//   a = b < c = d : paired sum S2_a S2_c
//   a = b = c = d : 3 S2^2 - 3 S4 + Z4
//   otherwise     : 0,
// Tc = V^3/N_pix^4 (qnum/N_pix - paired sum) / N_conn, N_conn the unpaired
// count (plan time).  NaN where a wait timed out or no unpaired quadruple is left.
//
// Every block first adds up the chunks of all moments, a warp per sum in a
// fixed order, into shared memory (one thread per quadruplet adding them from
// global memory was a chain of up to 3 x 16 dependent loads and adds).
__global__ void __launch_bounds__(256) connected_kernel(const double *__restrict__ qnum, const int *__restrict__ quad,
                                                        const double *__restrict__ nconn, int nquad,
                                                        const double *__restrict__ mom_part, int nbins, double L,
                                                        int N, double *__restrict__ Tc, const int *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char smraw[];
    double *const mom = reinterpret_cast<double *>(smraw);  // [bin][moment]
    for (int m = threadIdx.x >> 5; m < 3 * nbins; m += 8) {
        const double *src = mom_part + (long long)(m / 3) * kMomChunks * 3 + m % 3;
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < kMomChunks / 32; ++j) s += src[3 * ((threadIdx.x & 31) + 32 * j)];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) mom[m] = s;
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nquad) return;
    const double V = L * L * L, npix = (double)N * N * N;
    const double cT = V * V * V / (npix * npix * npix * npix);
    const int a = quad[4 * i], b = quad[4 * i + 1], c = quad[4 * i + 2], d = quad[4 * i + 3];
    double paired = 0.0;
    if (a == b && c == d) {
        const double s2 = mom[3 * a];
        paired = a != c ? s2 * mom[3 * c] : 3.0 * s2 * s2 - 3.0 * mom[3 * a + 1] + mom[3 * a + 2];
    }
    const bool bad = (err && *err) || !(nconn[i] > 0.0);
    Tc[i] = bad ? nan("") : cT * (qnum[i] / npix - paired) / nconn[i];
}

void launch_connected(Plan &p, double *d_Tc) {
    KTimer tm(p, KC_REDUCE);
    dim3 grid(kMomChunks, p.nbins);
    shell_moments_kernel<<<grid, 256, 0, p.stream>>>(p.d_box, p.box, p.d_geom, p.d_mom_part);
    FBS_CUDA(cudaGetLastError());
    const int nq = (int)p.nquad.size();
    if (nq == 0) return;
    const size_t sm = (size_t)p.nbins * 3 * sizeof(double);  // at most 128 bins
    connected_kernel<<<(nq + 255) / 256, 256, sm, p.stream>>>(
        p.d_qnum, p.d_quadtab, p.d_nconn, nq, p.d_mom_part, p.nbins, p.L, p.N, d_Tc,
        p.precision != FBS_PREC_FP32 ? tc_error_flag(p) : nullptr);
    FBS_CUDA(cudaGetLastError());
}

// ------------------------------------------------------------------ counts (FP64)
// den[item] = sum over the octant 0 <= x,y,z <= N/2 of w(x)w(y)w(z) prod N_i,
// w(v) = 1 for v in {0, N/2} and 2 otherwise (the reflections m_j -> -m_j map
// the octant onto the whole grid).  items: arity bins per item (3 or 4).
// kCntChunk: octant points staged per pass (fewer for many field rows).
__global__ void __launch_bounds__(256) count_kernel(const double *__restrict__ noct, int nbins, int H,
                                                    const int *__restrict__ items, int arity,
                                                    int nitems, int grp_items,
                                                    double *__restrict__ part, int kCntChunk) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int it0 = blockIdx.y * grp_items;
    const int nloc = min(grp_items, nitems - it0);
    if (nloc <= 0) return;
    double *acc = reinterpret_cast<double *>(smraw);
    double *sN = acc + grp_items;
    double *sw = sN + (size_t)nbins * kCntChunk;
    for (int i = threadIdx.x; i < nloc; i += blockDim.x) acc[i] = 0.0;
    const long long npts = (long long)H * H * H;
    const long long nchunks = (npts + kCntChunk - 1) / kCntChunk;
    const long long c0 = nchunks * blockIdx.x / gridDim.x;
    const long long c1 = nchunks * (blockIdx.x + 1) / gridDim.x;
    const int Nh = H - 1;  // N/2
    for (long long ch = c0; ch < c1; ++ch) {
        const long long q0 = ch * kCntChunk;
        __syncthreads();
        for (int i = threadIdx.x; i < nbins * kCntChunk; i += blockDim.x) {
            int b = i / kCntChunk, k = i - b * kCntChunk;
            long long q = q0 + k;
            sN[i] = q < npts ? noct[(long long)b * npts + q] : 0.0;
        }
        for (int k = threadIdx.x; k < kCntChunk; k += blockDim.x) {
            long long q = q0 + k;
            double w = 0.0;
            if (q < npts) {
                int z = (int)(q % H), y = (int)((q / H) % H), x = (int)(q / ((long long)H * H));
                w = (x == 0 || x == Nh ? 1.0 : 2.0) * (y == 0 || y == Nh ? 1.0 : 2.0) *
                    (z == 0 || z == Nh ? 1.0 : 2.0);
            }
            sw[k] = w;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nloc; i += blockDim.x) {
            const int *it = items + (long long)(it0 + i) * arity;
            const double *ra = sN + (size_t)it[0] * kCntChunk;
            const double *rb = sN + (size_t)it[1] * kCntChunk;
            const double *rc = sN + (size_t)it[2] * kCntChunk;
            double s = 0.0;
            if (arity == 3) {
#pragma unroll 8
                for (int k = 0; k < kCntChunk; ++k) s = fma(sw[k] * ra[k], rb[k] * rc[k], s);
            } else {
                const double *rd = sN + (size_t)it[3] * kCntChunk;
#pragma unroll 8
                for (int k = 0; k < kCntChunk; ++k) s = fma(sw[k] * ra[k] * rb[k], rc[k] * rd[k], s);
            }
            acc[i] += s;
        }
    }
    __syncthreads();
    double *row = part + (long long)blockIdx.x * nitems + it0;
    for (int i = threadIdx.x; i < nloc; i += blockDim.x) row[i] = acc[i];
}

// ------------------------------------------------------------------ host wrappers
static int num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        FBS_CUDA(cudaGetDevice(&dev));
        FBS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    }
    return sms;
}

int contract_blocks() { return 2 * num_sms(); }

// Groups of up to four outer pairs for the FP32 contraction, chosen so that
// the pairs of a group share inner rows (each row's values are loaded once per
// group): the next pair in order, then those of the following ones that add
// the fewest rows.  Blocks of groups bound the items of a CTA.
static void build_fp32_job(Plan &p, const TaskList &t, bool quads, FpJob &job) {
    const int nb = p.nbins;
    std::map<int, std::vector<std::pair<int, int>>> pairs;  // outer pair -> (inner row key, output)
    if (quads) {
        for (int i = 0; i < t.npairs; ++i)
            for (int e = t.pstart[i]; e < t.pstart[i + 1]; ++e)
                pairs[t.pb[i] * nb + t.pc[i]].push_back({t.ia[e] * nb + t.ib[e], t.iout[e]});
    } else {
        // each triplet by one of its three pairs: fewer pairs, more rows in common
        std::vector<std::array<int, 3>> trip;
        std::vector<int> out;
        for (int i = 0; i < t.npairs; ++i)
            for (int e = t.pstart[i]; e < t.pstart[i + 1]; ++e) {
                std::array<int, 3> tr = {t.ia[e], t.pb[i], t.pc[i]};
                std::sort(tr.begin(), tr.end());
                trip.push_back(tr);
                out.push_back(t.iout[e]);
            }
        const std::vector<int> key = cover_triplet_pairs(nb, trip);
        for (size_t i = 0; i < trip.size(); ++i)
            pairs[key[i]].push_back({trip[i][0] + trip[i][1] + trip[i][2] - key[i] / nb - key[i] % nb, out[i]});
    }
    std::vector<int> id;  // inner row keys -> bit
    std::vector<int> bit_of((size_t)nb * nb, -1);
    struct Outer {
        int key;
        std::vector<std::pair<int, int>> items;
        std::vector<unsigned long long> bits;
    };
    std::vector<Outer> outer;
    for (auto &kv : pairs) {
        std::sort(kv.second.begin(), kv.second.end());
        for (const auto &it : kv.second)
            if (bit_of[it.first] < 0) {
                bit_of[it.first] = (int)id.size();
                id.push_back(it.first);
            }
    }
    const size_t words = (id.size() + 63) / 64;
    for (const auto &kv : pairs)
        for (size_t i0 = 0; i0 < kv.second.size(); i0 += kGroupItems) {  // (a pair with more items: several times)
            const size_t i1 = std::min(kv.second.size(), i0 + kGroupItems);
            Outer o{kv.first, {kv.second.begin() + i0, kv.second.begin() + i1},
                    std::vector<unsigned long long>(words, 0ULL)};
            for (const auto &it : o.items) o.bits[bit_of[it.first] >> 6] |= 1ULL << (bit_of[it.first] & 63);
            outer.push_back(std::move(o));
        }
    std::vector<FpGroup> groups;
    std::vector<FpRow> rows;
    std::vector<int> iout;
    std::vector<int4> blocks;
    std::vector<char> used(outer.size(), 0);
    job.maxloc = 0;
    int4 blk = make_int4(0, 0, 0, 0);
    const auto close = [&] {
        const int n = (int)groups.size() - blk.x;
        if (n > 0) {
            // two tasks per warp at least: groups split by rows (six at least, an
            // even number) where there are fewer; the longest first
            const int want = 2 * kCThreads / 32, parts = n >= want ? 1 : (want + n - 1) / n;
            std::vector<FpGroup> tasks;
            for (int i = blk.x; i < (int)groups.size(); ++i) {
                FpGroup g = groups[i];
                const int last = g.row1, len = std::max(6, ((last - g.row0 + parts - 1) / parts + 1) / 2 * 2);
                while (g.row0 < last) {
                    g.row1 = std::min(last, g.row0 + len);
                    tasks.push_back(g);
                    g.row0 = g.row1;
                }
            }
            std::stable_sort(tasks.begin(), tasks.end(), [](const FpGroup &u, const FpGroup &v) {
                return u.row1 - u.row0 > v.row1 - v.row0;
            });
            groups.resize(blk.x);
            groups.insert(groups.end(), tasks.begin(), tasks.end());
            blk.y = (int)groups.size();
            job.maxloc = std::max(job.maxloc, blk.w);
            blocks.push_back(blk);
        }
        blk = make_int4((int)groups.size(), 0, (int)iout.size(), 0);
    };
    for (size_t s = 0; s < outer.size(); ++s) {
        if (used[s]) continue;
        std::vector<int> pick{(int)s};
        used[s] = 1;
        std::vector<unsigned long long> bits = outer[s].bits;
        size_t n = outer[s].items.size();
        while (pick.size() < 4) {
            int best = -1, score = -1000000, seen = 0;
            for (size_t k = s + 1; k < outer.size() && seen < 48; ++k) {
                if (used[k] || n + outer[k].items.size() > (size_t)kGroupItems) continue;
                ++seen;
                int both = 0;
                for (size_t w = 0; w < words; ++w) both += __builtin_popcountll(bits[w] & outer[k].bits[w]);
                const int sc = 2 * both - (int)outer[k].items.size();  // rows shared less rows added
                if (sc > score) {
                    score = sc;
                    best = (int)k;
                }
            }
            if (best < 0) break;
            pick.push_back(best);
            used[best] = 1;
            n += outer[best].items.size();
            for (size_t w = 0; w < words; ++w) bits[w] |= outer[best].bits[w];
        }
        if (blk.w > 0 && blk.w + n > (size_t)kGroupItems) close();
        // the bin that most of the pairs have is their first factor, those pairs lead
        int common = 0, most = 0;
        for (int k : pick)
            for (int bin : {outer[k].key / nb, outer[k].key % nb}) {
                int cnt = 0;
                for (int m : pick) cnt += outer[m].key / nb == bin || outer[m].key % nb == bin;
                if (cnt > most) {
                    most = cnt;
                    common = bin;
                }
            }
        const auto has = [&](int k) { return outer[k].key / nb == common || outer[k].key % nb == common; };
        std::stable_partition(pick.begin(), pick.end(), has);
        FpGroup g{};
        for (int j = 0; j < 4; ++j) {  // empty places of a group repeat its first pair, without items
            const int key = outer[pick[j < (int)pick.size() ? j : 0]].key;
            const bool swap = key / nb != common && key % nb == common;
            g.b[j] = swap ? key % nb : key / nb;
            g.c[j] = swap ? key / nb : key % nb;
        }
        std::map<int, std::array<int, 4>> by_row;  // inner row -> outputs of the four pairs (-1: none)
        for (size_t j = 0; j < pick.size(); ++j)
            for (const auto &it : outer[pick[j]].items) {
                auto at = by_row.emplace(it.first, std::array<int, 4>{-1, -1, -1, -1});
                at.first->second[j] = it.second;
            }
        g.row0 = (int)rows.size();
        for (const auto &kv : by_row) {
            FpRow r{};
            r.x = quads ? kv.first / nb : kv.first;
            r.y = quads ? kv.first % nb : 0;
            r.first = blk.w;
            for (int j = 0; j < 4; ++j)
                if (kv.second[j] >= 0) {
                    r.mask |= 1 << j;
                    iout.push_back(kv.second[j]);
                    ++blk.w;
                }
            rows.push_back(r);
        }
        if ((rows.size() - g.row0) % 2) rows.push_back(FpRow{});  // no items
        g.row1 = (int)rows.size();
        groups.push_back(g);
    }
    close();
    TableUpload up(p);
    job.d_groups = up.put(groups);
    job.d_rows = up.put(rows);
    job.d_iout = up.put(iout);
    job.d_blocks = up.put(blocks);
    up.wait();
    job.nblocks = (int)blocks.size();
    job.built = true;
}

// Tables of a level's FP32 contraction, built when the plan first has a use for
// them: its creation, or the first FP32 evaluation of one made for another
// precision.
void prepare_fp32(Plan &p, bool trip, bool quads) {
    if (trip && !p.fpt.built && p.ttask.nitems > 0) build_fp32_job(p, p.ttask, false, p.fpt);
    if (quads && !p.fpq.built && p.qtask.nitems > 0) build_fp32_job(p, p.qtask, true, p.fpq);
}

void launch_contract_fp32(Plan &p, const float *islab, long long npts, long long slab_stride,
                          bool quads, int nf, double *part_batch) {
    const TaskList &t = quads ? p.qtask : p.ttask;
    if (t.nitems == 0) return;
    prepare_fp32(p, !quads, quads);
    const FpJob &job = quads ? p.fpq : p.fpt;
    // 512 points per chunk; fewer where that leaves SMs without a chunk or two
    // stages do not fit
    int ppl = 16;
    const auto smem = [&] { return (size_t)job.maxloc * 12 + 16 + (size_t)p.nbins * 256 * ppl; };
    while (ppl > 4 && (smem() > 220 * 1024 || npts * nf < 32LL * ppl * num_sms())) ppl /= 2;
    const size_t sm = smem();
    KTimer tm(p, quads ? KC_QUAD : KC_CONTRACT);
    // one CTA per SM over the fields and blocks, or two rounds of them where one
    // would leave more than 3% of the SMs idle
    const int per = nf * job.nblocks, one = num_sms() / per;
    const int G = (num_sms() - one * per) * 33 > num_sms() ? std::max(1, 2 * num_sms() / per) : one;
    dim3 grid(std::min(G, p.part_blocks), job.nblocks, nf);
    const auto run = [&](auto k) {
        allow_smem(k);
        k<<<grid, kCThreads, sm, p.stream>>>(islab, slab_stride, npts, p.nbins, job.d_groups, job.d_rows, job.d_iout,
                                             job.d_blocks, t.nitems,
                                             part_batch ? part_batch : quads ? p.d_qpart : p.d_tpart, p.part_blocks,
                                             p.first_slab);
    };
    (quads ? p.qrows : p.trows) = (int)grid.x;
    if (quads) {
        if (ppl == 16) run(contract_fp32_kernel<16, true>);
        else if (ppl == 8) run(contract_fp32_kernel<8, true>);
        else run(contract_fp32_kernel<4, true>);
    } else {
        if (ppl == 16) run(contract_fp32_kernel<16, false>);
        else if (ppl == 8) run(contract_fp32_kernel<8, false>);
        else run(contract_fp32_kernel<4, false>);
    }
    FBS_CUDA(cudaGetLastError());
}

// A level's sums over its M^3 grid -> sums over the N^3 grid ((N/M)^3), into
// the root's global arrays: triplet and quadruplet sums through the level's
// output maps, sums of squares of the bins whose P this level provides.
void launch_level_reduce(Plan &p, bool quads) {
    Plan &R = p.root();
    launch_level_reduce_batch(p, quads, 1, p.fused_active ? p.d_fpart : p.d_tpart, p.d_sumsq_part, R.d_tnum,
                              R.d_sumsq, R.d_B, R.d_P);
}

static NormArgs norm_args(Plan &p, bool quads, double *B, double *P) {
    const bool tc = p.precision != FBS_PREC_FP32;
    return NormArgs{p.d_ntri, p.d_nquad, p.d_shell, B, P, quads ? p.d_T : nullptr, p.L, p.N, (int)p.ntri.size(),
                    quads ? (int)p.nquad.size() : 0, p.nbins, tc ? tc_error_flag(p) : nullptr,
                    tc ? tc_sticky_flag(p) : nullptr, p.h_err};
}

// The sums of nf fields (partials tpart: per field part_blocks rows; sumsq
// partials: per field nbins blocks) into tnum[nf][ntrip], sumsq[nf][nbins];
// the estimates of a plan of one level too.
void launch_level_reduce_batch(Plan &p, bool quads, int nf, const double *tpart, const double *sq,
                               double *tnum, double *sumsq, double *B, double *P) {
    Plan &R = p.root();
    KTimer tm(p, KC_REDUCE);
    const double r = (double)R.N / (double)p.M;
    ReduceArgs a{};
    a.scale = r * r * r;
    const int n = p.ttask.nitems, m = quads ? p.qtask.nitems : 0;
    const int ld = p.fused_active ? n + m : n;
    a.seg[0] = ReduceSeg{tpart, p.d_gtrip, tnum, n, ld, p.trows, (long long)p.part_blocks * ld,
                         (long long)R.ntri.size()};
    a.nblk[0] = (n + 31) / 32;
    if (p.fused_active) a.seg[1] = ReduceSeg{p.d_fpart + n, p.d_gquad, R.d_qnum, m, ld, p.trows, 0, 0};
    else a.seg[1] = ReduceSeg{p.d_qpart, p.d_gquad, R.d_qnum, m, m, p.qrows, 0, 0};
    a.nblk[1] = (m + 31) / 32;
    a.sq = sq;
    a.pbin = p.d_pbin;
    a.sumsq = sumsq;
    a.sqrows = p.M * zstage_row_groups(p.M);
    a.sfs = (long long)p.nbins * a.sqrows;
    a.ofs = R.nbins;
    const dim3 grid(a.nblk[0] + a.nblk[1] + p.nbins, nf);
    if (R.levels.size() == 1) {
        a.norm = norm_args(R, quads, B, P);
        level_reduce_kernel<true><<<grid, 256, 0, p.stream>>>(a);
    } else {
        level_reduce_kernel<false><<<grid, 256, 0, p.stream>>>(a);
    }
    FBS_CUDA(cudaGetLastError());
}

void launch_normalise(Plan &p, bool quads) { launch_normalise_batch(p, quads, 1, p.d_tnum, p.d_sumsq, p.d_B, p.d_P); }

// B[nf][ntrip], P[nf][nbins] from tnum[nf][ntrip], sumsq[nf][nbins]; T (single
// field only).  A plan of one level has them from its reduction.
void launch_normalise_batch(Plan &p, bool quads, int nf, const double *tnum, const double *sumsq, double *B,
                            double *P) {
    if (p.levels.size() != 1) {
        KTimer tm(p, KC_REDUCE);
        const NormArgs a = norm_args(p, quads, B, P);
        const int n_all = std::max(std::max(a.ntrip, a.nquad), a.nbins);
        normalise_kernel<<<dim3((n_all + 255) / 256, nf), 256, 0, p.stream>>>(a, tnum, p.d_qnum, sumsq);
        FBS_CUDA(cudaGetLastError());
    }
    if (p.precision != FBS_PREC_FP32 && tc_sticky_flag(p) && p.h_err) {
        FBS_CUDA(cudaEventRecord(p.ev_err, p.stream));
        p.err_recorded = true;
    }
}

// Count sums for `nitems` items (arity bins each, indices into the nbins
// octant fields), result den[nitems] (device).
void launch_count_contraction(Plan &p, const double *noct, int nbins_all, int, const int *d_items,
                              int nitems, int arity, double *d_den) {
    if (nitems == 0) return;
    const int H = p.M / 2 + 1;  // count fields are on the evaluation grid's octant
    int grp = 4096, kCntChunk = 128;
    auto smem = [&] { return (size_t)grp * 8 + (size_t)nbins_all * kCntChunk * 8 + kCntChunk * 8; };
    while (smem() > 200 * 1024 && kCntChunk > 16) kCntChunk /= 2;
    while (smem() > 200 * 1024 && grp > 256) grp /= 2;
    const size_t sm = smem();
    if (sm > 220 * 1024) throw Failure{FBS_ERR_ARG, "too many field rows for the count kernel"};
    const int ngrp = (nitems + grp - 1) / grp;
    const int blocks = 2 * num_sms();
    AsyncBuf pbuf((size_t)blocks * nitems * sizeof(double), p.stream, "count partials");
    double *part = pbuf.as<double>();
    KTimer tm(p, KC_COUNT);
    allow_smem(count_kernel);
    dim3 g(blocks, ngrp);
    count_kernel<<<g, 256, sm, p.stream>>>(noct, nbins_all, H, d_items, arity, nitems, grp, part, kCntChunk);
    FBS_CUDA(cudaGetLastError());
    ReduceArgs a{};
    a.scale = 1.0;
    a.seg[0] = ReduceSeg{part, nullptr, d_den, nitems, nitems, blocks, 0, 0};
    a.nblk[0] = (nitems + 31) / 32;
    level_reduce_kernel<false><<<a.nblk[0], 256, 0, p.stream>>>(a);
    FBS_CUDA(cudaGetLastError());
}

}  // namespace fbs
