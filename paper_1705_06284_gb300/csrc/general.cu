// Non-cubic grids and complex fields (Sec. 2: the footnote on non-cubic
// data, and the remark that Eq. Jeong_gen applies to complex data through
// complex DFTs instead of real FFTs).
//
// Grid N_x x N_y x N_z (each 2^a 3^b), box L_x x L_y x L_z; mode m with
// components in FFT order, k = 2 pi (m_x/L_x, m_y/L_y, m_z/L_z), and
// V = L_x L_y L_z, N_pix = N_x N_y N_z in place of L^3 and N^3.  A mode is in
// bin b when t_b <= s(m) < t_{b+1}, s(m) = (m_x/L_x)^2 + (m_y/L_y)^2 +
// (m_z/L_z)^2 and t_b = (edge_b / 2 pi)^2, both evaluated on the host in
// FP64 in that order (one bin table per plan).  The field is complex (a real
// field is the case of zero imaginary parts), so nothing is halved:
//   D = DFT[delta] by three complex passes (FP32),
//   I_b = unnormalised inverse DFT of D on S_b (complex, one per bin),
//   B_abc = V^2/N_pix^3 sum_n I_a I_b I_c / (N_pix N_tri)   (complex),
//   P_b   = V/N_pix^2   sum_n I_b I_b / (N_pix |S_b|)        (complex),
// sums over the grid of FP32 products, as FP32 pairs per thread (48 bits) and
// in FP64 across threads, counts from
// FP64 count fields (real: every shell is symmetric under m -> -m modulo the
// grid) rounded to integers at plan time.  Closure is modulo the grid along
// each axis; unless FBS_FLAG_ALLOW_ALIASED is given every mode of every bin
// has |m_j| < N_j/4, where that is exact closure.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "fbs_internal.h"
#include "fft_core.cuh"

struct fbs_gplan {
    int n[3] = {0, 0, 0};
    double L[3] = {0, 0, 0};
    long long npix = 0;
    int nbins = 0;
    uint32_t flags = 0;
    std::vector<double> thr;
    std::vector<long long> shell;
    std::vector<int32_t> trip;
    std::vector<int64_t> ntri;
    double count_margin = 0;
    cudaStream_t stream = nullptr;
    fbs::FftFactors f[3]{};
    std::vector<void *> allocs;
    long long reserved = 0;
    short *d_bin = nullptr;
    float2 *d_tw[3] = {nullptr, nullptr, nullptr};
    double2 *d_tw64[3] = {nullptr, nullptr, nullptr};
    float2 *d_X = nullptr, *d_I = nullptr, *d_in = nullptr;
    int *d_items = nullptr;  // ntrip triplets then nbins (b, b, -1) pairs
    int64_t *d_ntri = nullptr;
    long long *d_shell = nullptr;
    double2 *d_part = nullptr, *d_sum = nullptr;
    double *d_B = nullptr, *d_P = nullptr;
    int G = 0;       // point chunks per item of the count sums
    int Gs = 0;      // point chunks per item of the product sums
    int2 *d_R = nullptr;  // largest |m_y| and |m_z| of every bin (-1: empty)

    void *dalloc(size_t bytes) {
        bytes = std::max<size_t>(bytes, 16);
        fbs::budget_reserve((long long)bytes);
        void *p = nullptr;
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            fbs::budget_release((long long)bytes);
            throw fbs::Failure{FBS_ERR_OOM, "general plan: device allocation failed"};
        }
        reserved += (long long)bytes;
        allocs.push_back(p);
        return p;
    }
};

namespace fbs {

namespace {

constexpr int kT = 256;

// In place along `axis` of an n0 x n1 x n2 array [i0][i1][i2]: every line of
// length n_axis transformed (DIR -1 forward, +1 unnormalised inverse).
template <typename T, int DIR>
__global__ void __launch_bounds__(kT) axis_fft_kernel(typename V2<T>::t *__restrict__ d, int n0, int n1, int n2,
                                                     int axis, FftFactors f, const typename V2<T>::t *__restrict__ tw,
                                                     int nl) {
    typedef typename V2<T>::t C;
    extern __shared__ __align__(16) unsigned char smraw[];
    C *a = reinterpret_cast<C *>(smraw);
    const int n = axis == 0 ? n0 : (axis == 1 ? n1 : n2);
    C *b = a + (size_t)nl * n;
    const long long nlines = (long long)n0 * n1 * n2 / n;
    const long long L0 = (long long)blockIdx.x * nl;
    // element j of line L: lines along z are contiguous; along y and x,
    // consecutive lines are consecutive elements (coalesced with the line
    // index fastest)
    auto elem = [&](long long L, int j) -> long long {
        if (axis == 2) return L * n2 + j;
        if (axis == 1) return (L / n2) * ((long long)n1 * n2) + (long long)j * n2 + L % n2;
        return (long long)j * n1 * n2 + L;
    };
    auto split = [&](int i, int &r, int &j) {
        if (axis == 2) {
            r = i / n;
            j = i - r * n;
        } else {
            j = i / nl;
            r = i - j * nl;
        }
    };
    for (int i = threadIdx.x; i < nl * n; i += blockDim.x) {
        int r, j;
        split(i, r, j);
        const long long L = L0 + r;
        a[(size_t)r * n + j] = L < nlines ? d[elem(L, j)] : C{T(0), T(0)};
    }
    __syncthreads();
    const C *res = smem_fft<T, DIR>(a, b, nl, n, f, tw);
    for (int i = threadIdx.x; i < nl * n; i += blockDim.x) {
        int r, j;
        split(i, r, j);
        const long long L = L0 + r;
        if (L < nlines) d[elem(L, j)] = res[(size_t)r * n + j];
    }
}

// FP32 passes of the field (DIR -1) and of every bin's field at once (DIR +1,
// bin blockIdx.y): lines of `axis` from src to dst (the same array, or the
// field and the spectrum).  The inverse runs x, y, z: the x pass takes the
// modes of the bin (the mask of Sec. 2 while loading) on the lines that hold
// any, |m_y| <= R.x and |m_z| <= R.y; the y pass lines with |m_z| <= R.y; rows
// outside are read as zero by the next pass, so nobody writes them.
template <int DIR>
__global__ void __launch_bounds__(kT) gfft_kernel(const float2 *src, float2 *dst, int n0, int n1, int n2, int axis,
                                                  FftFactors f, const float2 *__restrict__ tw, int nl,
                                                  const short *__restrict__ bin, const int2 *__restrict__ R) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float2 *a = reinterpret_cast<float2 *>(smraw);
    const int n = axis == 0 ? n0 : (axis == 1 ? n1 : n2);
    float2 *b = a + (size_t)nl * (n + 1);
    const int nlines = (int)((long long)n0 * n1 * n2 / n);
    const int L0 = blockIdx.x * nl;
    const int bn = blockIdx.y;
    int Ry = n1, Rz = n2;
    if (DIR > 0) {
        const int2 r = R[bn];
        Ry = r.x;
        Rz = r.y;
        if (Rz < 0) return;  // an empty bin's field stays zero
        dst += (long long)bn * n0 * n1 * n2;
        if (axis > 0) src = dst;
    }
    const auto mag = [](int j, int len) { return min(j, len - j); };
    // first element of line r of this CTA and the element step; ok: the line is transformed
    const auto start = [&](int r, long long &e, bool &ok) {
        const int L = L0 + r;
        ok = L < nlines;
        if (axis == 2) {
            e = (long long)L * n2;
        } else if (axis == 1) {
            const int z = L % n2;
            e = (long long)(L / n2) * n1 * n2 + z;
            ok = ok && mag(z, n2) <= Rz;
        } else {
            e = L;
            ok = ok && mag(L % n2, n2) <= Rz && mag(L / n2, n1) <= Ry;
        }
    };
    const long long step = axis == 2 ? 1 : axis == 1 ? n2 : (long long)n1 * n2;
    int any = 0;
    for (int i = threadIdx.x; i < nl * n; i += kT) {
        int r, j;
        if (axis == 2) {
            r = i / n;
            j = i - r * n;
        } else {
            j = i / nl;
            r = i - j * nl;
        }
        long long e;
        bool ok;
        start(r, e, ok);
        any |= ok;
        const bool in = ok && (axis == 0 || (axis == 1 ? mag(j, n1) <= Ry : mag(j, n2) <= Rz));
        e += j * step;
        float2 v = make_float2(0.f, 0.f);
        if (in && (DIR < 0 || axis > 0 || bin[e] == bn)) v = src[e];
        a[r * (n + 1) + j] = v;
    }
    if (!__syncthreads_or(any)) return;
    const float2 *res = smem_fft<float, DIR>(a, b, nl, n + 1, f, tw);
    for (int i = threadIdx.x; i < nl * n; i += kT) {
        int r, j;
        if (axis == 2) {
            r = i / n;
            j = i - r * n;
        } else {
            j = i / nl;
            r = i - j * nl;
        }
        long long e;
        bool ok;
        start(r, e, ok);
        if (ok) dst[e + j * step] = res[r * (n + 1) + j];
    }
}

__global__ void indicator_kernel(const short *__restrict__ bin, int b, double2 *__restrict__ Y, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        Y[i] = make_double2(bin[i] == b ? 1.0 : 0.0, 0.0);
}

__global__ void real_part_kernel(const double2 *__restrict__ Y, double *__restrict__ out, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = Y[i].x;
}

// part[item][chunk] = sum over the chunk's points of N_a N_b N_c (FP64 count
// fields, item = three rows).
__global__ void __launch_bounds__(kT) count_sum_kernel(const double *__restrict__ C, long long npix,
                                                       const int *__restrict__ items, double *__restrict__ part) {
    __shared__ double red[kT];
    const int it = blockIdx.y;
    const double *x = C + (long long)items[3 * it] * npix, *y = C + (long long)items[3 * it + 1] * npix,
                 *z = C + (long long)items[3 * it + 2] * npix;
    const long long c0 = npix * blockIdx.x / gridDim.x, c1 = npix * (blockIdx.x + 1) / gridDim.x;
    double s = 0.0;
    for (long long i = c0 + threadIdx.x; i < c1; i += blockDim.x) s += x[i] * y[i] * z[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = kT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(long long)it * gridDim.x + blockIdx.x] = red[0];
}

// A running sum of FP32 values kept as an unevaluated pair (the error of every
// addition is recovered exactly, Knuth's two-sum): 48 bits in FP32 operations,
// where an FP64 add costs 64 times as much.  The products' own roundings (2^-24)
// decide the error: B against 64 bits is off by the same 3.3e-7 to 6.0e-7 with
// FP64 adds and with pairs (six boxes of sides 27 to 128, 4 to 9 bins).
__device__ __forceinline__ void pair_add(float2 &s, float v) {
    const float t = __fadd_rn(s.x, v);
    const float w = __fsub_rn(t, s.x);
    const float e = __fadd_rn(__fsub_rn(s.x, __fsub_rn(t, w)), __fsub_rn(v, w));
    s.x = t;
    s.y = __fadd_rn(s.y, e);
}

// u v w, or u v, in FP32.
__device__ __forceinline__ float2 product(float2 u, float2 v, float2 w, bool three) {
    const float pr = u.x * v.x - u.y * v.y, pi = u.x * v.y + u.y * v.x;
    if (!three) return make_float2(pr, pi);
    return make_float2(pr * w.x - pi * w.y, pr * w.y + pi * w.x);
}

// part[item][chunk] = sum over the chunk's points of I_a I_b I_c (I_a I_b for
// items with c = -1): products in FP32, sums as FP32 pairs per thread and in
// FP64 across threads.  A CTA stages every bin at `tile` points, [point][bin],
// and a thread runs one item over every `slices`-th of them: lanes read
// different bins of one point (at most 16 bins: no bank conflicts).  Measured
// at 96 x 72 x 108, 8 bins (120 triplets): 524 -> 116 us against one pass
// over the fields per item with an FP64 add per point, which was bound by
// those adds (two a cycle per SM).
__global__ void __launch_bounds__(kT) ctriple_kernel(const float2 *__restrict__ I, long long npix, int nbins,
                                                     const int *__restrict__ items, int nitems, int slices, int tile,
                                                     double2 *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float2 *const sI = reinterpret_cast<float2 *>(smraw);  // [tile][nbins]
    __shared__ double2 red[kT];
    const int per = kT / slices, slice = threadIdx.x / per, it = blockIdx.y * per + threadIdx.x % per;
    const bool on = it < nitems;
    const int a = on ? items[3 * it] : 0, b = on ? items[3 * it + 1] : 0, c = on ? items[3 * it + 2] : 0;
    const long long c0 = npix * blockIdx.x / gridDim.x, c1 = npix * (blockIdx.x + 1) / gridDim.x;
    float2 sr = make_float2(0.f, 0.f), si = make_float2(0.f, 0.f);
    for (long long q0 = c0; q0 < c1; q0 += tile) {
        const int n = (int)min((long long)tile, c1 - q0);
        __syncthreads();
        for (int i = threadIdx.x; i < nbins * n; i += kT) {
            const int r = i / n, k = i - r * n;
            sI[k * nbins + r] = I[(long long)r * npix + q0 + k];
        }
        __syncthreads();
        if (!on) continue;
#pragma unroll 4
        for (int k = slice; k < n; k += slices) {
            const float2 p = product(sI[k * nbins + a], sI[k * nbins + b],
                                     c >= 0 ? sI[k * nbins + c] : make_float2(0.f, 0.f), c >= 0);
            pair_add(sr, p.x);
            pair_add(si, p.y);
        }
    }
    double2 mine = make_double2((double)sr.x + (double)sr.y, (double)si.x + (double)si.y);
    if (on && !(isfinite(sr.x) && isfinite(si.x))) {
        // past FP32's range (or an infinite or undefined product): again with FP64 adds
        mine = make_double2(0.0, 0.0);
        for (long long q0 = c0; q0 < c1; q0 += tile)
            for (long long q = q0 + slice; q < min(q0 + tile, c1); q += slices) {
                const float2 p = product(I[a * npix + q], I[b * npix + q],
                                         c >= 0 ? I[c * npix + q] : make_float2(0.f, 0.f), c >= 0);
                mine.x += p.x;
                mine.y += p.y;
            }
    }
    red[threadIdx.x] = mine;
    __syncthreads();
    if (slice || !on) return;
    double2 s = red[threadIdx.x];
    for (int k = 1; k < slices; ++k) {
        s.x += red[threadIdx.x + k * per].x;
        s.y += red[threadIdx.x + k * per].y;
    }
    part[(long long)it * gridDim.x + blockIdx.x] = s;
}

// out[item] = sum of its G chunk partials: one warp per item, a fixed order.
__global__ void __launch_bounds__(kT) reduce_chunks_kernel(const double2 *__restrict__ part, int G, int n,
                                                           double2 *__restrict__ out) {
    const int i = blockIdx.x * (kT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n) return;
    double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int g = lane; g < G; g += 32) {
        s.x += part[(long long)i * G + g].x;
        s.y += part[(long long)i * G + g].y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    if (lane == 0) out[i] = s;
}

__global__ void general_normalise_kernel(const double2 *__restrict__ sum, const int64_t *__restrict__ ntri,
                                         int ntrip, const long long *__restrict__ shell, int nbins, double cB,
                                         double cP, double npix, double *__restrict__ B, double *__restrict__ P) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < ntrip) {
        const double d = npix * (double)ntri[i];
        B[2 * i] = cB * sum[i].x / d;
        B[2 * i + 1] = cB * sum[i].y / d;
    }
    if (i < nbins) {
        const double2 s = sum[ntrip + i];
        const double d = npix * (double)shell[i];
        P[2 * i] = shell[i] > 0 ? cP * s.x / d : nan("");
        P[2 * i + 1] = shell[i] > 0 ? cP * s.y / d : nan("");
    }
}

template <typename C>
std::vector<C> twiddle_table(int n) {
    std::vector<C> t(n);
    for (int k = 0; k < n; ++k) {
        double ang = -2.0 * M_PI * (double)k / (double)n;
        double c = cos(ang), s = sin(ang);
        if (4 * k == n) { c = 0.0; s = -1.0; }
        if (2 * k == n) { c = -1.0; s = 0.0; }
        if (4 * k == 3 * n) { c = 0.0; s = 1.0; }
        t[k].x = (decltype(t[k].x))c;
        t[k].y = (decltype(t[k].y))s;
    }
    return t;
}

int grid_blocks(long long n) { return (int)std::min<long long>(4096, std::max<long long>(1, (n + kT - 1) / kT)); }

template <typename T, int DIR>
void transform3(fbs_gplan &g, typename V2<T>::t *d, typename V2<T>::t *const *tw) {
    for (int axis = 0; axis < 3; ++axis) {
        const int n = g.n[axis];
        const int nl = std::max(1, std::min(16, (int)((64 * 1024) / (2 * n * sizeof(typename V2<T>::t)))));
        const size_t sm = 2 * (size_t)nl * n * sizeof(typename V2<T>::t);
        auto k = axis_fft_kernel<T, DIR>;
        if (sm > 48 * 1024) allow_smem(k);
        const long long nlines = g.npix / n;
        k<<<(unsigned)((nlines + nl - 1) / nl), kT, sm, g.stream>>>(d, g.n[0], g.n[1], g.n[2], axis, g.f[axis],
                                                                   tw[axis], nl);
        FBS_CUDA(cudaGetLastError());
    }
}

// One FP32 pass over `nb` fields (gfft_kernel).
template <int DIR>
void gfft_pass(fbs_gplan &g, const float2 *src, float2 *dst, int axis, int nb) {
    const int n = g.n[axis];
    // lines per CTA: two buffers within 64 KB, at most 16 (coalesced rows of the x and y passes)
    const int nl = std::max(1, std::min(16, (int)((64 * 1024) / (2 * (n + 1) * sizeof(float2)))));
    const size_t sm = 2 * (size_t)nl * (n + 1) * sizeof(float2);
    auto k = gfft_kernel<DIR>;
    if (sm > 48 * 1024) allow_smem(k);
    const long long nlines = g.npix / n;
    k<<<dim3((unsigned)((nlines + nl - 1) / nl), nb), kT, sm, g.stream>>>(src, dst, g.n[0], g.n[1], g.n[2], axis,
                                                                         g.f[axis], g.d_tw[axis], nl, g.d_bin, g.d_R);
    FBS_CUDA(cudaGetLastError());
}

void gplan_build(fbs_gplan &g, const double *edges) {
    FBS_CUDA(cudaStreamCreateWithFlags(&g.stream, cudaStreamNonBlocking));
    for (int a = 0; a < 3; ++a) g.f[a] = make_factors(g.n[a]);
    g.npix = (long long)g.n[0] * g.n[1] * g.n[2];
    const int nb = g.nbins;
    g.thr.resize(nb + 1);
    for (int i = 0; i <= nb; ++i) {
        const double u = edges[i] / (2.0 * M_PI);
        g.thr[i] = u * u;
    }
    // bin table (host, FP64, the evaluation order of the definition)
    std::vector<short> bin((size_t)g.npix, -1);
    std::vector<int2> R(nb, make_int2(-1, -1));
    g.shell.assign(nb, 0);
    const bool aliased = (g.flags & FBS_FLAG_ALLOW_ALIASED) != 0;
    auto freq = [](int j, int n) { return j < (n + 1) / 2 ? j : j - n; };
    for (int i0 = 0; i0 < g.n[0]; ++i0)
        for (int i1 = 0; i1 < g.n[1]; ++i1)
            for (int i2 = 0; i2 < g.n[2]; ++i2) {
                const int m[3] = {freq(i0, g.n[0]), freq(i1, g.n[1]), freq(i2, g.n[2])};
                const double ux = m[0] / g.L[0], uy = m[1] / g.L[1], uz = m[2] / g.L[2];
                // rounded products (volatile: no fused multiply-add), summed in order
                volatile double xx = ux * ux, yy = uy * uy, zz = uz * uz;
                const double s = (xx + yy) + zz;
                if (s < g.thr[0] || s >= g.thr[nb]) continue;
                const int b = (int)(std::upper_bound(g.thr.begin(), g.thr.end(), s) - g.thr.begin()) - 1;
                if (!aliased)
                    for (int a = 0; a < 3; ++a)
                        if (4 * std::abs(m[a]) >= g.n[a])
                            throw Failure{FBS_ERR_ARG, "a bin holds a mode with |m_j| >= N_j/4 (closure would wrap); "
                                                       "lower the top edge or pass FBS_FLAG_ALLOW_ALIASED"};
                bin[((size_t)i0 * g.n[1] + i1) * g.n[2] + i2] = (short)b;
                R[b].x = std::max(R[b].x, std::abs(m[1]));
                R[b].y = std::max(R[b].y, std::abs(m[2]));
                ++g.shell[b];
            }
    g.d_bin = (short *)g.dalloc(bin.size() * sizeof(short));
    FBS_CUDA(cudaMemcpyAsync(g.d_bin, bin.data(), bin.size() * sizeof(short), cudaMemcpyHostToDevice, g.stream));
    g.d_R = (int2 *)g.dalloc(R.size() * sizeof(int2));
    FBS_CUDA(cudaMemcpyAsync(g.d_R, R.data(), R.size() * sizeof(int2), cudaMemcpyHostToDevice, g.stream));
    for (int a = 0; a < 3; ++a) {
        auto t32 = twiddle_table<float2>(g.n[a]);
        auto t64 = twiddle_table<double2>(g.n[a]);
        g.d_tw[a] = (float2 *)g.dalloc(t32.size() * sizeof(float2));
        g.d_tw64[a] = (double2 *)g.dalloc(t64.size() * sizeof(double2));
        FBS_CUDA(cudaMemcpyAsync(g.d_tw[a], t32.data(), t32.size() * sizeof(float2), cudaMemcpyHostToDevice, g.stream));
        FBS_CUDA(cudaMemcpyAsync(g.d_tw64[a], t64.data(), t64.size() * sizeof(double2), cudaMemcpyHostToDevice,
                                 g.stream));
        FBS_CUDA(cudaStreamSynchronize(g.stream));  // t32, t64 go out of scope
    }
    // count fields N_b (FP64) and the count sums of every candidate a <= b <= c
    std::vector<int> ne;
    for (int b = 0; b < nb; ++b)
        if (g.shell[b]) ne.push_back(b);
    std::vector<int> cand;
    for (size_t i = 0; i < ne.size(); ++i)
        for (size_t j = i; j < ne.size(); ++j)
            for (size_t k = j; k < ne.size(); ++k) cand.insert(cand.end(), {ne[i], ne[j], ne[k]});
    const int ncand = (int)cand.size() / 3;
    g.G = (int)std::max<long long>(1, std::min<long long>(64, g.npix / (16 * kT)));
    std::vector<double> sums(ncand, 0.0);
    if (ncand > 0) {
        AsyncBuf work((size_t)g.npix * sizeof(double2), g.stream, "general count scratch");
        AsyncBuf cf((size_t)nb * g.npix * sizeof(double), g.stream, "general count fields");
        for (int b : ne) {
            indicator_kernel<<<grid_blocks(g.npix), kT, 0, g.stream>>>(g.d_bin, b, work.as<double2>(), g.npix);
            FBS_CUDA(cudaGetLastError());
            transform3<double, +1>(g, work.as<double2>(), g.d_tw64);
            real_part_kernel<<<grid_blocks(g.npix), kT, 0, g.stream>>>(work.as<double2>(),
                                                                       cf.as<double>() + (long long)b * g.npix, g.npix);
            FBS_CUDA(cudaGetLastError());
        }
        AsyncBuf d_cand(cand.size() * sizeof(int), g.stream, "general count scratch");
        AsyncBuf part((size_t)ncand * g.G * sizeof(double), g.stream, "general count scratch");
        FBS_CUDA(cudaMemcpyAsync(d_cand.ptr, cand.data(), cand.size() * sizeof(int), cudaMemcpyHostToDevice, g.stream));
        for (int c0 = 0; c0 < ncand; c0 += 65535) {
            const int nc = std::min(65535, ncand - c0);
            count_sum_kernel<<<dim3(g.G, nc), kT, 0, g.stream>>>(cf.as<double>(), g.npix, d_cand.as<int>() + 3 * c0,
                                                                part.as<double>() + (long long)c0 * g.G);
            FBS_CUDA(cudaGetLastError());
        }
        std::vector<double> h((size_t)ncand * g.G);
        FBS_CUDA(cudaMemcpyAsync(h.data(), part.ptr, h.size() * sizeof(double), cudaMemcpyDeviceToHost, g.stream));
        FBS_CUDA(cudaStreamSynchronize(g.stream));
        for (int i = 0; i < ncand; ++i)
            for (int c = 0; c < g.G; ++c) sums[i] += h[(size_t)i * g.G + c];
    }
    for (int i = 0; i < ncand; ++i) {
        const double v = sums[i] / (double)g.npix, r = nearbyint(v);
        g.count_margin = std::max(g.count_margin, fabs(v - r));
        if (fabs(v - r) > 0.25) throw Failure{FBS_ERR_NUMERIC, "count sum " + std::to_string(v) + " is not an integer"};
        if (r <= 0) continue;
        g.trip.insert(g.trip.end(), {cand[3 * i], cand[3 * i + 1], cand[3 * i + 2]});
        g.ntri.push_back((int64_t)r);
    }
    const int ntrip = (int)g.ntri.size();
    std::vector<int> items(g.trip.begin(), g.trip.end());
    for (int b = 0; b < nb; ++b) items.insert(items.end(), {b, b, -1});
    const int nitems = ntrip + nb;
    g.d_items = (int *)g.dalloc(items.size() * sizeof(int));
    g.d_ntri = (int64_t *)g.dalloc(std::max<size_t>(1, g.ntri.size()) * sizeof(int64_t));
    g.d_shell = (long long *)g.dalloc(nb * sizeof(long long));
    FBS_CUDA(cudaMemcpyAsync(g.d_items, items.data(), items.size() * sizeof(int), cudaMemcpyHostToDevice, g.stream));
    if (ntrip)
        FBS_CUDA(cudaMemcpyAsync(g.d_ntri, g.ntri.data(), g.ntri.size() * sizeof(int64_t), cudaMemcpyHostToDevice,
                                 g.stream));
    FBS_CUDA(cudaMemcpyAsync(g.d_shell, g.shell.data(), nb * sizeof(long long), cudaMemcpyHostToDevice, g.stream));
    g.d_X = (float2 *)g.dalloc((size_t)g.npix * sizeof(float2));
    g.d_in = (float2 *)g.dalloc((size_t)g.npix * sizeof(float2));
    g.d_I = (float2 *)g.dalloc((size_t)nb * g.npix * sizeof(float2));
    FBS_CUDA(cudaMemsetAsync(g.d_I, 0, (size_t)nb * g.npix * sizeof(float2), g.stream));  // empty bins stay zero
    // about four CTAs per SM over the items' blocks, partials within 64 MB
    g.Gs = (int)std::max<long long>(1, std::min<long long>({(g.npix + 255) / 256, 608, (4LL << 20) / nitems}));
    g.d_part = (double2 *)g.dalloc((size_t)nitems * g.Gs * sizeof(double2));
    g.d_sum = (double2 *)g.dalloc((size_t)nitems * sizeof(double2));
    g.d_B = (double *)g.dalloc(std::max<size_t>(1, 2 * (size_t)ntrip) * sizeof(double));
    g.d_P = (double *)g.dalloc(2 * (size_t)nb * sizeof(double));
    FBS_CUDA(cudaStreamSynchronize(g.stream));  // items goes out of scope
}

void gplan_run(fbs_gplan &g, const float *field) {
    const size_t bytes = (size_t)g.npix * sizeof(float2);
    // read in place where the kernels can: this device's memory or managed memory
    cudaPointerAttributes a;
    bool dev = false;
    if (cudaPointerGetAttributes(&a, field) == cudaSuccess) {
        int here = 0;
        FBS_CUDA(cudaGetDevice(&here));
        dev = (a.type == cudaMemoryTypeDevice && a.device == here) || a.type == cudaMemoryTypeManaged;
    } else {
        cudaGetLastError();
    }
    const float2 *in = reinterpret_cast<const float2 *>(field);
    if (!dev || (reinterpret_cast<uintptr_t>(field) & 7)) {
        FBS_CUDA(cudaMemcpyAsync(g.d_in, field, bytes, cudaMemcpyDefault, g.stream));
        in = g.d_in;
    }
    gfft_pass<-1>(g, in, g.d_X, 0, 1);
    gfft_pass<-1>(g, g.d_X, g.d_X, 1, 1);
    gfft_pass<-1>(g, g.d_X, g.d_X, 2, 1);
    const int nb = g.nbins, ntrip = (int)g.ntri.size();
    for (int axis = 0; axis < 3; ++axis) gfft_pass<+1>(g, g.d_X, g.d_I, axis, nb);
    const int nitems = ntrip + nb;
    // threads per item: as many slices of the points as the items leave
    int slices = 1;
    while (slices < kT / 32 && 2 * slices * nitems <= kT) slices *= 2;
    const int per = kT / slices;
    const int tile = (int)std::max<long long>(1, std::min<long long>(256, 32 * 1024 / (nb * 8)));
    const size_t sm = (size_t)tile * nb * sizeof(float2);  // at most 32 KB
    const int ny = (nitems + per - 1) / per;
    for (int y0 = 0; y0 < ny; y0 += 65535) {
        const int c0 = y0 * per;
        ctriple_kernel<<<dim3(g.Gs, std::min(65535, ny - y0)), kT, sm, g.stream>>>(
            g.d_I, g.npix, nb, g.d_items + 3 * (size_t)c0, nitems - c0, slices, tile, g.d_part + (long long)c0 * g.Gs);
        FBS_CUDA(cudaGetLastError());
    }
    reduce_chunks_kernel<<<(nitems + kT / 32 - 1) / (kT / 32), kT, 0, g.stream>>>(g.d_part, g.Gs, nitems, g.d_sum);
    FBS_CUDA(cudaGetLastError());
    const double V = g.L[0] * g.L[1] * g.L[2], np = (double)g.npix;
    const int nmax = std::max(ntrip, nb);
    general_normalise_kernel<<<(nmax + 255) / 256, 256, 0, g.stream>>>(
        g.d_sum, g.d_ntri, ntrip, g.d_shell, nb, V * V / (np * np * np), V / (np * np), np, g.d_B, g.d_P);
    FBS_CUDA(cudaGetLastError());
}

}  // namespace

}  // namespace fbs

using namespace fbs;

extern "C" {

fbs_status fbs_gplan_create(fbs_gplan **out, const int32_t *n, const double *L, const double *edges, int nbins,
                            uint32_t flags) {
    if (!out) return FBS_ERR_ARG;
    *out = nullptr;
    if (!n || !L || !edges || nbins < 1 || nbins > 4096) {
        set_error("fbs_gplan_create: bad argument");
        return FBS_ERR_ARG;
    }
    for (int a = 0; a < 3; ++a)
        if (n[a] < 2 || n[a] > 512 || !(L[a] > 0.0)) {
            set_error("fbs_gplan_create: grid sides must be 2..512 and box sides positive");
            return FBS_ERR_ARG;
        }
    for (int i = 0; i < nbins; ++i)
        if (!(edges[i] >= 0.0) || !(edges[i + 1] > edges[i])) {
            set_error("fbs_gplan_create: edges must be non-negative and ascending");
            return FBS_ERR_ARG;
        }
    fbs_gplan *g = new fbs_gplan();
    for (int a = 0; a < 3; ++a) {
        g->n[a] = n[a];
        g->L[a] = L[a];
    }
    g->nbins = nbins;
    g->flags = flags;
    try {
        gplan_build(*g, edges);
    } catch (const Failure &f) {
        set_error(f.msg);
        fbs_gplan_free(g);
        return f.status;
    }
    *out = g;
    return FBS_OK;
}

int fbs_gplan_num_triplets(const fbs_gplan *g) { return g ? (int)g->ntri.size() : FBS_ERR_ARG; }

fbs_status fbs_gplan_triplets(const fbs_gplan *g, int32_t *abc, int64_t *ntri) {
    if (!g) return FBS_ERR_ARG;
    if (abc && !g->trip.empty()) memcpy(abc, g->trip.data(), g->trip.size() * sizeof(int32_t));
    if (ntri && !g->ntri.empty()) memcpy(ntri, g->ntri.data(), g->ntri.size() * sizeof(int64_t));
    return FBS_OK;
}

fbs_status fbs_gplan_shells(const fbs_gplan *g, int64_t *sizes) {
    if (!g || !sizes) return FBS_ERR_ARG;
    for (int b = 0; b < g->nbins; ++b) sizes[b] = g->shell[b];
    return FBS_OK;
}

fbs_status fbs_gplan_bispectrum(fbs_gplan *g, const float *field, double *B, double *P) {
    if (!g || !field) {
        set_error("fbs_gplan_bispectrum: NULL argument");
        return FBS_ERR_ARG;
    }
    try {
        gplan_run(*g, field);
        const size_t nt = g->ntri.size();
        if (B && nt) FBS_CUDA(cudaMemcpyAsync(B, g->d_B, 2 * nt * sizeof(double), cudaMemcpyDefault, g->stream));
        if (P) FBS_CUDA(cudaMemcpyAsync(P, g->d_P, 2 * (size_t)g->nbins * sizeof(double), cudaMemcpyDefault, g->stream));
        FBS_CUDA(cudaStreamSynchronize(g->stream));
    } catch (const Failure &f) {
        set_error(f.msg);
        return f.status;
    }
    return FBS_OK;
}

void fbs_gplan_free(fbs_gplan *g) {
    if (!g) return;
    if (g->stream) cudaStreamSynchronize(g->stream);
    for (void *p : g->allocs) cudaFree(p);
    budget_release(g->reserved);
    if (g->stream) cudaStreamDestroy(g->stream);
    cudaGetLastError();
    delete g;
}

}  // extern "C"
