// Shared-operand tensor-core contraction (tcgen05, BF16x3, sm_103a): the
// product sums of Eqs. Jeong_BI and Jeong_gen with both MMA operands formed
// once in shared memory.
//
// A row is the product of two shell fields, or one of them; every item
// (triplet or quadruplet) is the inner product over the points of two rows.
// Row r's FP32 value v at a point is split into BF16 hi = bf16(v) and lo =
// bf16(v - hi).  Operand A stacks 64 rows' hi and lo parts on M = 128,
// operand B puts the hi and lo parts of up to 256 rows on N (two tiles of 256),
// so one MMA per 16 points and tile forms hi*hi, hi*lo, lo*hi and lo*lo, and
// the two operands are views of the same rows in shared memory: a product
// that stands on both sides is formed once.
//
// A producer lane owns two points and forms 16 rows (a unit) of them: its
// shell-field values are read along the points (conflict free, a factor that
// consecutive rows share once), eight rows' BF16 parts of one point are one
// 16-byte store, and the operands are M- and N-major (rows contiguous).  The
// lane = row layout of an operand in tensor memory (contract_tc_kernel) reads
// both factors of every product from shared memory row by row instead, four
// warp instructions where this takes one.  Which K index a point has is free
// as long as both operands agree: point 2l + i of a step is K row 32 i + l, so
// that the stores of eight neighbouring lanes fall into eight K rows of one
// swizzle atom (no bank conflicts).
//
// Roles (one CTA per SM, mbarrier hand-offs, every wait bounded): one thread
// streams 64-point steps of every shell field with TMA; kProd warps form
// units, taken in turn from the steps in flight; one thread issues the MMAs;
// eight warps add the accumulators (tensor memory, FP32, 1,024 points) to
// compensated FP32 sums per item while the MMAs of the next 1,024 points go to
// the other half of tensor memory (one tile of B; two tiles take turns).
//
// What bounds it: shared memory, where four operand stages fit.  The trispectrum
// pass of 16 log bins at 256^3 takes 1,386 cycles per 64-point step, of which the
// producers' and the accumulator warps' wavefronts fill 76% and the MMAs' operand
// reads (128 + N rows of 32 bytes per 16 points) most of the rest; the tensor
// pipe is active 42%.  Layouts of many rows have two or three stages: there the
// wavefronts fill 49 to 54%, the tensor pipe is active 28 to 33% and the rest is
// hand-off (the large levels of 192^3 x 48 and 384^3 x 29 linear bins).  Measured
// against the tensor-memory kernel (CUDA events): 512^3, 16 log bins, triplets
// and quadruplets 12.7 -> 8.5 ms; 64 log bins, triplets 7.7 -> 4.6 ms (its M =
// 384 level, 18 bins and 32 pairs, 3.8 -> 1.8 ms, its M = 288 level, 57 bins
// and 144 pairs, 3.3 -> 2.7 ms); 384^3, 29 linear bins 3.0 -> 2.75 ms; 162^3, 9
// log bins 358 -> 162 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <array>
#include <vector>

#include "fbs_internal.h"
#include "gram_rows.h"
#include "pair_cover.h"
#include "tc_ptx.cuh"

namespace fbs {

namespace {

constexpr int kPts = 64;                // points per step (LDS.64: two per lane)
constexpr int kProd = 20;               // producer warps
constexpr int kEpi0 = kProd, kEpi = 8;  // accumulator warps (warp mod 4 = lane quarter, two to a quarter)
constexpr int kMma = kProd + kEpi, kLoad = kMma + 1;
constexpr int kGThreads = (kLoad + 1) * 32;
constexpr int kMaxRing = 16;
constexpr int kAtomBytes = 8192;        // 32 rows, hi and lo, x 64 points
constexpr int kFlush = 1024 / kPts;     // steps between accumulator reads

// One CTA group: its units with any row, B's first chunk and chunks, its items
// (in the order of GramTable).
struct GramGroup {
    int unit0, nunits, jb0, nbch, item0, nitems, table;
};

// Which factors the eight rows of a chunk load: rows i = 0..7 are x[i] y[i] ...
enum {
    kRowsAny = 0,     // 16 loads
    kRowsStars,       // x[0] for rows 0..3, x[4] for rows 4..7: 10
    kRowsBlock,       // the same, and y[0..3] for both halves: 6
    kRowsSingle       // ... are y[i] alone: 8
};

// One unit (16 rows, chunks 2 unit and 2 unit + 1) that has any row: the byte
// offsets of its rows' factors in a field stage.  block: both chunks are
// kRowsBlock with the same y[0..3] (8 loads for 16 rows).
struct GramUnit {
    uint32_t y[16], x[16];
    int unit, kind[2], block;
};

// The units of every group are kernel arguments: read with a warp-uniform
// index they come through the constant port into uniform registers, and a
// factor's load is one LDS of lane address + uniform offset.  (Read from shared
// memory, the offsets cost as many vector instructions as the products: 4,503
// warp instructions per 64-point step at 256^3, 16 log bins, against 3,204.)
template <int CAP>
struct GramUnits {
    GramUnit u[CAP];
};

// Per group: the B rows that every A row meets in an item, and the first item
// of every accumulator warp.  Items are numbered in the order in which the
// accumulator warps visit them (warp, B chunk, row of the lane's four, lane), so
// that a warp's sums are consecutive in shared memory.
struct GramTable {
    unsigned mask[kGramARows][kGramBRows / 32];
    int first[kEpi];
};

struct GramBars {
    uint64_t ffull[kMaxRing], fempty[kMaxRing], xfull[kMaxRing], xempty[kMaxRing], dfull[2], dempty[2];
};

// M/N-major operand in the 128-byte swizzle: atoms of 64 slot-rows (128 B) x 8
// points (1024 B); the next 8 points 1024 B on, the next 64 slot-rows one
// kAtomBytes on.
__device__ __forceinline__ uint64_t gdesc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kAtomBytes >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// kind::f16: BF16 A and B, FP32 D, both operands transposed (M- and N-major), M = 128.
__device__ __forceinline__ uint32_t gidesc(int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) |
           ((128u >> 4) << 24);
}

__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float2 lds2(const unsigned char *p) { return *reinterpret_cast<const float2 *>(p); }

// The products v of eight rows at this lane's two points, st the field stage there.
template <int KIND>
__device__ __forceinline__ void load_chunk(const unsigned char *st, const uint32_t *oy, const uint32_t *ox, float2 *v) {
    float2 x[8], y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) y[i] = (KIND == kRowsBlock && i >= 4) ? y[i - 4] : lds2(st + oy[i]);
    if (KIND == kRowsSingle) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = y[i];
        return;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = (KIND != kRowsAny && (i & 3)) ? x[i & 4] : lds2(st + ox[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __fmul2_rn(x[i], y[i]);
}

// Eight rows' values split and stored: hi, lo are the chunk's slots at K row
// `lane`, the second point's 4096 B on.
__device__ __forceinline__ void store_chunk(const float2 *v8, unsigned char *hi, unsigned char *lo) {
    uint32_t h[2][4], l[2][4];
    const float2 minus = make_float2(-1.f, -1.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // rows 2i, 2i + 1 share a word
        const float2 u = v8[2 * i], v = v8[2 * i + 1];
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(u.x, v.x), h1 = __floats2bfloat162_rn(u.y, v.y);
        h[0][i] = *reinterpret_cast<const uint32_t *>(&h0);
        h[1][i] = *reinterpret_cast<const uint32_t *>(&h1);
        const float2 uh = make_float2(__uint_as_float(h[0][i] << 16), __uint_as_float(h[1][i] << 16));
        const float2 vh = make_float2(__uint_as_float(h[0][i] & 0xffff0000u), __uint_as_float(h[1][i] & 0xffff0000u));
        const float2 ul = __ffma2_rn(uh, minus, u), vl = __ffma2_rn(vh, minus, v);  // exact
        const __nv_bfloat162 l0 = __floats2bfloat162_rn(ul.x, vl.x), l1 = __floats2bfloat162_rn(ul.y, vl.y);
        l[0][i] = *reinterpret_cast<const uint32_t *>(&l0);
        l[1][i] = *reinterpret_cast<const uint32_t *>(&l1);
    }
    *reinterpret_cast<uint4 *>(hi) = make_uint4(h[0][0], h[0][1], h[0][2], h[0][3]);
    *reinterpret_cast<uint4 *>(lo) = make_uint4(l[0][0], l[0][1], l[0][2], l[0][3]);
    *reinterpret_cast<uint4 *>(hi + 4096) = make_uint4(h[1][0], h[1][1], h[1][2], h[1][3]);
    *reinterpret_cast<uint4 *>(lo + 4096) = make_uint4(l[1][0], l[1][1], l[1][2], l[1][3]);
}

// One unit: st the field stage at this lane's two points, xb the operand stage at
// this lane's K row.
__device__ __forceinline__ void form_unit(const unsigned char *st, const GramUnit &U, unsigned char *xb, int lane) {
    unsigned char *const xa = xb + (U.unit >> 1) * kAtomBytes;  // two units to an atom
    const uint32_t s0 = (uint32_t)(4 * (U.unit & 1)), sw = (uint32_t)(lane & 7);
    if (U.block) {
        float2 y[4], v[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = lds2(st + U.y[i]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float2 xa0 = lds2(st + U.x[8 * k]), xa1 = lds2(st + U.x[8 * k + 4]);
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __fmul2_rn(i < 4 ? xa0 : xa1, y[i & 3]);
            store_chunk(v, xa + (((s0 + 2 * k) ^ sw) << 4), xa + (((s0 + 2 * k + 1) ^ sw) << 4));
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        float2 v[8];
        const uint32_t *oy = U.y + 8 * k, *ox = U.x + 8 * k;
        const int kind = U.kind[k];
        if (kind == kRowsBlock) load_chunk<kRowsBlock>(st, oy, ox, v);
        else if (kind == kRowsStars) load_chunk<kRowsStars>(st, oy, ox, v);
        else if (kind == kRowsSingle) load_chunk<kRowsSingle>(st, oy, ox, v);
        else load_chunk<kRowsAny>(st, oy, ox, v);
        store_chunk(v, xa + (((s0 + 2 * k) ^ sw) << 4), xa + (((s0 + 2 * k + 1) ^ sw) << 4));
    }
}

// grid: (point-range CTAs, groups, fields of a batch).
// F field stages and S operand stages in shared memory.
template <int CAP>
__global__ void __launch_bounds__(kGThreads, 1)
    contract_gram_kernel(const __grid_constant__ CUtensorMap fmap, long long npts, int nbins,
                         const GramGroup *__restrict__ groups, const GramTable *__restrict__ tables,
                         const __grid_constant__ GramUnits<CAP> units, const int *__restrict__ iout, int nitems_total, double *__restrict__ part, int part_rows,
                         int F, int S, int lanes, int stage_atoms, int first, int *__restrict__ err, long long wait_limit) {
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ GramBars bars;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform to the compiler too
    const GramGroup g = groups[blockIdx.y];
    const int nu = g.nunits;
    const int ntile = (g.nbch + 15) / 16;
    const int nwords = (8 * g.nbch + 31) / 32;

    // ---- shared memory: operand stages (1024-aligned), field stages, item sums, masks
    unsigned char *const X0 = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    const int xstage = stage_atoms * kAtomBytes;
    unsigned char *const f0 = X0 + S * xstage;
    const int fstage = (nbins + 2) * kPts * 4;  // the bins, a row of ones, a row of zeros
    float2 *const sums = reinterpret_cast<float2 *>(f0 + F * fstage);
    unsigned *const smask = reinterpret_cast<unsigned *>(sums + g.nitems);
    int *const sfirst = reinterpret_cast<int *>(smask + kGramARows * nwords);  // [kEpi]

    if (tid == 0) {
        for (int i = 0; i < F; ++i) {
            mbar_init(&bars.ffull[i], 1);
            mbar_init(&bars.fempty[i], nu);
        }
        for (int i = 0; i < S; ++i) {
            mbar_init(&bars.xfull[i], nu);
            mbar_init(&bars.xempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars.dfull[i], 1);
            mbar_init(&bars.dempty[i], kEpi);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < S * xstage / 16; i += kGThreads)  // rows that no unit forms stay zero
        reinterpret_cast<uint4 *>(X0)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < F * 2 * kPts; i += kGThreads) {
        const int s = i / (2 * kPts), k = i % (2 * kPts);
        reinterpret_cast<float *>(f0 + s * fstage + nbins * kPts * 4)[k] = k < kPts ? 1.f : 0.f;
    }
    for (int i = tid; i < g.nitems; i += kGThreads) sums[i] = make_float2(0.f, 0.f);
    for (int i = tid; i < kGramARows * nwords; i += kGThreads)
        smask[i] = tables[g.table].mask[i / nwords][i % nwords];
    if (tid < kEpi) sfirst[tid] = tables[g.table].first[tid];
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    volatile int *abortp = &abort_flag;

    const long long nsteps_all = (npts + kPts - 1) / kPts;
    const long long c0 = nsteps_all * blockIdx.x / gridDim.x;
    const int nsteps = (int)(nsteps_all * (blockIdx.x + 1) / gridDim.x - c0);

    if (warp < kProd) {
        // ================= producers =================
        // A warp forms one unit of every `lanes`-th step; lanes divides F and S, so
        // a slot's previous use was this warp's own and the parity it waits for is
        // never two phases ahead.
        const uint32_t lane_off = (uint32_t)((lane >> 3) * 1024 + (lane & 7) * 128);
        const unsigned char *const fl = f0 + 8 * lane;
        unsigned char *const xl = X0 + lane_off;
        const auto wait_step = [&](int step, int fs, uint32_t fph, int xs, uint32_t xph) {
            const bool okf = mbar_try_wait(&bars.ffull[fs], fph);
            const bool okx = step < S || mbar_try_wait(&bars.xempty[xs], xph ^ 1u);
            if (!okf) role_wait(&bars.ffull[fs], fph, abortp, err, 61, wait_limit);
            if (!okx) role_wait(&bars.xempty[xs], xph ^ 1u, abortp, err, 62, wait_limit);
        };
        const auto hand_over = [&](int fs, int xs) {
            fence_proxy_async_smem();  // the stores, for the MMAs
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bars.xfull[xs]);
                mbar_arrive(&bars.fempty[fs]);
            }
        };
        if (warp < lanes * nu) {
            const GramUnit U = units.u[g.unit0 + warp % nu];
            int step = warp / nu, fs = step, xs = step;
            uint32_t fph = 0, xph = 0;
            for (; step < nsteps; step += lanes) {
                wait_step(step, fs, fph, xs, xph);
                form_unit(fl + fs * fstage, U, xl + xs * xstage, lane);
                hand_over(fs, xs);
                if ((fs += lanes) >= F) { fs -= F; fph ^= 1u; }
                if ((xs += lanes) >= S) { xs -= S; xph ^= 1u; }
            }
        }
    } else if (warp < kMma) {
        // ================= accumulators -> compensated sums =================
        const int q = (warp - kEpi0) & 3, part = (warp - kEpi0) >> 2;  // B chunks part, part + 2, ...
        const int m = 32 * q + lane;                    // accumulator row
        const int r = 8 * (m >> 4) + (m & 7);           // A row; its hi part in lanes with bit 3 clear, lo set
        const int half = (m >> 3) & 1;
        const uint32_t lanebase = tmem + ((uint32_t)(32 * q) << 16);
        const unsigned below = (1u << lane) - 1u;
        uint32_t ph[2] = {0, 0};
        const int nfl = (nsteps + kFlush - 1) / kFlush;
        for (int f = 0; f < nfl; ++f) {
            int idx = sfirst[warp - kEpi0];
            for (int t = 0; t < ntile; ++t) {
                const int d = ntile == 1 ? (f & 1) : t;
                role_wait(&bars.dfull[d], ph[d], abortp, err, 63, wait_limit);
                ph[d] ^= 1u;
                tc_fence_after();
                if (!__any_sync(0xffffffffu, *abortp)) {  // the same branch for the whole warp
                    const int nch = min(16, g.nbch - 16 * t);
                    for (int j = part; j < nch; j += kEpi / 4) {
                        const int b0 = 8 * (16 * t + j);
                        const unsigned w = (smask[r * nwords + (b0 >> 5)] >> (b0 & 31)) & 0xffu;
                        if (!__any_sync(0xffffffffu, w != 0)) continue;
                        float v[16];
                        tmem_ld16(lanebase + (uint32_t)(256 * d + 16 * j), v);
                        // columns: 8 hi then 8 lo B rows; lanes l and l ^ 8 hold the hi and lo
                        // part of the same A row and take four B rows each; lo*lo
                        // costs one add and halves the error of T against 64 bits
                        // (log bins, 96^3 to 162^3: 5.5e-6 -> 3e-6)
                        float mine[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float a = __fadd_rn(v[k], v[8 + k]);
                            const float b = __fadd_rn(v[4 + k], v[12 + k]);
                            const float got = __shfl_xor_sync(0xffffffffu, half ? a : b, 8);
                            mine[k] = __fadd_rn(half ? b : a, got);
                        }
                        const unsigned nib = half ? w >> 4 : w & 15u;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const bool on = (nib >> k) & 1u;
                            const unsigned all = __ballot_sync(0xffffffffu, on);
                            if (on) kahan_add(sums[idx + __popc(all & below)], mine[k]);
                            idx += __popc(all);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.dempty[d]);
            }
        }
    } else if (warp == kMma) {
        // ================= MMA issuer (one thread) =================
        if (elect_one()) {
            const uint64_t da0 = gdesc(smem_u32(X0)), db0 = gdesc(smem_u32(X0) + (uint32_t)(g.jb0 / 4) * kAtomBytes);
            const uint64_t dstage = (uint64_t)(uint32_t)(xstage >> 4);
            const uint32_t id0 = gidesc(16 * min(16, g.nbch)), id1 = gidesc(16 * max(1, g.nbch - 16));
            int xs = 0, step = 0;
            uint32_t xph = 0;
            const auto issue = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t id, bool first) {
                mma_ss(d, a, b, id, first ? 0u : 1u);
#pragma unroll
                for (int k = 1; k < kPts / 16; ++k) mma_ss(d, a + 128u * k, b + 128u * k, id, 1u);  // 16 points: 2048 B
            };
            // the accumulator flush f - 2 (one tile) or f - 1 (two) is read before flush f overwrites it
            for (int f = 0; step < nsteps; ++f) {
                const int n = min(kFlush, nsteps - step);
                bool okd = true;
                if (ntile == 1 && f >= 2) {
                    okd = role_wait(&bars.dempty[f & 1], (uint32_t)(((f >> 1) - 1) & 1), abortp, err, 65, wait_limit);
                    tc_fence_after();
                }
                for (int i = 0; i < n; ++i, ++step) {
                    const bool ok = role_wait(&bars.xfull[xs], xph, abortp, err, 64, wait_limit) && okd;
                    const uint64_t a = da0 + dstage * (uint64_t)(uint32_t)xs, b = db0 + dstage * (uint64_t)(uint32_t)xs;
                    if (ntile == 1) {
                        if (ok) issue(tmem + 256u * (uint32_t)(f & 1), a, b, id0, i == 0);
                    } else {
                        bool ok0 = ok, ok1 = ok;
                        if (i == 0 && f >= 1) {
                            ok0 = role_wait(&bars.dempty[0], (uint32_t)((f - 1) & 1), abortp, err, 65, wait_limit) && ok;
                            tc_fence_after();
                        }
                        if (ok0) issue(tmem, a, b, id0, i == 0);
                        if (i == n - 1) mma_commit(&bars.dfull[0]);
                        if (i == 0 && f >= 1) {
                            ok1 = role_wait(&bars.dempty[1], (uint32_t)((f - 1) & 1), abortp, err, 65, wait_limit) && ok;
                            tc_fence_after();
                        }
                        if (ok1) issue(tmem + 256u, a, b + (uint64_t)(4 * kAtomBytes >> 4), id1, i == 0);
                    }
                    mma_commit(&bars.xempty[xs]);
                    if (++xs == S) { xs = 0; xph ^= 1u; }
                }
                mma_commit(&bars.dfull[ntile == 1 ? (f & 1) : 1]);
            }
            // drain: every MMA complete before tensor memory is released (own limit)
            if (nsteps > 0) {
                const int ls = (nsteps - 1) % S;
                if (!mbar_wait(&bars.xempty[ls], (uint32_t)(((nsteps - 1) / S) & 1))) atomicExch(err, 66);
            }
        }
    } else {
        // ================= field loader (one thread) =================
        if (elect_one() && nsteps > 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&fmap)) : "memory");
            const uint32_t bytes = (uint32_t)nbins * kPts * 4u;
            int fs = 0, issued = 0;
            uint32_t fph = 0;
            for (int step = 0; step < nsteps; ++step) {
                if (step >= F && !role_wait(&bars.fempty[fs], fph ^ 1u, abortp, err, 67, wait_limit)) break;
                // after an abort a stage may be handed back before its load landed:
                // never a second load into a slot, so the drain below covers all
                if (*abortp) break;
                mbar_expect_tx(&bars.ffull[fs], bytes);
                tma_load_2d(smem_u32(f0 + fs * fstage), &fmap, (int)((c0 + step) * kPts), (int)blockIdx.z * nbins,
                            &bars.ffull[fs]);
                ++issued;
                if (++fs == F) { fs = 0; fph ^= 1u; }
            }
            // every copy into this CTA's shared memory has landed before it exits (own limit)
            for (int j = max(0, issued - F); j < issued; ++j)
                if (!mbar_wait(&bars.ffull[j % F], (uint32_t)((j / F) & 1))) atomicExch(err, 68);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    double *row = part + ((long long)blockIdx.z * part_rows + blockIdx.x) * nitems_total;
    for (int i = tid; i < g.nitems; i += kGThreads) {
        const double v = (double)sums[i].x - (double)sums[i].y;
        double &d = row[iout[g.item0 + i]];
        d = first ? v : d + v;
    }
}

}  // namespace

// ------------------------------------------------------------------ host side
// One job: the groups' tables on the device.
struct GramJob {
    bool built = false, usable = false;
    int ngroups = 0, maxitems = 0, maxatoms = 0, maxwords = 0, maxunits = 0, nrows = 0, nbrows = 0;
    GramGroup *d_groups = nullptr;
    GramTable *d_tables = nullptr;
    std::vector<GramUnit> units;  // kernel arguments of every launch
    int *d_iout = nullptr;
    int last_F = 0, last_S = 0;
};

struct GramState {
    GramJob trip, fused;
};

static GramState &gram_state(Plan &p) {
    if (!p.gram) p.gram = new GramState();
    return *reinterpret_cast<GramState *>(p.gram);
}

void free_gram_state(Plan &p) {
    delete reinterpret_cast<GramState *>(p.gram);  // device buffers belong to the plan's allocation list
    p.gram = nullptr;
}

static size_t gram_smem(const Plan &p, const GramJob &j, int F, int S) {
    return 1024 + (size_t)S * j.maxatoms * kAtomBytes + (size_t)F * (p.nbins + 2) * kPts * 4 + (size_t)j.maxitems * 8 +
           (size_t)kGramARows * j.maxwords * 4 + kEpi * 4;
}

constexpr size_t kGramSmemCap = 225 * 1024;
constexpr int kMaxUnits = 80;  // of all groups: 11.5 KB of kernel arguments

// Eight rows' factor offsets so that rows 0..3 have one x and rows 4..7
// another, by swapping the factors of single rows (empty rows take any): true
// when that is possible.
static bool share_factors(uint32_t *x, uint32_t *y, uint32_t zero) {
    uint32_t nx[8], ny[8];
    for (int h = 0; h < 8; h += 4) {
        bool ok = false;
        for (int s = 0; s < 8 && !ok; ++s) {  // candidate common factor: any factor of the four rows
            const uint32_t c = s < 4 ? x[h + s] : y[h + s - 4];
            ok = true;
            for (int i = h; i < h + 4 && ok; ++i) {
                nx[i] = c;
                if (x[i] == c) ny[i] = y[i];
                else if (y[i] == c) ny[i] = x[i];
                else if (x[i] == zero) ny[i] = zero;
                else ok = false;
            }
        }
        if (!ok) return false;
    }
    std::copy(nx, nx + 8, x);
    std::copy(ny, ny + 8, y);
    return true;
}

// The cheapest kRows* form of eight rows (their factors reordered for it).
static int chunk_kind(uint32_t *x, uint32_t *y, uint32_t one, uint32_t zero) {
    bool single = true;
    for (int i = 0; i < 8; ++i) single &= x[i] == one || x[i] == zero;
    if (single) return kRowsSingle;
    // two common factors, each for four rows with the same four partners: any
    // factor of row 0 and any of row 4, the partners in the order of rows 0..3
    for (int s = 0; s < 4; ++s) {
        const uint32_t a = s & 1 ? y[0] : x[0], b = s & 2 ? y[4] : x[4];
        bool ok = true;
        uint32_t py[4];
        for (int i = 0; i < 4 && ok; ++i) {
            ok = (x[i] == a || y[i] == a) && (x[4 + i] == b || y[4 + i] == b);
            py[i] = x[i] == a ? y[i] : x[i];
            ok = ok && py[i] == (x[4 + i] == b ? y[4 + i] : x[4 + i]);
        }
        if (!ok) continue;
        for (int i = 0; i < 8; ++i) {
            x[i] = i < 4 ? a : b;
            y[i] = py[i & 3];
        }
        return kRowsBlock;
    }
    return share_factors(x, y, zero) ? kRowsStars : kRowsAny;
}

// Device tables of a job from its groups' rows; out[i]: output column of item i.
static void finish_gram(Plan &p, GramJob &job, const std::vector<GramRows> &groups, const std::vector<int> &out) {
    std::vector<GramGroup> hg;
    std::vector<GramTable> ht;
    std::vector<int> iout;
    const uint32_t one = (uint32_t)p.nbins * kPts * 4, zero = one + kPts * 4;
    for (const GramRows &r : groups) {
        GramGroup g{};
        g.unit0 = (int)job.units.size();
        g.jb0 = r.jb0;
        g.nbch = r.nbch;
        g.item0 = (int)iout.size();
        g.nitems = (int)r.items.size();
        g.table = (int)ht.size();
        for (int u = 0; u < (int)r.rows.size() / 16; ++u) {
            GramUnit U{};
            U.unit = u;
            bool any = false;
            for (int i = 0; i < 16; ++i) {
                const auto &x = r.rows[16 * u + i];
                any |= x[0] >= 0;
                U.x[i] = x[0] < 0 ? zero : x[1] < 0 ? one : (uint32_t)x[0] * kPts * 4;
                U.y[i] = x[0] < 0 ? zero : (uint32_t)(x[1] < 0 ? x[0] : x[1]) * kPts * 4;
            }
            if (!any) continue;
            for (int k = 0; k < 2; ++k) U.kind[k] = chunk_kind(&U.x[8 * k], &U.y[8 * k], one, zero);
            U.block = U.kind[0] == kRowsBlock && U.kind[1] == kRowsBlock && std::equal(U.y, U.y + 4, U.y + 8);
            job.units.push_back(U);
        }
        g.nunits = (int)job.units.size() - g.unit0;
        GramTable t{};
        std::vector<int> at((size_t)kGramARows * kGramBRows, -1);
        for (const auto &it : r.items) {
            t.mask[it[0]][it[1] >> 5] |= 1u << (it[1] & 31);
            at[(size_t)it[0] * kGramBRows + it[1]] = out[it[2]];
        }
        for (int e = 0, n = 0; e < kEpi; ++e) {
            t.first[e] = n;
            for (int ch = e / 4; ch < g.nbch; ch += kEpi / 4)
                for (int k = 0; k < 4; ++k)
                    for (int l = 0; l < 32; ++l) {
                        const int m = 32 * (e & 3) + l, half = (m >> 3) & 1;
                        const int o = at[(size_t)(8 * (m >> 4) + (m & 7)) * kGramBRows + 8 * ch + 4 * half + k];
                        if (o < 0) continue;
                        iout.push_back(o);
                        ++n;
                    }
        }
        hg.push_back(g);
        ht.push_back(t);
        job.maxitems = std::max(job.maxitems, g.nitems);
        // A reads two whole atoms, B whole chunks of 16 columns
        job.maxatoms = std::max(job.maxatoms, std::max(2, (std::max((int)r.rows.size() / 8, g.jb0 + g.nbch) + 3) / 4));
        job.maxwords = std::max(job.maxwords, (8 * g.nbch + 31) / 32);
        job.maxunits = std::max(job.maxunits, g.nunits);
        job.nrows = std::max(job.nrows, (int)r.rows.size());
        job.nbrows = std::max(job.nbrows, 8 * g.nbch);
    }
    job.ngroups = (int)hg.size();
    // (a group's units never outnumber the producer warps that form them: at most
    // 64 rows of A and 256 of B in units of 16)
    if (job.maxunits > kProd || (int)job.units.size() > kMaxUnits || gram_smem(p, job, 2, 2) > kGramSmemCap) return;
    TableUpload up(p);
    job.d_groups = up.put(hg);
    job.d_tables = up.put(ht);
    job.d_iout = up.put(iout);
    up.wait();
    job.usable = true;
}

// A field stage (the bins, a row of ones, a row of zeros) within 64 KB.
static bool gram_bins(const Plan &p) { return p.nbins >= 1 && (p.nbins + 2) * kPts * 4 <= 65536; }

static void build_gram_trip(Plan &p, GramJob &job) {
    job.built = true;
    const TaskList &t = p.ttask;
    std::vector<std::array<int, 3>> trip;
    for (int i = 0; i < t.npairs; ++i)
        for (int e = t.pstart[i]; e < t.pstart[i + 1]; ++e) {
            std::array<int, 3> tr = {t.ia[e], t.pb[i], t.pc[i]};
            std::sort(tr.begin(), tr.end());
            trip.push_back(tr);
        }
    if (trip.empty() || !gram_bins(p)) return;
    std::vector<GramRows> g(1);
    const std::vector<int> cover = cover_triplet_pairs(p.nbins, trip);
    if (!gram_rows_pairs(p.nbins, trip, cover, g[0]) && !gram_rows_wide(p.nbins, trip, cover, g)) return;
    finish_gram(p, job, g, t.iout);
}

static void build_gram_fused(Plan &p, GramJob &job) {
    job.built = true;
    const TaskList &t = p.ttask, &q = p.qtask;
    std::vector<std::array<int, 4>> items;
    std::vector<int> out;
    for (int i = 0; i < t.npairs; ++i)
        for (int e = t.pstart[i]; e < t.pstart[i + 1]; ++e) {
            items.push_back({t.ia[e], t.pb[i], t.pc[i], -1});
            out.push_back(t.iout[e]);
        }
    for (int i = 0; i < q.npairs; ++i)
        for (int e = q.pstart[i]; e < q.pstart[i + 1]; ++e) {
            items.push_back({q.ia[e], q.ib[e], q.pb[i], q.pc[i]});
            out.push_back(t.nitems + q.iout[e]);
        }
    if (items.empty() || !gram_bins(p)) return;
    std::vector<GramRows> g(1);
    if (!gram_rows_shared(p.nbins, items, g[0])) return;
    finish_gram(p, job, g, out);
}

// BF16x3 with every tensor-core option at its default (an option names a form
// of the tensor-memory kernel).  Faster than that kernel at every job it can
// hold (the figures above; 64^3, 12 bins, 30 -> 19 us; 192^3, 48 bins, 787 ->
// 746 us), so there is no further rule on sizes: what does not fit (more than
// 64 bins on operand A, more than 256 rows or kMaxUnits units, or two operand
// and two field stages past kGramSmemCap: 46 to 48 linear bins at 256^3 and
// above) stays there.
static bool gram_options(const Plan &p) {
    return !p.gram_off && p.precision == FBS_PREC_BF16X3 && !p.tc_wide && !p.tc_roles && !p.tc_chunk && !p.tc_pairs && !p.tc_merge &&
           !p.tc_bstages && !p.tc_bfroma && !p.tc_stack;
}

bool gram_usable(Plan &p, bool fused) {
    if (!gram_options(p)) return false;
    GramJob &job = fused ? gram_state(p).fused : gram_state(p).trip;
    if (!job.built) {
        if (fused) build_gram_fused(p, job);
        else build_gram_trip(p, job);
    }
    return job.usable;
}

void launch_gram(Plan &p, bool fused, const float *islab, long long npts, long long slab_stride, double *part,
                 int nitems_total, int kclass, int nf) {
    GramJob &job = fused ? gram_state(p).fused : gram_state(p).trip;
    int sms = 0, dev = 0;
    FBS_CUDA(cudaGetDevice(&dev));
    FBS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // CTAs per field and group: one wave of one CTA per SM over all of them
    const int G = std::min(p.part_blocks, std::max(1, sms / (job.ngroups * nf)));
    // operand stages, and as many field stages as shared memory still holds: a
    // field load takes about 3,800 cycles (measured, all SMs loading) and a step
    // at least 130 cycles per unit, so about 30 / units of them have to be in flight
    const int fmin = std::max(3, (30 + job.maxunits - 1) / job.maxunits);
    int F = 2, S = 2, lanes = 1;
    for (int s : {8, 4, 3, 2}) {
        // steps that the producers have in flight: a power of two that divides S and F
        int l = 1;
        while (s % (2 * l) == 0 && 2 * l * job.maxunits <= kProd) l *= 2;
        int f = kMaxRing;
        while (f > 2 && (f % l || gram_smem(p, job, f, s) > kGramSmemCap)) --f;
        if (f % l || gram_smem(p, job, f, s) > kGramSmemCap || (f < fmin && s > 2)) continue;
        F = f;
        S = s;
        lanes = l;
        break;
    }
    const size_t sm = std::max<size_t>(gram_smem(p, job, F, S), 116 * 1024);  // one CTA per SM
    const CUtensorMap fmap = field_map(islab, npts, slab_stride, p.nbins, nf * p.nbins, kPts, false);
    KTimer tm(p, kclass);
    p.trows = G;
    job.last_F = F;
    job.last_S = S;
    const auto run = [&](auto kernel, auto units) {
        std::copy(job.units.begin(), job.units.end(), units.u);
        allow_smem(kernel);
        kernel<<<dim3(G, job.ngroups, nf), kGThreads, sm, p.stream>>>(
            fmap, npts, p.nbins, job.d_groups, job.d_tables, units, job.d_iout, nitems_total, part, p.part_blocks, F,
            S, lanes, job.maxatoms, p.first_slab, p.root().d_errbuf, p.tc_wait_limit > 0 ? p.tc_wait_limit : kWaitCycles);
    };
    // the argument block sized for the job (1.7, 3.5 or 11.5 KB)
    if (job.units.size() <= 12) run(contract_gram_kernel<12>, GramUnits<12>{});
    else if (job.units.size() <= 24) run(contract_gram_kernel<24>, GramUnits<24>{});
    else run(contract_gram_kernel<kMaxUnits>, GramUnits<kMaxUnits>{});
    FBS_CUDA(cudaGetLastError());
}

// Job shape diagnostics (fbs_plan_tc_info): false when the job was not launched
// here, or is not with the plan's present options.  Builds nothing.
bool gram_job_info(Plan &p, bool fused, int32_t *out) {
    if (!p.gram || !gram_options(p)) return false;
    const GramJob &j = fused ? gram_state(p).fused : gram_state(p).trip;
    if (!j.usable || !j.last_S) return false;
    out[0] = out[1] = 1;
    out[2] = (j.nbrows + 127) / 128;
    out[3] = j.nrows;
    out[4] = j.nbrows;
    out[5] = 2;
    out[6] = 1;
    out[7] = 0;
    out[8] = j.last_S;
    out[9] = j.last_F;
    out[10] = 0;
    return true;
}

}  // namespace fbs
