// Certified pruning of the correlation step.
//
// For a zone axis z and a pattern b the correlations over phi3 are inverse
// transforms of the spectra c_f = sum_s FFT{P}^*_sf FFT{X}_sf (direct) and of
// its mirror counterpart, so for every bin k
//
//   C[k] = (1/N) sum_f w_f Re(c_f e^{2 pi i f k / N}) <= (1/N) sum_f w_f |c_f|
//
// (w_0 = w_{N/2} = 1, else 2).  The contraction kernels reduce every (z, b)
// pair to U = (1/N) sum_f w_f max(|c_f^dir|, |c_f^mir|), which bounds both
// correlations at once, while the spectra are on chip; the full
// correlation of an axis is then evaluated (in FP32) only while its bound can
// still beat the best score found so far.  Rounding of the contraction is
// covered by a margin E_b = kappa (1/N) sum_f w_f max_z ||P^_zf|| ||X^_bf||,
// which bounds |c_f(computed) - c_f(exact)| for every axis through
// Cauchy-Schwarz over the shells.  The winner is the same as that of the
// exhaustive evaluation (up to FP32 ties).
#include <math_constants.h>

#include <algorithm>
#include <cmath>

#include "acom_internal.cuh"
#include "fft_warp.cuh"

namespace acom {

// ---------------------------------------------------------------------------
// FP32 contraction with the bound epilogue.  CTA tile: 64 zone axes x 64
// patterns; frequencies in turn; thread tile 8 x 4 pairs, four products a pair.
// Bound by the FP32 pipe and its operand reads (a register-only loop of these
// instructions reached 60 to 65 TFLOP/s here, without operand reuse 49).  The
// products run as packed pairs (fma.rn.f32x2: (A, B) += (Pr, Pi) (Xr, Xi),
// (C, D) += (Pr, Pi) (Xi, Xr)), each half the rounding of a scalar fmaf; an
// 8 x 4 tile because a 16-byte shared load takes four cycles of the SM whatever
// it broadcasts, and 4 x 4 needed as many of those as of the FP32 pipe (42
// against 47 TFLOP/s, both in this layout); the next 8 shells load into registers
// while this step is multiplied, one barrier a step; only shells k0 .. S - 1
// are summed (the plan's rows below k0 and the padding rows are zero, their
// products exactly 0).  Every sum keeps the order of its shells.  8,190
// patterns x 903 axes x 150 shells x 181 frequencies: 42.2 -> 26.5 ms.
// ---------------------------------------------------------------------------
constexpr int kBz = 64, kBb = 64, kBk = 8;
constexpr int kBPitch = kBz + 2;      // float2 per staged shell: conflict-free transposing stores
constexpr int kBThreads = 128;        // two CTAs an SM (250 registers)
constexpr int kBRows = kBThreads * 4 / kBk;    // operand rows a load pass covers

__device__ __forceinline__ void ffma2(unsigned long long& d, unsigned long long a,
                                      unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__device__ __forceinline__ unsigned long long swap2(unsigned long long x) {
    unsigned long long y;
    asm("{\n.reg .b32 l, h;\nmov.b64 {l, h}, %1;\nmov.b64 %0, {h, l};\n}" : "=l"(y) : "l"(x));
    return y;
}

__global__ void __launch_bounds__(kBThreads, 2)
k_contract_bound_fp32(const float* __restrict__ Pr, const float* __restrict__ Pi,
                      const float* __restrict__ Xr, const float* __restrict__ Xi, int F, int N,
                      int Spad, int k0, int steps, int Z, int nb, TileSplit ts,
                      float* __restrict__ U, float* __restrict__ extra) {
    static_assert(kBRows == kBz, "one load pass covers the tile's rows");
    __shared__ __align__(16) float2 sP[2][kBk][kBPitch];
    __shared__ __align__(16) float2 sX[2][kBk][kBPitch];
    const int z0 = blockIdx.x * kBz, b0 = blockIdx.y * kBb;
    const int g = blockIdx.z, f0 = g * ts.per, f1 = min(F, f0 + ts.per);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // loads: row lr of both operands, shells lc .. lc + 3 of the step
    const int lr = t / (kBk / 4), lc = (t % (kBk / 4)) * 4;
    const bool bvalid = (b0 + lr) < nb;
    const int64_t prow = ((int64_t)(z0 + lr) * F) * Spad + k0 + lc;
    const int64_t xrow = ((int64_t)(b0 + lr) * F) * Spad + k0 + lc;
    // products: a warp takes 64 axes x 16 patterns, a lane axes zt + {0, 1} + 16
    // {0, 1, 2, 3} and patterns bt + {0, 1, 8, 9}: conflict-free 16-byte loads
    const int zt = (lane & 7) * 2, bt = warp * 16 + (lane >> 3) * 2;
    float Ud[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) Ud[i][j] = 0.f;

    float4 pr, pi, xr = make_float4(0.f, 0.f, 0.f, 0.f), xi = xr;
    auto fetch = [&](int f, int step) {
        const int o = f * Spad + step * kBk;
        pr = *reinterpret_cast<const float4*>(Pr + prow + o);
        pi = *reinterpret_cast<const float4*>(Pi + prow + o);
        if (bvalid) {
            xr = *reinterpret_cast<const float4*>(Xr + xrow + o);
            xi = *reinterpret_cast<const float4*>(Xi + xrow + o);
        }
    };
    int buf = 0;
    if (f0 < f1) fetch(f0, 0);
    for (int f = f0; f < f1; ++f) {
        unsigned long long AB[8][4], CD[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) AB[i][j] = CD[i][j] = 0ull;
        for (int step = 0; step < steps; ++step, buf ^= 1) {
            // a buffer is refilled two steps after it was read, with the barrier of
            // the step between them in between
            sP[buf][lc + 0][lr] = make_float2(pr.x, pi.x);
            sP[buf][lc + 1][lr] = make_float2(pr.y, pi.y);
            sP[buf][lc + 2][lr] = make_float2(pr.z, pi.z);
            sP[buf][lc + 3][lr] = make_float2(pr.w, pi.w);
            sX[buf][lc + 0][lr] = make_float2(xr.x, xi.x);
            sX[buf][lc + 1][lr] = make_float2(xr.y, xi.y);
            sX[buf][lc + 2][lr] = make_float2(xr.z, xi.z);
            sX[buf][lc + 3][lr] = make_float2(xr.w, xi.w);
            __syncthreads();
            if (step + 1 < steps)
                fetch(f, step + 1);
            else if (f + 1 < f1)
                fetch(f + 1, 0);
#pragma unroll 4
            for (int kk = 0; kk < kBk; ++kk) {
                unsigned long long p[8], x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&sP[buf][kk][zt + 16 * q]);
                    p[2 * q] = v.x;
                    p[2 * q + 1] = v.y;
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&sX[buf][kk][bt + 8 * q]);
                    x[2 * q] = v.x;
                    x[2 * q + 1] = v.y;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const unsigned long long xs = swap2(x[j]);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        ffma2(AB[i][j], p[i], x[j]);
                        ffma2(CD[i][j], p[i], xs);
                    }
                }
            }
        }
        const float w = (f == 0 || 2 * f == N) ? 1.f : 2.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // max(|c_dir|, |c_mir|)^2 = p + 2 |AB - CD|, p = A^2 + B^2 + C^2 + D^2
                const float a_ = __uint_as_float((unsigned)AB[i][j]);
                const float b_ = __uint_as_float((unsigned)(AB[i][j] >> 32));
                const float c_ = __uint_as_float((unsigned)CD[i][j]);
                const float d_ = __uint_as_float((unsigned)(CD[i][j] >> 32));
                const float p = fmaf(a_, a_, fmaf(b_, b_, fmaf(c_, c_, d_ * d_)));
                const float q = fmaf(a_, b_, -c_ * d_);
                Ud[i][j] = fmaf(w, sqrtf(fmaf(2.0f, fabsf(q), p)), Ud[i][j]);
            }
    }
    const float invN = 1.0f / (float)N;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int b = b0 + bt + (j & 1) + 8 * (j >> 1);
        if (b >= nb) continue;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int z = z0 + zt + (i & 1) + 16 * (i >> 1);
            if (z < Z)
                *(g == 0 ? U + (int64_t)b * Z + z
                         : extra + ts.extra_at(g, ts.split_tile(b, z), b, z)) = Ud[i][j] * invN;
        }
    }
}

// A grid of fewer CTAs than the GPU holds (two an SM) leaves SMs idle while each
// CTA runs every frequency in turn, so a small batch's frequencies are split
// into groups.  From two CTAs an SM on there is no split: every SM has its CTAs
// anyway, and the partial bounds would only add traffic.  100 patterns x 231
// axes (8 tiles, 31 groups): 1.24 -> 0.049 ms.
TileSplit fp32_split(const acom_plan_s* p, int nb, bool split) {
    TileSplit ts;
    ts.ZT = (p->Z + kBz - 1) / kBz;
    ts.PTu = (nb + kBb - 1) / kBb;
    ts.lb = ts.lz = 6;
    const int slots = 2 * sm_count();
    ts.set(ts.all() < slots ? slots : 1, slots, p->F, split);
    return ts;
}

void launch_contract_bound_fp32(const acom_plan_s* p, const float* Xr, const float* Xi, int nb,
                                const TileSplit& ts, float* U, float* extra, cudaStream_t st) {
    dim3 grid(ts.ZT, ts.PTu, ts.groups);
    const int steps = (p->S - p->k0 + kBk - 1) / kBk;
    prof_begin(kKContract, st);
    k_contract_bound_fp32<<<grid, kBThreads, 0, st>>>(p->Pr, p->Pi, Xr, Xi, p->F, p->N, p->Spad,
                                                      p->k0, steps, p->Z, nb, ts, U, extra);
    prof_end(kKContract, st);
}

// Adds `left` values `plane` apart to u, 32 at a time: their loads go out together, and
// their sum is a tree of fours, then a chain.
__device__ __noinline__ float add_groups(const float* __restrict__ p, int64_t plane, int left,
                                         float u) {
    for (; left > 0; left -= 32, p += 32 * plane) {
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = j < left ? p[j * plane] : 0.f;
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 32; j += 4) s += (v[j] + v[j + 1]) + (v[j + 2] + v[j + 3]);
        u += s;
    }
    return u;
}

// A split tile's later groups onto its first.  A small batch's tiles are cut into up to a
// frequency a group, and one chain of that many FP32 additions rounds more than a whole
// tile's sum (split_shells).  Called and not inlined: most tiles of a large batch are not
// split, and the select kernel is faster without the code.  Select, in one chain inlined /
// here: 65,536 patterns x 903 axes 7.78 / 7.76 ms, 16,000 x 3,486 2.47 / 2.43 ms, 100 x 231
// (45 later groups) 38.4 / 34.8 us, one pattern x 903 (18) the same within 4 %.
__device__ __forceinline__ float later_groups(const TileSplit& ts, const float* __restrict__ extra,
                                              int b, int z, float u) {
    const int t = ts.groups > 1 ? ts.split_tile(b, z) : -1;
    return t < 0 ? u
                 : add_groups(extra + ts.extra_at(1, t, b, z),
                              (int64_t)ts.tiles() << (ts.lb + ts.lz), ts.groups - 1, u);
}

__global__ void k_sum_groups(TileSplit ts, float* __restrict__ U, const float* __restrict__ extra,
                             int64_t n, int Z) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(i / Z);
        U[i] = later_groups(ts, extra, b, (int)(i - (int64_t)b * Z), U[i]);
    }
}

void launch_sum_groups(const TileSplit& ts, float* U, const float* extra, int nb, int Z,
                       cudaStream_t st) {
    if (ts.groups <= 1) return;
    const int64_t n = (int64_t)nb * Z;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 8 * (int64_t)sm_count());
    prof_begin(kKMisc, st);
    k_sum_groups<<<blocks, 256, 0, st>>>(ts, U, extra, n, Z);
    prof_end(kKMisc, st);
}

// bit s of word [z][s / 32]: shell row s of axis z (re or im) has a non-zero
// entry; one warp per row
__global__ void k_plan_shell_mask(const float* __restrict__ Pr, const float* __restrict__ Pi,
                                  int64_t rows, int Spad, int Fs, uint32_t* __restrict__ mask) {
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= rows) return;
    bool nz = false;
    for (int f = lane; f < Fs; f += 32) nz |= Pr[row * Fs + f] != 0.f || Pi[row * Fs + f] != 0.f;
    if (__any_sync(0xffffffffu, nz) && lane == 0) {
        const int64_t z = row / Spad;
        const int s = (int)(row - z * Spad);
        atomicOr(mask + z * (Spad >> 5) + (s >> 5), 1u << (s & 31));
    }
}

void launch_plan_shell_mask(const acom_plan_s* p, cudaStream_t st) {
    const int64_t rows = (int64_t)p->Zp * p->Spad;
    cudaMemsetAsync(p->smask, 0, sizeof(uint32_t) * (size_t)p->Zp * (p->Spad / 32), st);
    prof_begin(kKMisc, st);
    k_plan_shell_mask<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(
        p->Psr, p->Psi, rows, p->Spad, shell_row_stride(p->F), p->smask);
    prof_end(kKMisc, st);
}

// ---------------------------------------------------------------------------
// Selection and exact evaluation.  Persistent CTAs take the patterns in turn.
// The candidate axes of a pattern are evaluated in batches of up to kBatch:
//  * spectra: thread (shell part, candidate, frequency quad) runs down its
//    share of the shells that both the pattern and the axis reach, 16 bytes of
//    each row at a time (four frequencies), the plan's rows on their way three
//    shells ahead in shared memory, the pattern's in registers, and accumulates
//    the four real products; the shell parts are summed in shared memory;
//  * transform: the inverse transform along phi3 of c_dir + i c_mir (both
//    correlations are real, so one complex transform carries both), for 360 bins
//    by the whole block, else one warp per candidate, and the argmax over (phi3,
//    mirror) by one warp per candidate;
//  * selection: the first batch (two largest bounds) is picked as the bounds
//    load, the later ones from a list sorted once (search_order).
// Bound by the latency and the L1 throughput of the row loads: ncu on 8,190
// patterns x 903 axes shows L1 61 %, L2 37 %, DRAM 14 % and issue 33 % busy, and
// warps waiting on loads and, behind them, on the block's barriers.  Each axis
// evaluated moves its rows (140 KB on the 1-degree plan) from L2.
// ---------------------------------------------------------------------------
constexpr int kSelThreads = 256;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kBatch = 8;
constexpr int kStateBit = 11;           // 2 N <= 1440 < 2^11
constexpr int kNbrCap = 32;             // neighbours kept in shared memory and handed on
static_assert(2 * kMaxPhi <= 1 << kStateBit, "bin and mirror below the state bits");
// Shells of plan and pattern rows in flight per thread.  Three of each measured best:
// 16,000 patterns x 3,486 axes 2.95 -> 2.44 ms, 2,000 x 3 matches 9.8 -> 8.5 ms, one
// pattern 70 -> 61 us, 65,536 x 903 axes 7.68 -> 7.77; two 8.2 ms on the last, four 8.2
// (more shared memory, less L1), plan rows cached in L1 (.ca) 11.6.
constexpr int kRing = 3;
constexpr int kOrderCap = 512;          // pending axes sorted once per pattern

struct SelState {
    float T;             // best exact score so far
    unsigned Tidx;       // (z * 2 + mirror) * N + k of the best
    int bz, bk, bm;      // its axis, bin and mirror flag
    int nc;              // candidates of the current main batch
    int64_t next;        // the CTA's next pattern
    int nref;            // candidates of the current refinement batch (a field of
                         // its own: thread 0 fills it right after the main loop's
                         // last barrier, while slower threads may still read nc)
    int q0, q, qe;       // the winner's neighbours: first, next to consider, end
    int n_order, at;     // pending axes counted, the next of `order` to consider
    float best3[3];      // winning correlation at bins k - 1, k, k + 1
    float Emax;          // rounding margin of the bounds
    float next_u;        // bound of the best pending axis after a batch's picks
    float Tp[kMaxPhases];  // best exact score so far of each phase
    int ru_z;            // runner-up: best evaluated axis outside the winner's
    float ru_v;          // grid neighbourhood (-1: none), and its score
};

struct SelSmem {
    float2* tw;      // [N] (cos, sin)(2 pi i / N)
    float2* y;       // [kBatch][N] spectra of the batch, transformed in place
    float4* ring;    // [kRing][2][kSelThreads] plan rows on their way (shares space with y)
    float2* yt;      // [kBatch][N] transform ping-pong (shares space with part)
    float4* part;    // [4][sel_items(F)] partial A, B, C, D of a shell part
    float* U;        // [Z] bound, replaced by the exact score once evaluated
    // [Z] bin + mirror * N of an evaluated axis' maximum, and above kStateBit its
    // state: 0 pending, 1 evaluated, 2 in the current batch (4: of the winner's
    // neighbourhood, while the runner-up is searched)
    uint16_t* ax;
    int* nbr;        // [kNbrCap] the winner's first neighbours
    uint16_t* order; // [kOrderCap] pending axes in decreasing bound (search_order)
    float* wv;       // [kSelWarps][kBatch] per-warp top-K values
    int* wi;         // [kSelWarps][kBatch] and axes
    int* cand;       // [kBatch]
    float* res;      // [kBatch][5] best value, its index bits, values at k - 1, k, k + 1
    float* red;      // [2][kSelWarps]
    int* poff;       // [kMaxPhases + 1] first axis of each phase, then Z
    uint32_t* pmask; // [Spad / 32] shells the pattern's tents reach: its rows that may
                     // be non-zero, and the only ones the raster wrote
    uint16_t* slist; // [kBatch][Spad] shells of each candidate: pattern and plan rows both
                     // not zero
    int* slen;       // [kBatch]
    // N = 360: the spectra rows hold frequency f at perm[f] (the prime-factor
    // transform's input order), and the transform leaves bin k at pout[k]
    uint16_t* perm;
    uint16_t* pout;
    SelState* st;
};

__device__ __forceinline__ int state_of(const SelSmem& sm, int z) { return sm.ax[z] >> kStateBit; }
__device__ __forceinline__ void set_state(SelSmem& sm, int z, int v) {
    sm.ax[z] = (uint16_t)((sm.ax[z] & ((1 << kStateBit) - 1)) | (v << kStateBit));
}

// Phase of axis z: the last p with poff[p] <= z.
__device__ __forceinline__ int phase_of(const int* poff, int nph, int z) {
    int p = 0;
    while (p + 1 < nph && z >= poff[p + 1]) ++p;
    return p;
}

__device__ inline bool better(float v, unsigned i, float bv, unsigned bi) {
    return v > bv || (v == bv && i < bi);
}

__device__ inline void warp_argmax(float& v, unsigned& i) {
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const unsigned oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (better(ov, oi, v, i)) {
            v = ov;
            i = oi;
        }
    }
}

// Argmax over the warp of bounds (not negative, so their bit patterns order like
// their values; -1 marks none), ties to the lowest axis: two warp reductions.
__device__ __forceinline__ void warp_argmax_bound(float& v, unsigned& i) {
    const unsigned key = v >= 0.f ? __float_as_uint(v) + 1u : 0u;
    const unsigned m = __reduce_max_sync(0xffffffffu, key);
    i = __reduce_min_sync(0xffffffffu, m != 0u && key == m ? i : 0xffffffffu);
    v = m ? __uint_as_float(m - 1u) : -CUDART_INF_F;
}

// The up to K pending axes of largest bound with U rel + Emax >= thr
// (with per_phase, thr is the best score so far of the axis' own phase), in
// decreasing bound (ties: lowest axis), into cand and st->nc; marks them
// in the batch.  Each warp takes its K best by repeated argmax over entries strictly
// below its previous pick; warp 0 merges the warps' lists the same way.
__device__ void block_topk(SelSmem& sm, int Z, int K, float thr, float rel, float Emax,
                           bool per_phase, int nph) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float lv = CUDART_INF_F;
    unsigned li = 0u;                       // previous pick (nothing is above it)
    for (int r = 0; r < K; ++r) {
        float v = -CUDART_INF_F;
        unsigned zi = 0xffffffffu;
        for (int z = warp * 32 + lane; z < Z; z += kSelThreads) {
            if (state_of(sm, z) != 0) continue;
            const float u = sm.U[z];
            const float tz = per_phase ? sm.st->Tp[phase_of(sm.poff, nph, z)] : thr;
            if (u * rel + Emax < tz || !better(lv, li, u, (unsigned)z)) continue;
            if (better(u, (unsigned)z, v, zi)) {
                v = u;
                zi = (unsigned)z;
            }
        }
        warp_argmax(v, zi);
        if (lane == 0) {
            sm.wv[warp * kBatch + r] = v;
            sm.wi[warp * kBatch + r] = (int)zi;
        }
        if (zi == 0xffffffffu) {
            for (int r2 = r + 1 + lane; r2 < K; r2 += 32) sm.wi[warp * kBatch + r2] = -1;
            break;
        }
        lv = v;
        li = zi;
    }
    __syncthreads();
    if (warp == 0) {
        const int ne = kSelWarps * K;
        lv = CUDART_INF_F;
        li = 0u;
        int n = 0;
        for (int r = 0; r < K; ++r) {
            float v = -CUDART_INF_F;
            unsigned zi = 0xffffffffu;
            for (int e = lane; e < ne; e += 32) {
                const int w = e / K, j = e - w * K;
                const int z = sm.wi[w * kBatch + j];
                if (z < 0) continue;
                const float u = sm.wv[w * kBatch + j];
                if (better(lv, li, u, (unsigned)z) && better(u, (unsigned)z, v, zi)) {
                    v = u;
                    zi = (unsigned)z;
                }
            }
            warp_argmax(v, zi);
            if (zi == 0xffffffffu) break;
            if (lane == 0) {
                sm.cand[n] = (int)zi;
                set_state(sm, (int)zi, 2);
            }
            ++n;
            lv = v;
            li = zi;
        }
        if (lane == 0) {
            sm.st->nc = n;
        }
    }
    __syncthreads();
}

// 16 bytes of global memory on their way to shared memory, seen after a wait of the
// same thread
__device__ __forceinline__ void copy16_async(float4* dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int Pending>
__device__ __forceinline__ void copies_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(Pending) : "memory");
}

__device__ __forceinline__ void fma4(float4& acc, const float4 p, const float4 x) {
    acc.x = fmaf(p.x, x.x, acc.x);
    acc.y = fmaf(p.y, x.y, acc.y);
    acc.z = fmaf(p.z, x.z, acc.z);
    acc.w = fmaf(p.w, x.w, acc.w);
}

struct SelectArgs {
    const float *Psr, *Psi, *Xsr, *Xsi;   // FP32 spectra, shell-major [.][Spad][Fs]
    const float* U;                   // [nb][Z] bounds
    const float* extra;               // their later groups (TileSplit)
    TileSplit ts;
    const float* xfn;                 // [nb][F] ||X^_bf||
    const int2* srange;               // [nb] non-zero shell range
    const uint32_t* rmask;            // [nb][Spad / 32] shells the pattern's tents reach
    const float* pfmax;               // [F] max_z ||P^_zf||
    const float* xnorm2;              // [nb] ||X||^2
    const double* za;                 // [Z][3]
    const double* frames;             // [Z][9]
    const int* nbr_ptr;
    const int* nbr_idx;
    const int* phase_off;             // [n_phases + 1]
    int n_phases;
    int Z, F, N, S, Spad, nb, refine;
    float kappa;                      // contraction rounding constant
    FftRadix rad;                     // inverse-transform factorisation
    acom_result out;
    int64_t off;
    int* n_eval;                      // [0] total axes evaluated, [1] patterns taken
    int taken;                        // n_eval[1] when this launch starts
    const float* xscale;              // [nb] 2^e of FP16 pattern spectra or pairs, or nullptr
    float inv_pscale;                 // 2^-k of the plan operand's scale
    float xs_mul;                     // the pattern operand holds xscale * xs_mul times X^
    float eta;                        // absolute error of an operand below its normal range
    int rescore_top;                  // > 0: evaluate only the top axes by bound (no certificate)
    const uint32_t* smask;            // [Zp][Spad / 32] non-zero plan shells
    OrientIn* oin;                    // [nb] the winners, for k_orient_compose
    float2* onbr;                     // [nb][kNbrCap] their neighbours (score, axis)
    float eta_rs = 0.f;               // eta sqrt(Spad), from the host (FP64 there)
};

__host__ __device__ inline size_t sel_items(int F) {
    const int Fq = shell_row_stride(F) >> 2;
    return (size_t)(kSelThreads > kBatch * Fq ? kSelThreads : kBatch * Fq);
}

// Spectra c_dir + i c_mir of the batch's candidate axes, scaled by 1/N, into
// the rows y[c] (both halves of the conjugate-symmetric spectrum), stored as
// their complex conjugates.
template <bool PFA>
__device__ void batch_spectra(const SelectArgs& a, int64_t b, int nc, int s_lo, int s_hi,
                              SelSmem& sm) {
    const int F = a.F, N = a.N, Fq = shell_row_stride(F) >> 2;
    const int items = nc * Fq;
    const int len = s_hi - s_lo;
    int h = kSelThreads / items;
    h = h < 1 ? 1 : (h > 8 ? 8 : h);
    if (h > len) h = len > 1 ? len : 1;
    const int total = items * h;
    const int pl = (int)sel_items(F);
    // each candidate's shells: rows of both the pattern and the axis not zero
    // (a product with a zero row is exactly 0 and is skipped); warp c lists
    // candidate c in increasing shell order
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, MW = a.Spad >> 5;
        for (int c = warp; c < nc; c += kSelWarps) {
            const uint32_t* pm = a.smask + (int64_t)sm.cand[c] * MW;
            const uint32_t m = lane < MW ? (sm.pmask[lane] & pm[lane]) : 0u;
            uint16_t* L = sm.slist + c * a.Spad;
            int tot = 0;
            for (int w = 0; w < MW; ++w) {
                const uint32_t mw = __shfl_sync(0xffffffffu, m, w);
                if (mw >> lane & 1u) L[tot + __popc(mw & ((1u << lane) - 1u))] = (uint16_t)(32 * w + lane);
                tot += __popc(mw);
            }
            if (lane == 0) sm.slen[c] = tot;
        }
        __syncthreads();
    }
    const int64_t blk = (int64_t)a.Spad * Fq;       // float4 per pattern or axis
    const float4* xr0 = reinterpret_cast<const float4*>(a.Xsr) + b * blk;
    const float4* xi0 = reinterpret_cast<const float4*>(a.Xsi) + b * blk;
    for (int idx = threadIdx.x; idx < total; idx += kSelThreads) {
        const int hh = idx / items, rem = idx - hh * items;
        const int c = rem / Fq, fq = rem - c * Fq;
        const uint16_t* L = sm.slist + c * a.Spad;
        const int ln = sm.slen[c];
        const int sa = (ln * hh) / h, se = (ln * (hh + 1)) / h;   // positions in the list
        const int64_t pb = (int64_t)sm.cand[c] * blk + fq;
        const float4* pr = reinterpret_cast<const float4*>(a.Psr) + pb;
        const float4* pi = reinterpret_cast<const float4*>(a.Psi) + pb;
        const float4* xr = xr0 + fq;
        const float4* xi = xi0 + fq;
        float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = A, C = A, D = A;
        // the plan rows of the next kRing shells are on their way to this thread's own
        // slots (no barrier, no registers), the pattern rows of as many in registers
        float4* ring = sm.ring + threadIdx.x;
        auto fetch = [&](int i, int d) {
            if (i < se) {
                const int o = L[i] * Fq;
                copy16_async(ring + 2 * d * kSelThreads, pr + o);
                copy16_async(ring + (2 * d + 1) * kSelThreads, pi + o);
            }
            copies_commit();
        };
        float4 xn1[kRing], xn2[kRing];
        auto load_x = [&](int i, int d) {
            if (i < se) {
                const int o = L[i] * Fq;
                xn1[d] = __ldg(xr + o);
                xn2[d] = __ldg(xi + o);
            }
        };
#pragma unroll
        for (int d = 0; d < kRing; ++d) fetch(sa + d, d);
#pragma unroll
        for (int d = 0; d < kRing; ++d) load_x(sa + d, d);
        for (int i0 = sa; i0 < se; i0 += kRing) {
#pragma unroll
            for (int d = 0; d < kRing; ++d) {
                const int i = i0 + d;
                if (i >= se) break;
                copies_wait<kRing - 1>();
                const float4 p1 = ring[2 * d * kSelThreads], p2 = ring[(2 * d + 1) * kSelThreads];
                const float4 x1 = xn1[d], x2 = xn2[d];
                fma4(A, p1, x1);
                fma4(B, p2, x2);
                fma4(C, p1, x2);
                fma4(D, p2, x1);
                fetch(i + kRing, d);
                load_x(i + kRing, d);
            }
        }
        copies_wait<0>();
        sm.part[idx] = A;
        sm.part[pl + idx] = B;
        sm.part[2 * pl + idx] = C;
        sm.part[3 * pl + idx] = D;
    }
    __syncthreads();
    const float invN = 1.0f / (float)N;
    for (int e = threadIdx.x; e < nc * F; e += kSelThreads) {
        const int c = e / F, f = e - c * F;
        float A = 0.f, B = 0.f, C = 0.f, D = 0.f;
        for (int hh = 0; hh < h; ++hh) {
            const float* q = reinterpret_cast<const float*>(sm.part + hh * items + c * Fq) + f;
            A += q[0];
            B += q[4 * pl];
            C += q[8 * pl];
            D += q[12 * pl];
        }
        const float dre = (A + B) * invN, dim = (C - D) * invN;
        const float mre = (A - B) * invN, mim = -(C + D) * invN;
        // stored conjugated: the inverse transform runs as a forward one
        float2* y = sm.y + c * N;
        y[PFA ? (int)sm.perm[f] : f] = make_float2(dre - mim, -(dim + mre));
        if (f > 0 && 2 * f < N) y[PFA ? (int)sm.perm[N - f] : N - f] = make_float2(dre + mim, dim - mre);
    }
    __syncthreads();
}

// C_dir[k] + i C_mir[k] = sum_f y_f exp(2 pi i f k / N) of each candidate, taken as
// the conjugate of the forward transform of conj(y) (the rows hold conj(y)); the
// argmax over (k, mirror) with the correlation at k - 1, k, k + 1 goes to res[c].
// The prime-factor transform's three stages run over all candidates' small DFTs
// with every thread (a warp a candidate left five of eight warps idle at the usual
// three candidates); other lengths and the argmax take one warp per candidate.
template <bool PFA>
__device__ void batch_transforms(const SelectArgs& a, int nc, SelSmem& sm) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, N = a.N;
    if constexpr (PFA) {
        for (int t = threadIdx.x; t < nc * 45; t += kSelThreads)
            pfa360_stage8(sm.y + (t / 45) * 360, nullptr, t % 45);
        __syncthreads();
        for (int t = threadIdx.x; t < nc * 40; t += kSelThreads)
            pfa360_stage9(sm.y + (t / 40) * 360, t % 40);
        __syncthreads();
        for (int t = threadIdx.x; t < nc * 72; t += kSelThreads)
            pfa360_stage5(sm.y + (t / 72) * 360, t % 72);
        __syncthreads();
    }
    for (int c = warp; c < nc; c += kSelWarps) {
        float2* row = sm.y + c * N;
        float2* alt = sm.yt + c * N;
        const float2* out;
        const uint16_t* pout = sm.pout;     // PFA: bin k at out[pout[k]]
        if constexpr (PFA) {
            out = row;
        } else if (a.rad.n > 0) {
            out = warp_fft_fixed(row, alt, N, a.rad, sm.tw, lane);
        } else {
            for (int k = lane; k < N; k += 32) {
                float2 acc = make_float2(0.f, 0.f);
                int idx = 0;
                for (int f = 0; f < N; ++f) {
                    const float2 t = cmul_conj(row[f], sm.tw[idx]);
                    acc.x += t.x;
                    acc.y += t.y;
                    idx += k;
                    if (idx >= N) idx -= N;
                }
                alt[k] = acc;
            }
            __syncwarp();
            out = alt;
        }
        float bv = -CUDART_INF_F;
        unsigned bi = 0xffffffffu;
        for (int k = lane; k < N; k += 32) {
            const float2 v = out[PFA ? (int)pout[k] : k];
            if (better(v.x, (unsigned)k, bv, bi)) {
                bv = v.x;
                bi = (unsigned)k;
            }
            if (better(-v.y, (unsigned)(N + k), bv, bi)) {
                bv = -v.y;
                bi = (unsigned)(N + k);
            }
        }
        // the largest value, then the lowest index that holds it (+ 0: a zero's sign
        // must not order equal values)
        const unsigned key = bi == 0xffffffffu ? 0u : float_order_key(bv + 0.f);
        const unsigned top = __reduce_max_sync(0xffffffffu, key);
        bi = __reduce_min_sync(0xffffffffu, key == top ? bi : 0xffffffffu);
        if (lane < 3) {
            // lane 0 the bin, lanes 1 and 2 those before and after it
            float v = 0.f;
            if (bi != 0xffffffffu) {
                const int m = (int)(bi / (unsigned)N), k = (int)bi - m * N;
                const int kk = lane == 0 ? k : (lane == 1 ? (k + N - 1) % N : (k + 1) % N);
                const float2 y = out[PFA ? (int)pout[kk] : kk];
                v = m ? -y.y : y.x;
            }
            float* r = sm.res + 5 * c;
            if (lane == 0) {
                r[0] = bi == 0xffffffffu ? -CUDART_INF_F : v;
                r[1] = __uint_as_float(bi);
            }
            r[lane == 0 ? 3 : (lane == 1 ? 2 : 4)] = v;
        }
        __syncwarp();
    }
    __syncthreads();
}

// Record the batch's exact scores; with update, fold them into the best.
// Every score also updates its phase's best.  Lane c of warp 0 takes candidate c.
__device__ void fold_batch(int nc, int N, bool update, int nph, SelSmem& sm) {
    if (threadIdx.x < 32) {
        const int c = threadIdx.x;
        SelState& st = *sm.st;
        float bv = -CUDART_INF_F;
        unsigned gidx = 0xffffffffu, bi = 0;
        int ph = -1;
        if (c < nc) {
            const int z = sm.cand[c];
            bv = sm.res[5 * c];
            bi = __float_as_uint(sm.res[5 * c + 1]);
            gidx = (unsigned)z * 2u * (unsigned)N + bi;
            ph = phase_of(sm.poff, nph, z);
            sm.U[z] = bv;
            sm.ax[z] = (uint16_t)(bi | (1u << kStateBit));
        }
        for (int p = 0; p < nph; ++p) {
            float v = ph == p ? bv : -CUDART_INF_F;
            for (int o = kBatch / 2; o > 0; o >>= 1)
                v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (c == 0 && v > st.Tp[p]) st.Tp[p] = v;
        }
        if (update) {
            float tv = bv;
            unsigned ti = gidx;
            for (int o = kBatch / 2; o > 0; o >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, tv, o);
                const unsigned oi = __shfl_xor_sync(0xffffffffu, ti, o);
                if (better(ov, oi, tv, ti)) {
                    tv = ov;
                    ti = oi;
                }
            }
            if (c < nc && ti == gidx && better(bv, gidx, st.T, st.Tidx)) {
                st.T = bv;
                st.Tidx = gidx;
                st.bz = sm.cand[c];
                st.bm = (int)(bi / (unsigned)N);
                st.bk = (int)(bi - (unsigned)st.bm * N);
                st.best3[0] = sm.res[5 * c + 2];
                st.best3[1] = sm.res[5 * c + 3];
                st.best3[2] = sm.res[5 * c + 4];
            }
        }
    }
    __syncthreads();
}

// The bound an axis must reach to be evaluated: the best score so far, of its own
// phase when every phase is certified.
__device__ __forceinline__ float search_threshold(const SelSmem& sm, bool per_phase, int nph, int z) {
    return per_phase ? sm.st->Tp[phase_of(sm.poff, nph, z)] : sm.st->T;
}

// After the first batch: the pending axes whose bound can reach their threshold, in
// decreasing bound (ties: lowest axis), into `order`.  The thresholds only rise, so
// no other axis becomes pending and the later batches take the list in turn: one
// scan of the axes a pattern instead of kBatch a batch (phases workload, 2,001
// axes and 17 batches a pattern: 33,000 of a batch's 66,000 cycles).  More than
// kOrderCap axes: -1, the batch scans (block_topk) and the next tries again.  Returns
// the length, the same in every thread.
__device__ int search_order(SelSmem& sm, int Z, float rel, float Emax, bool per_phase, int nph) {
    float* lu = reinterpret_cast<float*>(sm.part);                    // not in use here
    uint16_t* lz = reinterpret_cast<uint16_t*>(lu + kOrderCap);
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) sm.st->n_order = 0;
    __syncthreads();
    for (int z0 = threadIdx.x - lane; z0 < Z; z0 += kSelThreads) {
        const int z = z0 + lane;
        const float u = z < Z ? sm.U[z] : 0.f;
        const bool in = z < Z && state_of(sm, z) == 0 && u == u &&
                        !(u * rel + Emax < search_threshold(sm, per_phase, nph, z));
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (m == 0u) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(&sm.st->n_order, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
        if (in && base < kOrderCap) {
            lu[base] = u;
            lz[base] = (uint16_t)z;
        }
    }
    __syncthreads();
    const int n = sm.st->n_order;
    __syncthreads();
    if (n > kOrderCap) return -1;
    for (int i = threadIdx.x; i < n; i += kSelThreads) {
        const float u = lu[i];
        const unsigned z = lz[i];
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += better(lu[j], lz[j], u, z) ? 1 : 0;
        sm.order[rank] = (uint16_t)z;
    }
    if (threadIdx.x == 0) sm.st->at = 0;
    __syncthreads();
    return n;
}

// The next up to K axes of `order` that can still reach their threshold, into cand
// and st->nc; marks them in the batch.  The first K of the list in order are the K
// largest bounds still pending.
__device__ void next_in_order(SelSmem& sm, int n, int K, float rel, float Emax, bool per_phase,
                              int nph) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int at = sm.st->at, nc = 0;
        while (at < n && nc < K) {
            const int z = at + lane < n ? sm.order[at + lane] : -1;
            const bool in = z >= 0 &&
                            !(sm.U[z] * rel + Emax < search_threshold(sm, per_phase, nph, z));
            const unsigned m = __ballot_sync(0xffffffffu, in);
            const int r = nc + __popc(m & ((1u << lane) - 1u));
            if (in && r < K) {
                sm.cand[r] = z;
                set_state(sm, z, 2);
            }
            // past the K-th taken entry, or the whole group
            const unsigned kth = __ballot_sync(0xffffffffu, in && r == K - 1);
            nc = min(K, nc + __popc(m));
            at += kth ? __ffs(kth) : 32;
        }
        if (lane == 0) {
            sm.st->at = at;
            sm.st->nc = nc;
        }
    }
    __syncthreads();
}

__device__ inline void matmul3d(const double* a, const double* b, double* c) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            c[3 * i + j] = a[3 * i] * b[j] + a[3 * i + 1] * b[3 + j] + a[3 * i + 2] * b[6 + j];
}

// neighbour q of the winner
__device__ __forceinline__ int neighbour(const SelectArgs& a, const SelSmem& sm, int q) {
    const int i = q - sm.st->q0;
    return i < kNbrCap ? sm.nbr[i] : a.nbr_idx[q];
}

// Outputs of the winner (warp 0).  For the orientation, the neighbour axes within
// 0.9 of the best with their scores (of more than kNbrCap neighbours their
// score-weighted FP64 sum, by a butterfly) and the correlation at bins k - 1, k,
// k + 1 go to oin[b] and onbr[b]; the FP64 sum and composition run in
// k_orient_compose, one thread per pattern, so that they do not hold up the block.
__device__ __noinline__ void write_outputs(const SelectArgs& a, int64_t b, const SelSmem& sm,
                                           bool want_ref, int lane) {
    const SelState& st = *sm.st;
    const int N = a.N, bz = st.bz, bk = st.bk, bm = st.bm;
    const float T = st.T;
    const int64_t o = a.off + b;
    const float score = T == -CUDART_INF_F ? 0.f : T;
    double a0 = 0, a1 = 0, a2 = 0;
    int n = 0;
    // (an axis not evaluated has a true score below 0.9 of the best)
    if (st.qe - st.q0 <= kNbrCap) {
        const int z2 = st.q0 + lane < st.qe ? sm.nbr[lane] : -1;
        const bool in = z2 >= 0 && state_of(sm, z2) && sm.U[z2] >= 0.9f * T;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        n = __popc(m);
        if (in)
            a.onbr[b * kNbrCap + __popc(m & ((1u << lane) - 1u))] =
                make_float2(sm.U[z2], __int_as_float(z2));
    } else {
        for (int q = st.q0 + lane; q < st.qe; q += 32) {
            const int z2 = neighbour(a, sm, q);
            if (!state_of(sm, z2)) continue;
            const float sc = sm.U[z2];
            if (sc >= 0.9f * T) {
                a0 += (double)sc * a.za[3 * z2];
                a1 += (double)sc * a.za[3 * z2 + 1];
                a2 += (double)sc * a.za[3 * z2 + 2];
            }
        }
        for (int w = 16; w > 0; w >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, w);
            a1 += __shfl_xor_sync(0xffffffffu, a1, w);
            a2 += __shfl_xor_sync(0xffffffffu, a2, w);
        }
        n = -1;
    }
    if (lane != 0) return;
    a.out.za_idx[o] = bz;
    a.out.phi3_bin[o] = bk;
    a.out.mirror[o] = (uint8_t)bm;
    a.out.score[o] = score;
    if (a.out.phase) a.out.phase[o] = phase_of(sm.poff, a.n_phases, bz);
    if (a.out.runner_za || a.out.runner_score || a.out.runner_orient) {
        // the runner-up's grid orientation frame Rz(-2 pi k / N) [Ry(pi)] in
        // FP32 (a start for refinement); the winner's grid orientation when
        // there is no runner-up
        const int rz = st.ru_z;
        const int z = rz >= 0 ? rz : bz;
        const int kbz = rz >= 0 ? (int)(sm.ax[rz] & ((1 << kStateBit) - 1)) : bk + bm * N;
        const int mm = kbz >= N ? 1 : 0, kk = kbz - mm * N;
        if (a.out.runner_za) a.out.runner_za[o] = rz;
        if (a.out.runner_score) a.out.runner_score[o] = rz >= 0 ? st.ru_v : 0.f;
        if (a.out.runner_orient) {
            float sp, cp;
            sincospif(-2.0f * (float)kk / (float)N, &sp, &cp);
            const double* Fz = a.frames + 9 * z;
            for (int i = 0; i < 3; ++i) {
                const float f0 = (float)Fz[3 * i], f1 = (float)Fz[3 * i + 1], f2 = (float)Fz[3 * i + 2];
                float c0 = f0 * cp + f1 * sp, c1 = f1 * cp - f0 * sp, c2 = f2;
                if (mm) {
                    c0 = -c0;
                    c2 = -c2;
                }
                a.out.runner_orient[9 * o + 3 * i] = c0;
                a.out.runner_orient[9 * o + 3 * i + 1] = c1;
                a.out.runner_orient[9 * o + 3 * i + 2] = c2;
            }
        }
    }
    if (a.out.phase_score)
        for (int p = 0; p < a.n_phases; ++p)      // a phase left unevaluated: all-zero image
            a.out.phase_score[o * a.n_phases + p] = st.Tp[p] == -CUDART_INF_F ? 0.f : st.Tp[p];
    if (a.out.score_cos) {
        const float xn = sqrtf(a.xnorm2[b]);
        a.out.score_cos[o] = xn > 0.f ? score / xn : 0.f;
    }
    if (!want_ref) return;
    OrientIn& r = a.oin[b];
    r.w[0] = a0;
    r.w[1] = a1;
    r.w[2] = a2;
    r.c3[0] = st.best3[0];
    r.c3[1] = st.best3[1];
    r.c3[2] = st.best3[2];
    r.z = bz;
    r.km = bk + bm * N;
    r.n = n;
}

// Orientation of each winner, one thread per pattern: parabolic phi3 offset
// from the correlation at k - 1, k, k + 1; the zone axis refined toward the
// normalised score-weighted neighbour sum; m = T frame Rz(phi3) [Ry(pi)]
// composed in FP64.
__global__ void k_orient_compose(const OrientIn* __restrict__ oin,
                                 const float2* __restrict__ onbr, int nb, int N, int refine,
                                 const double* __restrict__ za, const double* __restrict__ frames,
                                 acom_result out, int64_t off) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const OrientIn r = oin[b];
    const int bz = r.z, bm = r.km >= N ? 1 : 0, bk = r.km - bm * N;
    const int64_t o = off + b;
    double dk = 0.0, wref[3];
    if (refine) {
        const double cm = r.c3[0], c0 = r.c3[1], cp = r.c3[2];
        const double den = cm - 2.0 * c0 + cp;
        if (den < 0.0) {
            dk = (cm - cp) / (2.0 * den);
            dk = dk > 0.5 ? 0.5 : (dk < -0.5 ? -0.5 : dk);
        }
        double a0 = r.w[0], a1 = r.w[1], a2 = r.w[2];
        for (int i = 0; i < r.n; ++i) {
            const float2 v = onbr[(int64_t)b * kNbrCap + i];
            const int z2 = __float_as_int(v.y);
            a0 += (double)v.x * za[3 * z2];
            a1 += (double)v.x * za[3 * z2 + 1];
            a2 += (double)v.x * za[3 * z2 + 2];
        }
        const double nrm = sqrt(a0 * a0 + a1 * a1 + a2 * a2);
        wref[0] = nrm > 0 ? a0 / nrm : za[3 * bz];
        wref[1] = nrm > 0 ? a1 / nrm : za[3 * bz + 1];
        wref[2] = nrm > 0 ? a2 / nrm : za[3 * bz + 2];
    } else {
        wref[0] = za[3 * bz];
        wref[1] = za[3 * bz + 1];
        wref[2] = za[3 * bz + 2];
    }
    const double phi3 = -2.0 * CUDART_PI * ((double)bk + dk) / (double)N;
    if (out.phi3) out.phi3[o] = (float)phi3;
    if (!out.orient) return;
    double Rz[9], m1[9], m2[9], Tm[9];
    double c3, s3;
    sincos(phi3, &s3, &c3);
    Rz[0] = c3; Rz[1] = -s3; Rz[2] = 0; Rz[3] = s3; Rz[4] = c3; Rz[5] = 0; Rz[6] = 0; Rz[7] = 0; Rz[8] = 1;
    matmul3d(frames + 9 * bz, Rz, m1);
    if (bm) {
        for (int i = 0; i < 3; ++i) {
            m1[3 * i] = -m1[3 * i];
            m1[3 * i + 2] = -m1[3 * i + 2];
        }
    }
    const double u0 = za[3 * bz], u1 = za[3 * bz + 1], u2 = za[3 * bz + 2];
    double ax0 = u1 * wref[2] - u2 * wref[1];
    double ax1 = u2 * wref[0] - u0 * wref[2];
    double ax2 = u0 * wref[1] - u1 * wref[0];
    const double sn = sqrt(ax0 * ax0 + ax1 * ax1 + ax2 * ax2);
    const double cs = u0 * wref[0] + u1 * wref[1] + u2 * wref[2];
    for (int i = 0; i < 9; ++i) Tm[i] = (i % 4 == 0) ? 1.0 : 0.0;
    if (sn > 1e-15) {
        ax0 /= sn; ax1 /= sn; ax2 /= sn;
        const double K[9] = {0, -ax2, ax1, ax2, 0, -ax0, -ax1, ax0, 0};
        double K2[9];
        matmul3d(K, K, K2);
        for (int i = 0; i < 9; ++i) Tm[i] += sn * K[i] + (1.0 - cs) * K2[i];
    }
    matmul3d(Tm, m1, m2);
    for (int i = 0; i < 9; ++i) out.orient[9 * o + i] = (float)m2[i];
}

void launch_orient_compose(const acom_plan_s* p, const OrientIn* oin, const float2* onbr, int nb, int refine,
                           acom_result out, int64_t off, cudaStream_t st) {
    if (nb <= 0) return;
    prof_begin(kKRefine, st);
    k_orient_compose<<<(nb + 127) / 128, 128, 0, st>>>(oin, onbr, nb, p->N, refine, p->za, p->frames,
                                                       out, off);
    prof_end(kKRefine, st);
}

// the batch's spectra, and before them the plan rows on their way
__host__ __device__ inline size_t sel_row_bytes(int N) {
    const size_t y = sizeof(float2) * kBatch * (size_t)N, r = sizeof(float4) * 2 * kRing * kSelThreads;
    return y > r ? y : r;
}

// PFA: N = 360 with the prime-factor inverse transform, compiled alone (the
// radix transforms' code stays out of this kernel).  FULL: per-phase
// certificates, top-K rescoring or the runner-up may be asked for; without
// them the kernel carries only the one-certificate search and the winner's
// neighbours (a smaller kernel runs faster).
template <bool PFA, bool FULL>
__global__ void __launch_bounds__(kSelThreads, 3) k_select_exact(SelectArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Z = a.Z, F = a.F, N = a.N;
    SelSmem sm;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        unsigned char* p = smem_raw + off;
        off += (bytes + 15) & ~(size_t)15;
        return p;
    };
    sm.tw = PFA ? nullptr : reinterpret_cast<float2*>(take(sizeof(float2) * N));
    sm.y = reinterpret_cast<float2*>(take(sel_row_bytes(N)));
    sm.ring = reinterpret_cast<float4*>(sm.y);
    {
        const size_t pb = sizeof(float4) * 4 * sel_items(F), yb = sizeof(float2) * kBatch * N;
        unsigned char* shared_area = take(pb > yb ? pb : yb);
        sm.part = reinterpret_cast<float4*>(shared_area);
        sm.yt = reinterpret_cast<float2*>(shared_area);
    }
    sm.U = reinterpret_cast<float*>(take(sizeof(float) * Z));
    sm.wv = reinterpret_cast<float*>(take(sizeof(float) * kSelWarps * kBatch));
    sm.wi = reinterpret_cast<int*>(take(sizeof(int) * kSelWarps * kBatch));
    sm.cand = reinterpret_cast<int*>(take(sizeof(int) * kBatch));
    sm.res = reinterpret_cast<float*>(take(sizeof(float) * 5 * kBatch));
    sm.red = reinterpret_cast<float*>(take(sizeof(float) * 2 * kSelWarps));
    sm.poff = reinterpret_cast<int*>(take(sizeof(int) * (kMaxPhases + 1)));
    sm.pmask = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (a.Spad >> 5)));
    sm.slist = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * kBatch * a.Spad));
    sm.slen = reinterpret_cast<int*>(take(sizeof(int) * kBatch));
    sm.perm = sm.pout = nullptr;
    if (PFA) {
        sm.perm = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * 360));
        sm.pout = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * 360));
    }
    sm.st = reinterpret_cast<SelState*>(take(sizeof(SelState)));
    sm.ax = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * Z));
    sm.nbr = reinterpret_cast<int*>(take(sizeof(int) * kNbrCap));
    sm.order = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * kOrderCap));
    const int nph = a.n_phases;
    for (int i = threadIdx.x; i <= nph; i += kSelThreads) sm.poff[i] = a.phase_off[i];
    // with per-phase scores requested, every phase's best is certified
    const bool per_phase = FULL && a.out.phase_score != nullptr && nph > 1;
    const int rescore_top = FULL ? a.rescore_top : 0;

    for (int i = threadIdx.x; i < N; i += kSelThreads) {
        if constexpr (PFA) {
            sm.perm[i] = (uint16_t)pfa360_in(i);
            sm.pout[i] = (uint16_t)pfa360_out(i);
        } else {
            double s, c;
            sincospi(2.0 * (double)i / (double)N, &s, &c);
            sm.tw[i] = make_float2((float)c, (float)s);
        }
    }
    const float rel = 1.0f + 1e-5f;     // FP32 accumulation of U and of the scores
    const bool want_ref = (a.out.phi3 != nullptr) || (a.out.orient != nullptr);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    // A pattern's evaluations vary several-fold, so a CTA takes the next pattern not yet
    // taken (a fixed share left 13 % of the SM time idle on 8,190 patterns); thread 0
    // takes it while this one is set up.
    for (int64_t b = blockIdx.x; b < a.nb; b = sm.st->next) {
        // the bounds, and the three largest of each lane's (ties: lowest axis) for
        // the first batch
        float tv[3] = {-1.f, -1.f, -1.f};
        unsigned tz[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu};
        for (int z = threadIdx.x; z < Z; z += kSelThreads) {
            const float u = later_groups(a.ts, a.extra, (int)b, z, a.U[b * Z + z]);
            sm.U[z] = u;
            sm.ax[z] = 0;
            if (u > tv[2]) {
                const bool b1 = u > tv[1], b0 = u > tv[0];
                tv[2] = b1 ? tv[1] : u;
                tz[2] = b1 ? tz[1] : (unsigned)z;
                if (b1) {
                    tv[1] = b0 ? tv[0] : u;
                    tz[1] = b0 ? tz[0] : (unsigned)z;
                }
                if (b0) {
                    tv[0] = u;
                    tz[0] = (unsigned)z;
                }
            }
        }
        // the shells some peak's tent reached (recorded by the raster, which
        // wrote only those rows; every other row of the pattern is zero)
        for (int w = threadIdx.x; w < (a.Spad >> 5); w += kSelThreads)
            sm.pmask[w] = a.rmask[b * (a.Spad >> 5) + w];
        // E_b: rounding margin valid for every axis (its partial sums load
        // together with the bounds, before the first barrier).  FP16 operands add an
        // absolute term for values below the normal range: an operand x is off
        // by at most 2^-11 |x| + eta, so a dot product over Spad shells of
        // 2^e X^ and 2^k P^ gains eta sqrt(Spad) (2^e ||X^_bf|| + 2^k ||P^_zf||)
        // + Spad eta^2, i.e. after dividing by 2^(e+k)
        //   eta sqrt(Spad) (||X^_bf|| 2^-k + ||P^_zf|| 2^-e + sqrt(Spad) eta 2^-(e+k)),
        // charged four times for the four real products of c_f
        const float inv_sc = a.xscale ? 1.0f / (a.xscale[b] * a.xs_mul) : 0.f;
        const float tiny = a.eta_rs * inv_sc * a.inv_pscale;
        float e = 0.f, ea = 0.f;
        for (int f = threadIdx.x; f < F; f += kSelThreads) {
            const float w = (f == 0 || 2 * f == N) ? 1.f : 2.f;
            e = fmaf(w * a.pfmax[f], a.xfn[b * F + f], e);
            ea = fmaf(w, a.xfn[b * F + f] * a.inv_pscale + a.pfmax[f] * inv_sc + tiny, ea);
        }
        for (int o = 16; o > 0; o >>= 1) {
            e += __shfl_xor_sync(0xffffffffu, e, o);
            ea += __shfl_xor_sync(0xffffffffu, ea, o);
        }
        if (lane == 0) {
            sm.red[warp] = e;
            sm.red[kSelWarps + warp] = ea;
        }
        for (int r = 0; r < 3; ++r) {
            float v = tv[0];
            unsigned zi = tz[0];
            warp_argmax_bound(v, zi);
            if (lane == 0) {
                sm.wv[warp * kBatch + r] = v;
                sm.wi[warp * kBatch + r] = (int)zi;
            }
            if (tz[0] == zi) {               // this lane's: on to its next (none left: -1)
                tv[0] = tv[1];
                tz[0] = tz[1];
                tv[1] = tv[2];
                tz[1] = tz[2];
                tv[2] = -1.f;
                tz[2] = 0xffffffffu;
            }
        }
        __syncthreads();
        if (warp == 1) {
            // the block's two largest bounds are the first batch; the third's bound
            // tells whether a second one can follow
            float v = -1.f;
            unsigned zi = 0xffffffffu;
            if (lane < 3 * kSelWarps) {
                v = sm.wv[(lane / 3) * kBatch + lane % 3];
                zi = (unsigned)sm.wi[(lane / 3) * kBatch + lane % 3];
            }
            int n = 0;
            for (int r = 0; r < 3; ++r) {
                float bv = v;
                unsigned bz = zi;
                warp_argmax_bound(bv, bz);
                if (lane == 0) {
                    if (r == 2) sm.st->next_u = bv;
                    else if (bz != 0xffffffffu && rescore_top == 0) {
                        sm.cand[n++] = (int)bz;
                        set_state(sm, (int)bz, 2);
                    }
                }
                if (zi == bz) {
                    v = -1.f;
                    zi = 0xffffffffu;
                }
            }
            if (lane == 0) sm.st->nc = n;
        }
        if (threadIdx.x == 0) {
            float t = 0.f, ta = 0.f;
            for (int w = 0; w < kSelWarps; ++w) {
                t += sm.red[w];
                ta += sm.red[kSelWarps + w];
            }
            SelState& st = *sm.st;
            st.next = gridDim.x + (int64_t)(atomicAdd(a.n_eval + 1, 1) - a.taken);
            const float abs_term =
                a.xscale ? 4.0f * a.eta_rs * ta : 0.f;
            st.Emax = (a.kappa * t + abs_term) / (float)N * 1.01f;
            st.q0 = st.q = st.qe = 0;
            st.T = -CUDART_INF_F;
            st.Tidx = 0xffffffffu;
            st.bz = st.bk = st.bm = 0;
            st.best3[0] = st.best3[1] = st.best3[2] = 0.f;
            for (int p = 0; p < kMaxPhases; ++p) st.Tp[p] = -CUDART_INF_F;
        }
        __syncthreads();
        // the next pattern's bounds and norms on their way to L2 meanwhile
        if (sm.st->next < a.nb) {
            const char* un = reinterpret_cast<const char*>(a.U + sm.st->next * Z);
            for (int i = threadIdx.x * 128; i < 4 * Z; i += kSelThreads * 128)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(un + i));
            const char* xn = reinterpret_cast<const char*>(a.xfn + sm.st->next * F);
            if ((int)threadIdx.x * 128 < 4 * F)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(xn + threadIdx.x * 128));
        }
        const float Emax = sm.st->Emax;
        const int2 sr = a.srange[b];
        int evals = 0;
        // Three stages share one evaluation site (one copy of the batch code):
        //  0 search: batches in decreasing bound, the first the 2 largest
        //    bounds, later ones every axis whose bound can still reach the best
        //    exact score (rescore_top: the top axes by bound only);
        //  1 the winner's grid neighbours that may reach 0.9 of the best (their
        //    exact scores weight the orientation refinement);
        //  2 the runner-up: the best axis outside the winner and its grid
        //    neighbours (state 4 marks them meanwhile), certified like the
        //    winner.
        const bool single = !per_phase && rescore_top == 0;
        const bool want_ru = FULL && (a.out.runner_za || a.out.runner_score || a.out.runner_orient);
        int stage = 0, batch = 0, n_order = -1;     // n_order: axes in `order` (-1: not sorted)
        for (;;) {
            int nc = 0;
            bool update = false;
            if (stage == 0) {
                if (rescore_top > 0) {
                    const int left = rescore_top - evals;
                    if (left > 0) {
                        block_topk(sm, Z, left < kBatch ? left : kBatch, -CUDART_INF_F, rel, Emax,
                                   false, nph);
                        nc = sm.st->nc;
                    }
                } else {
                    // the first batch (two largest bounds) was picked as they loaded
                    if (batch > 0) {
                        if (n_order < 0) n_order = search_order(sm, Z, rel, Emax, per_phase, nph);
                        if (n_order >= 0)
                            next_in_order(sm, n_order, kBatch, rel, Emax, per_phase, nph);
                        else
                            block_topk(sm, Z, kBatch, sm.st->T, rel, Emax, per_phase, nph);
                    }
                    nc = sm.st->nc;
                }
                update = true;
            } else if (stage == 1) {
                // warp 0 gathers the next batch of neighbours; all threads run it
                if (warp == 0) {
                    SelState& st = *sm.st;
                    const float T = st.T;
                    int q = st.q, n = 0;
                    while (q < st.qe && n < kBatch) {
                        const int z2 = q + lane < st.qe ? neighbour(a, sm, q + lane) : -1;
                        const bool in = z2 >= 0 && state_of(sm, z2) == 0 &&
                                        !(sm.U[z2] * rel + Emax < 0.9f * T);
                        const unsigned m = __ballot_sync(0xffffffffu, in);
                        const int r = n + __popc(m & ((1u << lane) - 1u));
                        if (in && r < kBatch) {
                            sm.cand[r] = z2;
                            set_state(sm, z2, 2);
                        }
                        const unsigned kth = __ballot_sync(0xffffffffu, in && r == kBatch - 1);
                        n = min(kBatch, n + __popc(m));
                        q += kth ? __ffs(kth) : 32;
                    }
                    __syncwarp();
                    if (lane == 0) {
                        st.q = q;
                        st.nref = n;
                    }
                }
                __syncthreads();
                nc = sm.st->nref;
            } else if (FULL && stage == 2) {
                // the best evaluated axis outside the neighbourhood so far
                float v = -CUDART_INF_F;
                unsigned zi = 0xffffffffu;
                for (int z = threadIdx.x; z < Z; z += kSelThreads)
                    if (state_of(sm, z) == 1 && better(sm.U[z], (unsigned)z, v, zi)) {
                        v = sm.U[z];
                        zi = (unsigned)z;
                    }
                warp_argmax(v, zi);
                if (lane == 0) {
                    sm.wv[warp * kBatch] = v;
                    sm.wi[warp * kBatch] = (int)zi;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    float bv = -CUDART_INF_F;
                    unsigned bi = 0xffffffffu;
                    for (int w = 0; w < kSelWarps; ++w)
                        if (better(sm.wv[w * kBatch], (unsigned)sm.wi[w * kBatch], bv, bi)) {
                            bv = sm.wv[w * kBatch];
                            bi = (unsigned)sm.wi[w * kBatch];
                        }
                    sm.st->ru_z = bi == 0xffffffffu ? -1 : (int)bi;
                    sm.st->ru_v = bv;
                }
                __syncthreads();
                const bool have = sm.st->ru_z >= 0;
                // an all-zero image: every axis ties at 0, nothing to certify
                if (!(have && sm.st->T == 0.f && sm.st->Tidx == 0u)) {
                    block_topk(sm, Z, have ? kBatch : 2, have ? sm.st->ru_v : -CUDART_INF_F,
                               rel, Emax, false, nph);
                    nc = sm.st->nc;
                }
            } else {
                break;
            }
            if (nc > 0) {
                batch_spectra<PFA>(a, b, nc, sr.x, sr.y, sm);
                batch_transforms<PFA>(a, nc, sm);
                fold_batch(nc, N, update, nph, sm);
                evals += nc;
            }
            bool next = nc == 0;
            if (stage == 0 && nc > 0) {
                ++batch;
                // an all-zero image: every axis ties at 0 and the lowest index has won
                if (sm.st->T == 0.f && sm.st->Tidx == 0u) next = true;
                if (single && batch == 1 && sm.st->next_u * rel + Emax < sm.st->T) next = true;
            }
            if (!next) continue;
            // the next stage that applies
            const int bz = sm.st->bz;
            if (stage == 2) {
                for (int q = a.nbr_ptr[bz] + threadIdx.x; q < a.nbr_ptr[bz + 1]; q += kSelThreads)
                    set_state(sm, a.nbr_idx[q], state_of(sm, a.nbr_idx[q]) & 3);
                if (threadIdx.x == 0) set_state(sm, bz, state_of(sm, bz) & 3);
                __syncthreads();
                stage = 3;
                continue;
            }
            if (stage == 0 && want_ref && a.refine && sm.st->T > 0.f) {
                __syncthreads();                 // every thread has read nc
                if (warp == 0) {
                    const int q0 = a.nbr_ptr[bz], qe = a.nbr_ptr[bz + 1];
                    if (q0 + lane < qe) sm.nbr[lane] = a.nbr_idx[q0 + lane];
                    if (lane == 0) {
                        sm.st->q0 = sm.st->q = q0;
                        sm.st->qe = qe;
                    }
                    __syncwarp();
                }
                stage = 1;
                continue;
            }
            if (want_ru) {
                for (int q = a.nbr_ptr[bz] + threadIdx.x; q < a.nbr_ptr[bz + 1]; q += kSelThreads)
                    set_state(sm, a.nbr_idx[q], state_of(sm, a.nbr_idx[q]) | 4);
                if (threadIdx.x == 0) set_state(sm, bz, state_of(sm, bz) | 4);
                __syncthreads();
                stage = 2;
                continue;
            }
            stage = 3;
        }
        if (a.out.za_scores)
            for (int z = threadIdx.x; z < Z; z += kSelThreads)
                a.out.za_scores[(a.off + b) * Z + z] = state_of(sm, z) ? sm.U[z] : sm.U[z] * rel + Emax;
        if (warp == 0) {
            if (lane == 0) atomicAdd(a.n_eval, evals);
            write_outputs(a, b, sm, want_ref, lane);
        }
        __syncthreads();
    }
}

// Exhaustive mode: each phase's best score, the maximum of the exact per-axis
// scores over its axes, and the phase of the winning axis.  One warp per
// pattern.
__global__ void k_phase_outputs(const float* __restrict__ za_scores, int Z, int nb,
                                const int* __restrict__ poff, int nph, acom_result out,
                                int64_t off) {
    const int lane = threadIdx.x & 31;
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (b >= nb) return;
    const int64_t o = off + b;
    if (out.phase && lane == 0) out.phase[o] = phase_of(poff, nph, out.za_idx[o]);
    if (!out.phase_score) return;
    for (int p = 0; p < nph; ++p) {
        float m = -CUDART_INF_F;
        for (int z = poff[p] + lane; z < poff[p + 1]; z += 32) m = fmaxf(m, za_scores[b * Z + z]);
        for (int s = 16; s > 0; s >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, s));
        if (lane == 0) out.phase_score[o * nph + p] = m;
    }
}

void launch_phase_outputs(const acom_plan_s* p, const float* za_scores, int nb, acom_result out,
                          int64_t off, cudaStream_t st) {
    if (nb <= 0) return;
    prof_begin(kKMisc, st);
    k_phase_outputs<<<(nb + 3) / 4, 128, 0, st>>>(za_scores, p->Z, nb, p->phase_off, p->n_phases,
                                                   out, off);
    prof_end(kKMisc, st);
}

size_t select_smem_bytes(int Z, int N, int F, int Spad) {
    auto r16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    const size_t pb = sizeof(float4) * 4 * sel_items(F), yb = sizeof(float2) * kBatch * (size_t)N;
    return (N == 360 ? 0 : r16(sizeof(float2) * N)) + r16(sel_row_bytes(N)) + r16(pb > yb ? pb : yb) +
           r16(sizeof(float) * Z) + 2 * r16(sizeof(float) * kSelWarps * kBatch) +
           r16(sizeof(int) * kBatch) + r16(sizeof(float) * 5 * kBatch) +
           r16(sizeof(float) * 2 * kSelWarps) + r16(sizeof(int) * (kMaxPhases + 1)) +
           r16(sizeof(uint32_t) * (Spad >> 5)) + r16(sizeof(uint16_t) * kBatch * Spad) +
           r16(sizeof(int) * kBatch) +
           (N == 360 ? 2 * r16(sizeof(uint16_t) * 360) : 0) +
           r16(sizeof(SelState)) + r16(sizeof(uint16_t) * Z) + r16(sizeof(int) * kNbrCap) +
           r16(sizeof(uint16_t) * kOrderCap);
}

void launch_select_exact(const acom_plan_s* p, const float* Xsr, const float* Xsi, const float* U,
                         const float* extra, const TileSplit& ts, const float* xfn, const int2* srange, const uint32_t* rmask,
                         const float* pfmax, const float* xnorm2, int nb,
                         float kappa, int refine, acom_result out, int64_t off, int* n_eval,
                         cudaStream_t st, const float* xscale, int rescore_top, OrientIn* oin,
                         float2* onbr, int* taken) {
    SelectArgs a{p->Psr, p->Psi, Xsr, Xsi, U, extra, ts, xfn, srange, rmask, pfmax, xnorm2, p->za, p->frames,
                 p->nbr_ptr,
                 p->nbr_idx, p->phase_off, p->n_phases, p->Z, p->F, p->N, p->S, p->Spad, nb, refine, kappa,
                 fft_radices(p->N), out, off, n_eval, *taken, xscale,
                 1.0f / (p->Ps ? fp16_plan_scale(p->N) : p->pscale),
                 p->precision == ACOM_PREC_FP8 ? kFp8Shift : 1.0f,
                 (float)(p->precision == ACOM_PREC_FP8 ? kFp8Eta : (p->Ps ? kPairEta : kFp16Eta)),
                 rescore_top, p->smask, oin, onbr};
    a.eta_rs = (float)((double)a.eta * std::sqrt((double)p->Spad));
    const size_t smem = select_smem_bytes(p->Z, p->N, p->F, p->Spad);
    const bool pfa = p->N == 360;
    const bool full = (out.phase_score != nullptr && p->n_phases > 1) || rescore_top > 0 ||
                      out.runner_za || out.runner_score || out.runner_orient;
    const void* kern = pfa ? (full ? (const void*)k_select_exact<true, true>
                                   : (const void*)k_select_exact<true, false>)
                           : (full ? (const void*)k_select_exact<false, true>
                                   : (const void*)k_select_exact<false, false>);
    set_max_dynamic_smem(kern, smem);
    int dev = 0, nsm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSelThreads, smem);
    int64_t grid = (int64_t)nsm * (per_sm > 0 ? per_sm : 1);
    if (grid > nb) grid = nb;
    if (grid <= 0) return;
    *taken += nb;                    // every CTA takes one number for each pattern it had
    prof_begin(kKSelect, st);
    void* args[] = {(void*)&a};
    cudaLaunchKernel(kern, dim3((unsigned)grid), dim3(kSelThreads), args, smem, st);
    prof_end(kKSelect, st);
}

}  // namespace acom
