// Orientation-plan builder (section "Generation of an Orientation Plan").
//
//   k_reflections   every lattice point 0 < |g| < q_max (Eq. 2) and its
//                   structure factor F_hkl = sum_n f_n(|g|) exp(-2 pi i hkl.p_n)
//                   (Eq. 3), in FP64.
//   k_compact_reflections  those with |F| >= 1e-9 max|F| (V_g of Eq. 4 is zero
//                   below) in lexicographic (h, k, l) order.
//   raster (raster.cu, PlanLoader)  P0 per zone axis and its Fourier
//                   transform along phi3, plus ||P0||^2.
//   k_plan_layouts (match_tc.cu)  P = A P0, A = 1/||P0||_2, in every layout.
//
//   k_neighbours    the grid neighbours of every axis, counted, then listed.
//
// The zone-axis grid and the rotations R = Rz(phi1) Rx(theta2) (first two factors
// of Eq. 10) are small host computations in FP64.
#include <math_constants.h>

#include <algorithm>
#include <cmath>

#include "acom_internal.cuh"

namespace acom {

struct ReflParams {
    double rb[9];       // reciprocal basis rows a*, b*, c*
    int n0, n1, n2;     // index box |h| <= n0, |k| <= n1, |l| <= n2
    double q_max;
    double omega;
    int n_atoms;
};

constexpr int kReflThreads = 128, kCompactThreads = 1024;

// A thread per point of the index box: its g, |F| (-1 outside the sphere) and |F|^omega,
// and the largest |F| in *fmax (non-negative doubles order like their bits).  Bound by
// the FP64 rate, some 10^3 operations a point at 2 a clock and SM: in the single CTA that
// also compacted, the 2,197 points of Au to 1.5 / A took 168 us; over the SMs, with the
// compaction below, 30 us.
__global__ void __launch_bounds__(kReflThreads)
k_reflections(ReflParams prm, const double* __restrict__ atoms,  // [n][5]: px py pz A B
              double* __restrict__ tmp_g, double* __restrict__ tmp_F,
              double* __restrict__ tmp_amp, unsigned long long* fmax) {
    const int64_t n1w = 2 * prm.n1 + 1, n2w = 2 * prm.n2 + 1;
    const int64_t total = (int64_t)(2 * prm.n0 + 1) * n1w * n2w;
    const int64_t idx = (int64_t)blockIdx.x * kReflThreads + threadIdx.x;
    double absF = -1.0;
    if (idx < total) {
        int h = (int)(idx / (n1w * n2w)) - prm.n0;
        int k = (int)((idx / n2w) % n1w) - prm.n1;
        int l = (int)(idx % n2w) - prm.n2;
        double gx = h * prm.rb[0] + k * prm.rb[3] + l * prm.rb[6];
        double gy = h * prm.rb[1] + k * prm.rb[4] + l * prm.rb[7];
        double gz = h * prm.rb[2] + k * prm.rb[5] + l * prm.rb[8];
        double q = sqrt(gx * gx + gy * gy + gz * gz);
        if ((q > 0.0) && (q < prm.q_max)) {
            double re = 0.0, im = 0.0;
            for (int n = 0; n < prm.n_atoms; ++n) {
                const double* a = atoms + 5 * n;
                double fn = a[3] * exp(-a[4] * q * q);
                double ph = h * a[0] + k * a[1] + l * a[2];
                double sn, cs;
                sincospi(2.0 * ph, &sn, &cs);     // exp(-2 pi i ph)
                re += fn * cs;
                im -= fn * sn;
            }
            absF = sqrt(re * re + im * im);
            tmp_g[3 * idx] = gx;
            tmp_g[3 * idx + 1] = gy;
            tmp_g[3 * idx + 2] = gz;
            tmp_amp[idx] = pow(absF, prm.omega);
        }
        tmp_F[idx] = absF;
    }
    double m = absF > 0.0 ? absF : 0.0;
    for (int o = 16; o > 0; o >>= 1) m = ::fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(fmax, (unsigned long long)__double_as_longlong(m));
}

// Single CTA, one pass over the index box (at most 4M points), order kept.
__global__ void __launch_bounds__(kCompactThreads)
k_compact_reflections(int total, const double* __restrict__ tmp_g,
                      const double* __restrict__ tmp_F, const double* __restrict__ tmp_amp,
                      const unsigned long long* fmax, double* __restrict__ out_g,
                      double* __restrict__ out_amp, int* out_count) {
    __shared__ int s_warp[2][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double thr = 1e-9 * __longlong_as_double((long long)*fmax);
    int out = 0;
    for (int base = 0, t = 0; base < total; base += kCompactThreads, t ^= 1) {
        const int i = base + threadIdx.x;
        const double f = i < total ? tmp_F[i] : -1.0;
        const bool keep = f >= 0.0 && f >= thr;
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) s_warp[t][warp] = __popc(m);
        __syncthreads();
        int before = 0, all = 0;
        for (int w = 0; w < kCompactThreads / 32; ++w) {
            before += w < warp ? s_warp[t][w] : 0;
            all += s_warp[t][w];
        }
        if (keep) {
            const int pos = out + before + __popc(m & ((1u << lane) - 1u));
            out_g[3 * pos] = tmp_g[3 * i];
            out_g[3 * pos + 1] = tmp_g[3 * i + 1];
            out_g[3 * pos + 2] = tmp_g[3 * i + 2];
            out_amp[pos] = tmp_amp[i];
        }
        out += all;
    }
    if (threadIdx.x == 0) *out_count = out;
}

// Grid neighbours: for each axis the axes within 1.5 steps of it (itself among them), in
// ascending order.  A warp per axis tests 32 axes at a time; FILL false leaves the count
// at ptr[z + 1], FILL true writes the indices from ptr[z].  Bound by the latency of the
// FP64 products (Z^2 of them, twice, over all SMs): on the host the same test took 0.58
// of the 2.05 ms that a 1 degree cubic plan's build took, 8.5 of 11.6 ms at 0.5 degrees.
constexpr int kNbrWarps = 4;

template <bool FILL>
__global__ void __launch_bounds__(32 * kNbrWarps)
k_neighbours(const double* __restrict__ za, int Z, double lim, int* ptr, int* __restrict__ idx) {
    const int lane = threadIdx.x & 31, z = blockIdx.x * kNbrWarps + (threadIdx.x >> 5);
    if (z >= Z) return;
    const double x = za[3 * z], y = za[3 * z + 1], w = za[3 * z + 2];
    int n = FILL ? ptr[z] : 0;
    for (int base = 0; base < Z; base += 32) {
        const int q = base + lane;
        bool near = false;
        if (q < Z)
            near = fma(w, za[3 * q + 2], fma(y, za[3 * q + 1], x * za[3 * q])) >= lim;
        const unsigned m = __ballot_sync(0xffffffffu, near);
        if (FILL && near) idx[n + __popc(m & ((1u << lane) - 1u))] = q;
        n += __popc(m);
    }
    if (!FILL && lane == 0) ptr[z + 1] = n;
}

// ptr[0] = 0 and the running sum of the counts at ptr[1 ..]; a single CTA (at most 65,535
// counts, 64 to a thread).
__global__ void __launch_bounds__(1024) k_sum_counts(int* ptr, int Z) {
    __shared__ int s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, per = (Z + 1023) / 1024;
    const int lo = min(Z, (int)threadIdx.x * per), hi = min(Z, lo + per);
    int own = 0;
    for (int i = lo; i < hi; ++i) own += ptr[i + 1];
    int sum = own;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += v;
    }
    if (lane == 31) s_warp[warp] = sum;
    __syncthreads();
    int acc = sum - own;
    for (int k = 0; k < warp; ++k) acc += s_warp[k];
    for (int i = lo; i < hi; ++i) {
        acc += ptr[i + 1];
        ptr[i + 1] = acc;
    }
    if (threadIdx.x == 0) ptr[0] = 0;
}

static void cross3(const double* a, const double* b, double* c) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}

acom_status build_plan_device(acom_plan_s* p, const acom_crystal* cr, cudaStream_t st) {
    // Eq. 1: reciprocal basis without 2 pi
    const double* a = cr->lattice[0];
    const double* b = cr->lattice[1];
    const double* c = cr->lattice[2];
    double bxc[3], cxa[3], axb[3];
    cross3(b, c, bxc);
    cross3(c, a, cxa);
    cross3(a, b, axb);
    const double V = a[0] * bxc[0] + a[1] * bxc[1] + a[2] * bxc[2];
    if (!(std::fabs(V) > 1e-12)) return set_error(ACOM_ERR_INVALID_ARG, "degenerate lattice");
    ReflParams prm{};
    for (int i = 0; i < 3; ++i) {
        prm.rb[i] = bxc[i] / V;
        prm.rb[3 + i] = cxa[i] / V;
        prm.rb[6 + i] = axb[i] / V;
    }
    // |h| = |g . a| <= q_max |a|: the box holds every point of the sphere
    auto nrm = [](const double* v) { return std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]); };
    prm.n0 = (int)std::floor(p->q_max * nrm(a));
    prm.n1 = (int)std::floor(p->q_max * nrm(b));
    prm.n2 = (int)std::floor(p->q_max * nrm(c));
    const int64_t cand = (int64_t)(2 * prm.n0 + 1) * (2 * prm.n1 + 1) * (2 * prm.n2 + 1);
    if (cand > (int64_t)4 << 20)
        return set_error(ACOM_ERR_UNSUPPORTED, "q_max * |a_i| too large (index box > 4M points)");
    prm.q_max = p->q_max;
    prm.omega = p->omega;
    prm.n_atoms = cr->n_atoms;

    std::vector<double> atoms(5 * cr->n_atoms);
    for (int n = 0; n < cr->n_atoms; ++n) {
        for (int d = 0; d < 3; ++d) atoms[5 * n + d] = cr->frac_pos[3 * n + d];
        atoms[5 * n + 3] = cr->ff_A[n];
        atoms[5 * n + 4] = cr->ff_B[n];
    }
    double *d_atoms = nullptr, *d_tmp_g = nullptr, *d_tmp_F = nullptr, *d_tmp_amp = nullptr,
           *d_g = nullptr, *d_amp = nullptr;
    unsigned long long* d_cnt = nullptr;           // largest |F|, then the count
    cudaError_t e;
#define ACOM_TRY(x)                                        \
    do {                                                   \
        e = (x);                                           \
        if (e != cudaSuccess) goto fail;                   \
    } while (0)
    {
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_atoms), sizeof(double) * atoms.size(), st));
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_tmp_g), sizeof(double) * 3 * cand, st));
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_tmp_F), sizeof(double) * cand, st));
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_tmp_amp), sizeof(double) * cand, st));
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_g), sizeof(double) * 3 * cand, st));
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_amp), sizeof(double) * cand, st));
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_cnt), 2 * sizeof(*d_cnt), st));
        ACOM_TRY(cudaMemsetAsync(d_cnt, 0, 2 * sizeof(*d_cnt), st));
        ACOM_TRY(cudaMemcpyAsync(d_atoms, atoms.data(), sizeof(double) * atoms.size(),
                                 cudaMemcpyHostToDevice, st));
        const double lim = std::cos(1.5 * p->step_deg * M_PI / 180.0);
        const unsigned nbr_grid = (unsigned)((p->Z + kNbrWarps - 1) / kNbrWarps);
        prof_begin(kKMisc, st);
        k_neighbours<false><<<nbr_grid, 32 * kNbrWarps, 0, st>>>(p->za, p->Z, lim, p->nbr_ptr,
                                                                 nullptr);
        k_sum_counts<<<1, 1024, 0, st>>>(p->nbr_ptr, p->Z);
        prof_end(kKMisc, st);
        prof_begin(kKReflections, st);
        k_reflections<<<(unsigned)((cand + kReflThreads - 1) / kReflThreads), kReflThreads, 0, st>>>(
            prm, d_atoms, d_tmp_g, d_tmp_F, d_tmp_amp, d_cnt);
        k_compact_reflections<<<1, kCompactThreads, 0, st>>>((int)cand, d_tmp_g, d_tmp_F, d_tmp_amp,
                                                             d_cnt, d_g, d_amp, (int*)(d_cnt + 1));
        prof_end(kKReflections, st);
        ACOM_TRY(cudaGetLastError());
        ACOM_TRY(cudaMemcpyAsync(p->host_words, d_cnt + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        ACOM_TRY(cudaMemcpyAsync(p->host_words + 1, p->nbr_ptr + p->Z, sizeof(int),
                                 cudaMemcpyDeviceToHost, st));
        ACOM_TRY(cudaStreamSynchronize(st));
        p->G = p->host_words[0];
        const size_t n_nbr = (size_t)p->host_words[1];
        p->host_words[0] = p->host_words[1] = 0;
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&p->nbr_idx), sizeof(int) * n_nbr, st));
        p->bytes += sizeof(int) * n_nbr;
        prof_begin(kKMisc, st);
        k_neighbours<true><<<nbr_grid, 32 * kNbrWarps, 0, st>>>(p->za, p->Z, lim, p->nbr_ptr,
                                                                p->nbr_idx);
        prof_end(kKMisc, st);
        ACOM_TRY(cudaGetLastError());
        p->refl_g = d_g;
        p->refl_amp = d_amp;
        p->bytes += sizeof(double) * 4 * cand;
        d_g = d_amp = nullptr;
        pool_free(d_atoms, st);
        pool_free(d_tmp_g, st);
        pool_free(d_tmp_F, st);
        pool_free(d_tmp_amp, st);
        pool_free(d_cnt, st);
        d_atoms = d_tmp_g = d_tmp_F = d_tmp_amp = nullptr;
        d_cnt = nullptr;

        // P0 -> FFT along phi3 -> scale by A
        float* d_sumsq = nullptr;
        ACOM_TRY(pool_alloc(reinterpret_cast<void**>(&d_sumsq), sizeof(float) * p->Zp, st));
        ACOM_TRY(cudaMemsetAsync(d_sumsq, 0, sizeof(float) * p->Zp, st));
        RasterGeom geo{p->S, p->Spad, p->N, p->F, (float)p->dq, (float)p->delta,
                       (float)p->gamma_pow, 1};
        PlanSource src{p->refl_g, p->refl_amp, p->frames, p->G, p->lambda};
        RasterOut ro;
        ro.sre = p->Psr;
        ro.sim = p->Psi;
        ro.sumsq = d_sumsq;
        launch_raster_plan(geo, src, p->Z, ro, p->err, st);
        ACOM_TRY(cudaGetLastError());
        launch_plan_layouts(p, d_sumsq, st);
        ACOM_TRY(cudaGetLastError());
        int herr = 0;
        ACOM_TRY(cudaMemcpyAsync(&herr, p->err, sizeof(int), cudaMemcpyDeviceToHost, st));
        ACOM_TRY(cudaStreamSynchronize(st));
        prof_resolve();
        pool_free(d_sumsq, st);
        if (herr & kErrTooManyPeaks)
            return set_error(ACOM_ERR_UNSUPPORTED,
                             "more than 1024 reflections near the Ewald sphere for one zone axis");
        return ACOM_OK;
    }
fail:
    pool_free(d_atoms, st);
    pool_free(d_tmp_g, st);
    pool_free(d_tmp_F, st);
    pool_free(d_tmp_amp, st);
    pool_free(d_g, st);
    pool_free(d_amp, st);
    pool_free(d_cnt, st);
    if (e == cudaErrorMemoryAllocation) return set_error(ACOM_ERR_OOM, "plan: device allocation");
    return cuda_error(e, "plan build");
#undef ACOM_TRY
}

}  // namespace acom
