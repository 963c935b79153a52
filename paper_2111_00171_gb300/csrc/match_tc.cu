// Tensor-core (tcgen05) contraction over shells with the spectral-bound
// epilogue (section "Correlation Pattern Matching"; see match_prune.cu for the
// bound).
//
// Per frequency f the pattern spectra (shells x patterns, BF16) meet the plan
// spectra (zone axes x shells, BF16) on the 5th-generation tensor cores in one
// MMA per 16 shells:
//   D = X_f [Pr_f ; Pi_f]^T,  M = 128 pattern rows, N = 256 axis rows,
// FP32 accumulation in tensor memory.  Each 16-row group of the pattern tile
// holds the real parts of 8 patterns and then their imaginary parts, so TMEM
// lanes L and L + 8 carry Xr and Xi of one pattern; D columns 0..127 are the
// axes' real parts and 128..255 their imaginary parts.  A 16x256b TMEM load
// hands one thread (Xr.Pr, Xi.Pr) of lanes (L, L + 8), and the same load 128
// columns on gives (Xr.Pi, Xi.Pi): the four products A = Pr.Xr, C = Pr.Xi,
// D = Pi.Xr, B = Pi.Xi of a pair meet in one thread, which accumulates
// w_f max(|(A+B) + i(C-D)|, |(A-B) - i(C+D)|) over f.  The spectra never leave
// the chip; only U is written.
//
// CTA tile: 128 patterns (two MMA tiles of 64) x 128 axes.  Per frequency the plan
// operand (64 KB on the 1-degree plan) is loaded once and multiplied with both
// pattern tiles: 128 KB of L2 reads per 16 MMAs instead of 192 with one pattern
// tile, whose loads alone took 6.2 of its 9.0 ms on 65,536 patterns x 903 axes.
// That scan: 9.06 -> 7.14 ms (1,810 TFLOP/s of 8 Z S F algorithmic flops); 16,000
// patterns x 3,486 axes: 8.04 -> 6.34 ms.  What bounds it now, from timed copies of the
// kernel: an MMA reads 12 KB of shared memory in its 128 cycles and the copies
// write 62 bytes a cycle, 1.2 times the 128 bytes a cycle there are; and the epilogue
// is as long as the MMAs it runs under (without its arithmetic 6.3 ms, without the
// copies 6.6, without both 5.9).  The two pattern tiles alternate between two TMEM
// accumulators, so a tile's epilogue has the other tile's MMAs to run under.
//
// Warps: 0 loads the pattern operand (three 32 KB slots of two K tiles), 3 the plan
// operand (two 64 KB slots; one box of 256 rows, the axis tile's real rows followed
// by its imaginary rows), 1 issues every MMA, 2 hands slots back, 4 to 19 are the
// epilogue.  Issuing costs the thread about 50 cycles an MMA, whatever its size, and
// a commit 220 (measured; 380 under a `lane == 0` branch instead of elect.sync), and
// the M = 128, N = 256, K = 16 MMA takes 128: one thread keeps the tensor pipe
// busy as long as it commits about once per 8 MMAs.  So the issuer commits once per
// accumulation, and warp 2, which waits for that, releases its operand slots; only
// the earlier K stages of plans of more than 128 shells commit their own slots.
// Each K tile has its own full barrier, so MMAs start on the first K tile while
// the second lands.
// Every mbarrier wait is bounded: a timeout sets the device error word, stops
// all roles, drains copies and MMAs in flight, frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cudaTypedefs.h>
#include <math_constants.h>

#include <algorithm>
#include <type_traits>

#include "acom_internal.cuh"

namespace acom {
namespace tc {

constexpr int kM = 128;               // zone axes per tile (MMA N = 256 rows: re, im)
constexpr int kNP = 64;               // patterns per tile (MMA M = 128 rows: re, im)
constexpr int kKT = 64;               // 16-bit operands per K tile row (128 bytes)
constexpr int kKT8 = 128;             // 8-bit operands per K tile row (128 bytes)
constexpr int kTileBytes = 128 * kKT * 2;      // 16 KB
constexpr int kEpiWarps = 16;
constexpr int kIssuers = 2;                    // MMA-issuing warps of a CTA pair, one per TMEM buffer
constexpr int kProdP = 3;                      // warp of the plan-operand producer
constexpr int kEpi0 = kProdP + 1;               // first epilogue warp
constexpr int kThreads = (kEpi0 + kEpiWarps) * 32;
constexpr uint32_t kTmemCols = 512;
constexpr long long kWaitCycles = 4000000000LL;   // ~2 s at 2 GHz

// instruction descriptors: D f32, A and B both bf16 (format 1) or both f16
// (format 0), both K-major, N = 256, M = 128
constexpr uint32_t kIdescF16 = (1u << 4) | ((256u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kIdescBF16 = kIdescF16 | (1u << 7) | (1u << 10);

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait of at most `budget` clock cycles; false on timeout (recorded)
// or when another role aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* err, long long budget) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > budget) {
            atomicOr(err, kErrTimeout);
            *abort_flag = 1;
            return false;
        }
    }
}

// one lane of the (converged) warp, known to the compiler to be one
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "elect.sync _|p, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;               // leading byte offset (unused with swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset
    d |= (uint64_t)1 << 46;               // descriptor version
    d |= (uint64_t)2 << 61;               // 128-byte swizzle
    return d;
}

__device__ __forceinline__ void mma_f16kind(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                            uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// E4M3 x E4M3 -> FP32 (both operands the same type; K = 32 per instruction,
// the same 32 bytes of each operand row as K = 16 of a 16-bit type)
__device__ __forceinline__ void mma_f8kind(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                           uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ---- CTA pairs (cta_group::2): a cluster of two CTAs shares each MMA ----
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the shared::cluster address of the same shared-memory offset in CTA `rank`
__device__ __forceinline__ uint32_t mapa_rank(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t caddr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(caddr)
                 : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t caddr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(caddr), "r"(v) : "memory");
}
// a TMA copy into this CTA's shared memory that completes on a barrier of
// either CTA of the pair (`bar` a shared::cluster address)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y,
                                                 uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void mma_f16kind_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                                 uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_f8kind_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                                uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrive on the barrier at this offset in both CTAs once this thread's MMAs complete
__device__ __forceinline__ void mma_commit_pair_both(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
        " [%0], %1;" ::"r"(bar), "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

// 16 TMEM lanes x 32 columns: thread t receives, for n = 0..3, lane t/4 at
// columns 8n + 2(t%4) + {0, 1} in r[4n], r[4n+1] and lane t/4 + 8 at the same
// columns in r[4n+2], r[4n+3]
#define ACOM_TMEM_LD16x256_X4(taddr, r)                                                      \
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,"    \
                 "%10,%11,%12,%13,%14,%15}, [%16];"                                          \
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),   \
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), \
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])                        \
                 : "r"(taddr))

// wait for this thread's TMEM loads; the registers are tied to the wait so no
// use can be scheduled before it
#define ACOM_TMEM_WAIT32(p, q)                                                             \
    asm volatile("tcgen05.wait::ld.sync.aligned;"                                          \
                 : "+r"(p[0]), "+r"(p[1]), "+r"(p[2]), "+r"(p[3]), "+r"(p[4]), "+r"(p[5]), \
                   "+r"(p[6]), "+r"(p[7]), "+r"(p[8]), "+r"(p[9]), "+r"(p[10]),            \
                   "+r"(p[11]), "+r"(p[12]), "+r"(p[13]), "+r"(p[14]), "+r"(p[15]),        \
                   "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), \
                   "+r"(q[6]), "+r"(q[7]), "+r"(q[8]), "+r"(q[9]), "+r"(q[10]),            \
                   "+r"(q[11]), "+r"(q[12]), "+r"(q[13]), "+r"(q[14]), "+r"(q[15])         \
                 :                                                                         \
                 : "memory")

// |c| from |c|^2 (approximate square root, relative error ~2^-23, covered by
// the bound's rounding margin)
__device__ __forceinline__ float mag_from_sq(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// w max(|c_dir|, |c_mir|) added to the bound of two pairs (axes z and z + 1,
// adjacent registers of a 16x256b load): with p = A^2+B^2+C^2+D^2 and
// q = AB - CD, |c_dir|^2 = |(A+B) + i(C-D)|^2 = p + 2q and
// |c_mir|^2 = |(A-B) - i(C+D)|^2 = p - 2q, so the larger is p + 2|q|.  Packed
// FP32x2 arithmetic halves the epilogue's instructions, which share the issue
// slots with the MMA-issuing warps.
__device__ __forceinline__ void accumulate_pair2(uint32_t a0, uint32_t a1, uint32_t c0,
                                                 uint32_t c1, uint32_t d0, uint32_t d1,
                                                 uint32_t b0, uint32_t b1, float w, float& acc0,
                                                 float& acc1) {
    float t0, t1;
    asm("{\n"
        ".reg .b64 A, B, C, D, P, Q, R;\n"
        "mov.b64 A, {%2, %3};\n"
        "mov.b64 C, {%4, %5};\n"
        "mov.b64 D, {%6, %7};\n"
        "mov.b64 B, {%8, %9};\n"
        "mul.rn.f32x2 P, D, D;\n"
        "fma.rn.f32x2 P, C, C, P;\n"
        "fma.rn.f32x2 P, B, B, P;\n"
        "fma.rn.f32x2 P, A, A, P;\n"
        "mul.rn.f32x2 Q, C, D;\n"
        "mul.rn.f32x2 R, A, B;\n"
        "sub.rn.f32x2 Q, R, Q;\n"
        "and.b64 Q, Q, 0x7FFFFFFF7FFFFFFF;\n"
        "mov.b64 R, 0x4000000040000000;\n"
        "fma.rn.f32x2 P, Q, R, P;\n"
        "mov.b64 {%0, %1}, P;\n"
        "}\n"
        : "=f"(t0), "=f"(t1)
        : "r"(a0), "r"(a1), "r"(c0), "r"(c1), "r"(d0), "r"(d1), "r"(b0), "r"(b1));
    acc0 = fmaf(w, mag_from_sq(t0), acc0);
    acc1 = fmaf(w, mag_from_sq(t1), acc1);
}

struct TcArgs {
    int F, N, Z, nb, ZT, PT, KT;   // frequencies, bins, axes, patterns, axis tiles, pattern tiles, K stages
    TileSplit ts;                  // tiles (axis tile x two pattern tiles) and their frequency groups
    int PTs;                       // pattern tiles per frequency in the pattern map (row stride)
    int Spad;                      // shells (K) in the operand rows
    int k0;                        // first shell of the contraction's K range (the
                                   // plan's rows below it are zero for every axis)
    int Zrows;                     // rows per frequency in the plan map (ZT * 256)
    float* U;                      // [nb][Z]
    float* extra;                  // the later groups' bounds of split tiles (TileSplit)
    int* err;
    uint32_t idesc;                // MMA instruction descriptor (operand format)
    const float* xscale;           // [nb] 2^e of FP16 pattern spectra, or nullptr
    float xs_mul;                  // the operands hold xscale * xs_mul times X^
    float inv_pscale;              // 2^-k of the plan operand's scale (1 for BF16)
    long long wait_cycles;         // budget of each pipeline wait (the drain waits
                                   // that precede the exit always take kWaitCycles)
};

// One unit of work: an axis tile x two pattern tiles and a range of frequencies.
struct Unit {
    int zt, pu, g, f0, f1;
    bool split;
    int t;
};
__device__ __forceinline__ Unit unit_of(const TcArgs& a, int u) {
    Unit w;
    const TileSplit& ts = a.ts;
    w.split = u >= ts.first;
    w.t = w.split ? ts.first + (u - ts.first) / ts.groups : u;
    w.g = w.split ? (u - ts.first) % ts.groups : 0;
    w.f0 = w.split ? w.g * ts.per : 0;
    w.f1 = w.split ? min(a.F, w.f0 + ts.per) : a.F;
    w.zt = ts.zmajor ? w.t / ts.PTu : w.t % a.ZT;
    w.pu = ts.zmajor ? w.t % ts.PTu : w.t / a.ZT;
    return w;
}
// where the unit's bound of pattern b, axis z goes
__device__ __forceinline__ float* bound_at(const TcArgs& a, const Unit& w, int b, int z) {
    return w.g == 0 ? a.U + (int64_t)b * a.Z + z : a.extra + a.ts.extra_at(w.g, w.t, b, z);
}

// products of 16 axes' columns and 8 patterns' lanes into ud[0..8)
#define ACOM_ACCUMULATE(R, I, ud, w)                                                           \
    _Pragma("unroll") for (int n = 0; n < 4; ++n)                                              \
        accumulate_pair2(R[4 * n], R[4 * n + 1], R[4 * n + 2], R[4 * n + 3], I[4 * n],         \
                         I[4 * n + 1], I[4 * n + 2], I[4 * n + 3], w, (ud)[2 * n], (ud)[2 * n + 1])

constexpr int kSub = 2;                            // K tiles a slot holds
constexpr int kXSlots = 3, kPSlots = 2;
constexpr int kXBytes = kSub * kTileBytes;         // 32 KB: 128 rows
constexpr int kPBytes = 2 * kSub * kTileBytes;     // 64 KB: 256 rows
constexpr int kBars = kXSlots * (kSub + 1) + kPSlots * (kSub + 1) + 5;

// F8: E4M3 operands (kind::f8f6f4, 128 elements per K tile), else 16-bit
// (kind::f16, 64 elements per K tile); a template parameter, so the MMA issue
// loop carries no branch on it.
template <bool F8>
__global__ void __launch_bounds__(kThreads, 1)
k_contract_bound_tc(const __grid_constant__ CUtensorMap map_p,
                    const __grid_constant__ CUtensorMap map_x, TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring_p = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* ring_x = ring_p + kPSlots * kPBytes;
    uint64_t* xfull = reinterpret_cast<uint64_t*>(ring_x + kXSlots * kXBytes);   // [kXSlots][kSub]
    uint64_t* xempty = xfull + kXSlots * kSub;      // [kXSlots]
    uint64_t* pfull = xempty + kXSlots;             // [kPSlots][kSub]
    uint64_t* pempty = pfull + kPSlots * kSub;      // [kPSlots]
    uint64_t* done = pempty + kPSlots;              // [2] accumulation finished, per TMEM buffer
    uint64_t* tempty = done + 2;                    // [2] accumulator read (epilogue warps, warp 2)
    uint64_t* drain = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kXSlots * kSub; ++i) mbar_init(smem_u32(xfull + i), 1);
        for (int i = 0; i < kPSlots * kSub; ++i) mbar_init(smem_u32(pfull + i), 1);
        for (int i = 0; i < kXSlots; ++i) mbar_init(smem_u32(xempty + i), 1);
        for (int i = 0; i < kPSlots; ++i) mbar_init(smem_u32(pempty + i), 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(done + i), 1);
            mbar_init(smem_u32(tempty + i), kEpiWarps + 1);
        }
        mbar_init(smem_u32(drain), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_p)));
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)));
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int n_units = a.ts.units();
    constexpr int ktel = F8 ? kKT8 : kKT;

    if (warp == 0 || warp == kProdP) {
        // ------------------------------------------------ TMA producers
        if (elect_one()) {
            const bool xprod = warp == 0;
            const int slots = xprod ? kXSlots : kPSlots;
            uint64_t* full = xprod ? xfull : pfull;
            uint64_t* empty = xprod ? xempty : pempty;
            int slot = 0;
            uint32_t phase = 0;          // parity of the slots' current use
            uint32_t used = 0, last = 0; // per slot: used at all, parity of its last use
            bool ok = true;
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const Unit w = unit_of(a, u);
                const int nsub = min(2, a.PT - 2 * w.pu);
                for (int f = w.f0; f < w.f1 && ok; ++f)
                    for (int kt = 0; kt < a.KT && ok; ++kt) {
                        const int kbase = a.k0 + kt * ktel * kSub;
                        for (int sub = 0; sub < (xprod ? nsub : 1); ++sub) {
                            if (!mbar_wait(smem_u32(empty + slot), phase ^ 1u, abort_flag, a.err,
                                           a.wait_cycles)) {
                                ok = false;
                                break;
                            }
#pragma unroll
                            for (int k = 0; k < kSub; ++k) {
                                const uint32_t fb = smem_u32(full + slot * kSub + k);
                                const int x = kbase + k * ktel;
                                if (x >= a.Spad) {           // past the padded shells: not
                                    mbar_arrive(fb);         // loaded, not multiplied
                                } else if (xprod) {
                                    mbar_expect_tx(fb, kTileBytes);
                                    tma_load_2d(smem_u32(ring_x + slot * kXBytes + k * kTileBytes),
                                                &map_x, x, (f * a.PTs + 2 * w.pu + sub) * 128, fb);
                                } else {
                                    mbar_expect_tx(fb, 2 * kTileBytes);
                                    tma_load_2d(smem_u32(ring_p + slot * kPBytes + k * 2 * kTileBytes),
                                                &map_p, x, f * a.Zrows + w.zt * 256, fb);
                                }
                            }
                            used |= 1u << slot;
                            last = (last & ~(1u << slot)) | (phase << slot);
                            if (++slot == slots) {
                                slot = 0;
                                phase ^= 1u;
                            }
                        }
                    }
            }
            // every copy lands before the CTA's shared memory goes away
            for (int i = 0; i < slots; ++i)
                if (used & (1u << i))
                    for (int k = 0; k < kSub; ++k) {
                        const long long w0 = clock64();
                        while (!mbar_try(smem_u32(full + i * kSub + k), (last >> i) & 1u) &&
                               clock64() - w0 < kWaitCycles) {
                        }
                    }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (elect_one()) {
            int xs = 0, ps = 0;
            uint32_t xph = 0, pph = 0, tph = 0;      // tph: bit b, parity of buffer b's next use
            uint32_t buf = 0;                        // TMEM buffer of the next accumulation
            bool ok = true;
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const Unit w = unit_of(a, u);
                const int nsub = min(2, a.PT - 2 * w.pu);
                for (int f = w.f0; f < w.f1 && ok; ++f) {
                    for (int kt = 0; kt < a.KT && ok; ++kt) {
                        const bool last_k = kt + 1 == a.KT;
                        // K steps of 32 bytes inside the shells (16 16-bit or 32 8-bit
                        // elements; E4M3 rounds up into the zero fill past the shells when k0
                        // is an odd multiple of 16); a step moves the descriptors by 32 bytes
                        // (2 units)
                        const int nk = (min(ktel * kSub, a.Spad - a.k0 - kt * ktel * kSub) * (F8 ? 1 : 2) + 31) >> 5;
                        const uint64_t pd = sdesc(smem_u32(ring_p + ps * kPBytes));
                        for (int sub = 0; sub < nsub; ++sub) {
                            const uint32_t b = buf ^ (uint32_t)sub;
                            if (kt == 0) {
                                if (!mbar_wait(smem_u32(tempty + b), ((tph >> b) & 1u) ^ 1u,
                                               abort_flag, a.err, a.wait_cycles)) {
                                    ok = false;
                                    break;
                                }
                                tph ^= 1u << b;
                            }
                            const uint64_t xd = sdesc(smem_u32(ring_x + xs * kXBytes));
                            const uint32_t dacc = tmem + b * 256;
#pragma unroll
                            for (int j = 0; j < 4 * kSub; ++j) {
                                const int k = j >> 2;
                                if ((j & 3) == 0) {
                                    if ((sub == 0 &&
                                         !mbar_wait(smem_u32(pfull + ps * kSub + k), pph, abort_flag,
                                                    a.err, a.wait_cycles)) ||
                                        !mbar_wait(smem_u32(xfull + xs * kSub + k), xph, abort_flag,
                                                   a.err, a.wait_cycles)) {
                                        ok = false;
                                        break;
                                    }
                                    fence_after();
                                }
                                if (j < nk) {
                                    const uint64_t xa = xd + k * (kTileBytes >> 4) + 2 * (j & 3);
                                    const uint64_t pa = pd + k * (2 * kTileBytes >> 4) + 2 * (j & 3);
                                    if constexpr (F8)
                                        mma_f8kind(dacc, xa, pa, a.idesc, (kt | j) ? 1u : 0u);
                                    else
                                        mma_f16kind(dacc, xa, pa, a.idesc, (kt | j) ? 1u : 0u);
                                }
                            }
                            if (!ok) break;
                            if (last_k) {
                                mma_commit(smem_u32(done + b));
                            } else {
                                mma_commit(smem_u32(xempty + xs));
                                if (sub + 1 == nsub) mma_commit(smem_u32(pempty + ps));
                            }
                            if (++xs == kXSlots) {
                                xs = 0;
                                xph ^= 1u;
                            }
                        }
                        if (++ps == kPSlots) {
                            ps = 0;
                            pph ^= 1u;
                        }
                    }
                    buf ^= (uint32_t)(nsub & 1);
                }
            }
            // all MMAs issued by this thread complete before TMEM is released
            mma_commit(smem_u32(drain));
            const long long w0 = clock64();
            while (!mbar_try(smem_u32(drain), 0) && clock64() - w0 < kWaitCycles) {
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ------------------------------------------------ slot release: a finished
        // accumulation hands back the slots its last K stage read
        if (elect_one()) {
            int xs = 0, ps = 0;
            uint32_t dph = 0, buf = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const Unit w = unit_of(a, u);
                const int nsub = min(2, a.PT - 2 * w.pu);
                for (int f = w.f0; f < w.f1 && ok; ++f) {
                    // the last K stage's slots: nsub pattern slots a stage, one plan slot
                    xs = (xs + (a.KT - 1) * nsub) % kXSlots;
                    ps = (ps + a.KT - 1) % kPSlots;
                    for (int sub = 0; sub < nsub; ++sub) {
                        const uint32_t b = buf ^ (uint32_t)sub;
                        if (!mbar_wait(smem_u32(done + b), (dph >> b) & 1u, abort_flag, a.err,
                                       a.wait_cycles)) {
                            ok = false;
                            break;
                        }
                        dph ^= 1u << b;
                        mbar_arrive(smem_u32(xempty + xs));
                        if (sub + 1 == nsub) mbar_arrive(smem_u32(pempty + ps));
                        mbar_arrive(smem_u32(tempty + b));
                        xs = xs + 1 == kXSlots ? 0 : xs + 1;
                    }
                    ps = ps + 1 == kPSlots ? 0 : ps + 1;
                    buf ^= (uint32_t)(nsub & 1);
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue
        const int q = warp & 3;                  // TMEM lane quarter: patterns 16q .. 16q + 15
        const int zq = (warp - kEpi0) >> 2;      // axis columns 32 zq .. 32 zq + 31
        const float invN = 1.0f / (float)a.N;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + zq * 32;
        float ud[2][16];
#pragma unroll
        for (int j = 0; j < 16; ++j) ud[0][j] = ud[1][j] = 0.f;
        uint32_t dph = 0, buf = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
            const Unit w = unit_of(a, u);
            const int nsub = min(2, a.PT - 2 * w.pu);
            for (int f = w.f0; f < w.f1; ++f) {
                const float wf = (f == 0 || 2 * f == a.N) ? 1.f : 2.f;
#pragma unroll
                for (int sub = 0; sub < 2; ++sub) {
                    if (sub >= nsub) break;
                    const uint32_t b = buf ^ (uint32_t)sub;
                    if (!mbar_wait(smem_u32(done + b), (dph >> b) & 1u, abort_flag, a.err,
                                   a.wait_cycles)) {
                        ok = false;
                        break;
                    }
                    dph ^= 1u << b;
                    fence_after();
                    // two halves of 8 patterns (16 lanes each)
                    const uint32_t tb = tq + b * 256;
                    uint32_t R[16], I[16];
                    ACOM_TMEM_LD16x256_X4(tb, R);                          // (Xr, Xi) . Pr
                    ACOM_TMEM_LD16x256_X4(tb + 128, I);                    // (Xr, Xi) . Pi
                    ACOM_TMEM_WAIT32(R, I);
                    ACOM_ACCUMULATE(R, I, ud[sub], wf);
                    ACOM_TMEM_LD16x256_X4(tb + (16u << 16), R);
                    ACOM_TMEM_LD16x256_X4(tb + (16u << 16) + 128, I);
                    ACOM_TMEM_WAIT32(R, I);
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(tempty + b));
                    ACOM_ACCUMULATE(R, I, ud[sub] + 8, wf);
                }
                if (!ok) break;
                buf ^= (uint32_t)(nsub & 1);
            }
            if (!ok) break;
#pragma unroll
            for (int sub = 0; sub < 2; ++sub)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int b = (2 * w.pu + sub) * kNP + 8 * (2 * q + h) + (lane >> 2);
                    // FP16 spectra carry power-of-two scales: divide them out
                    const float sc = (a.xscale && b < a.nb)
                                         ? invN * a.inv_pscale / (a.xscale[b] * a.xs_mul)
                                         : invN * a.inv_pscale;
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int z = w.zt * kM + zq * 32 + 8 * n + 2 * (lane & 3) + e;
                            if (b < a.nb && z < a.Z)
                                *bound_at(a, w, b, z) = ud[sub][h * 8 + 2 * n + e] * sc;
                            ud[sub][h * 8 + 2 * n + e] = 0.f;
                        }
                }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols)
                     : "memory");
    }
}

constexpr size_t tc_smem_bytes() {
    return 1024 + (size_t)kPSlots * kPBytes + (size_t)kXSlots * kXBytes + 8 * kBars + 16;
}

// ---- FP32 operands as FP16 pairs.  x = hi + lo (hi = FP16(x), lo = FP16(x - hi)
// hold 22 bits and more of x), and a product of two is hi hi + hi lo + lo hi, so
// three MMAs stand in for FP32 multiply-adds that the CUDA cores run at 1/30 of
// the rate: 8,190 patterns x 903 axes 26.5 -> 3.7 ms (their match 29.4 -> 6.4 ms).  The tensor core
// truncates its FP32 accumulation, about 2^-25 a step downwards on a coherent
// sum (measured), so a K tile of 64 shells is an accumulation of its own: first
// the cross terms, 2^-11 of the rest, then four hi hi steps; the epilogue adds
// the two tiles' accumulators of a frequency rounding to nearest, and the sum
// over frequencies runs in groups of a quarter (a split tile's: a group a unit, added
// by add_groups).  The bound's error against FP64 is then no larger than the FP32
// kernel's with its one sum over all frequencies.  Relative 2-norms over whole and split
// tiles, 8 to 8,000 patterns of three kinds of peak lists, 66 to 1,378 axes: 1.1e-7 to
// 1.7e-7 against 3.0e-7 to 3.4e-7 on 150 shells and 360 bins, 0.9e-7 to 1.5e-7 against
// 2.0e-7 to 2.2e-7 on 75 and 180, 0.6e-7 to 1.4e-7 against 2.4e-7 to 3.1e-7 on 100 and 240
// and on 117 and 300; the same shares on a hexagonal crystal (split_shells says where not).
// With the up to 91 groups of a small batch of few axes added in one chain the 75 x 180
// plan was at 2.6e-7 against 2.0e-7.
// Roles and tiles as in k_contract_bound_tc.  A pattern slot holds a pattern
// tile's hi and lo of one K tile, a plan slot the axis tile's; both K tiles of a
// frequency stay for the second pattern tile.
#define ACOM_TMEM_LD16x256_X2(taddr, r)                                                      \
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"   \
                 : "=r"((r)[0]), "=r"((r)[1]), "=r"((r)[2]), "=r"((r)[3]), "=r"((r)[4]),     \
                   "=r"((r)[5]), "=r"((r)[6]), "=r"((r)[7])                                  \
                 : "r"(taddr))

__device__ __forceinline__ void add_pair2(uint32_t& a0, uint32_t& a1, uint32_t b0, uint32_t b1) {
    asm("{\n"
        ".reg .b64 A, B;\n"
        "mov.b64 A, {%0, %1};\n"
        "mov.b64 B, {%2, %3};\n"
        "add.rn.f32x2 A, A, B;\n"
        "mov.b64 {%0, %1}, A;\n"
        "}\n"
        : "+r"(a0), "+r"(a1)
        : "r"(b0), "r"(b1));
}

// a.Spad: columns of the hi half (the lo half follows); a.KT: K tiles, 1 or 2
__global__ void __launch_bounds__(kThreads, 1)
k_contract_bound_split(const __grid_constant__ CUtensorMap map_p,
                       const __grid_constant__ CUtensorMap map_x, TcArgs a, int flush) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* ring_p = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* ring_x = ring_p + kPSlots * kPBytes;
    uint64_t* xfull = reinterpret_cast<uint64_t*>(ring_x + kXSlots * kXBytes);   // [kXSlots]
    uint64_t* xempty = xfull + kXSlots;
    uint64_t* pfull = xempty + kXSlots;             // [kPSlots]
    uint64_t* pempty = pfull + kPSlots;
    uint64_t* done = pempty + kPSlots;              // [2] accumulation finished, per TMEM buffer
    uint64_t* tempty = done + 2;                    // [2] accumulator read (epilogue warps, warp 2)
    uint64_t* drain = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kXSlots; ++i) mbar_init(smem_u32(xfull + i), 1);
        for (int i = 0; i < kXSlots; ++i) mbar_init(smem_u32(xempty + i), 1);
        for (int i = 0; i < kPSlots; ++i) mbar_init(smem_u32(pfull + i), 1);
        for (int i = 0; i < kPSlots; ++i) mbar_init(smem_u32(pempty + i), 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(done + i), 1);
            mbar_init(smem_u32(tempty + i), kEpiWarps + 1);
        }
        mbar_init(smem_u32(drain), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_p)));
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)));
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int n_units = a.ts.units();
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        return mbar_wait(smem_u32(bar), parity, abort_flag, a.err, a.wait_cycles);
    };

    if (warp == 0 || warp == kProdP) {
        // ------------------------------------------------ TMA producers
        if (elect_one()) {
            const bool xprod = warp == 0;
            const int slots = xprod ? kXSlots : kPSlots;
            uint64_t* full = xprod ? xfull : pfull;
            uint64_t* empty = xprod ? xempty : pempty;
            int slot = 0;
            uint32_t phase = 0;          // parity of the slots' current use
            uint32_t used = 0, last = 0; // per slot: used at all, parity of its last use
            bool ok = true;
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const Unit w = unit_of(a, u);
                const int nsub = min(2, a.PT - 2 * w.pu);
                for (int f = w.f0; f < w.f1 && ok; ++f)
                    for (int sub = 0; sub < (xprod ? nsub : 1) && ok; ++sub)
                        for (int k = 0; k < a.KT; ++k) {
                            if (!(ok = wait(empty + slot, phase ^ 1u))) break;
                            const uint32_t fb = smem_u32(full + slot);
                            mbar_expect_tx(fb, (xprod ? 2 : 4) * kTileBytes);
#pragma unroll
                            for (int h = 0; h < 2; ++h)              // hi, lo
                                if (xprod)
                                    tma_load_2d(smem_u32(ring_x + slot * kXBytes + h * kTileBytes),
                                                &map_x, h * a.Spad + k * kKT,
                                                (f * a.PTs + 2 * w.pu + sub) * 128, fb);
                                else
                                    tma_load_2d(smem_u32(ring_p + slot * kPBytes + h * 2 * kTileBytes),
                                                &map_p, h * a.Spad + k * kKT,
                                                f * a.Zrows + w.zt * 256, fb);
                            used |= 1u << slot;
                            last = (last & ~(1u << slot)) | (phase << slot);
                            if (++slot == slots) {
                                slot = 0;
                                phase ^= 1u;
                            }
                        }
            }
            // every copy lands before the CTA's shared memory goes away
            for (int i = 0; i < slots; ++i)
                if (used & (1u << i)) {
                    const long long w0 = clock64();
                    while (!mbar_try(smem_u32(full + i), (last >> i) & 1u) &&
                           clock64() - w0 < kWaitCycles) {
                    }
                }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (elect_one()) {
            int xs = 0, pi = 0;                      // pattern slot, plan uses so far
            uint32_t xph = 0, tph = 0, buf = 0;      // tph: bit b, parity of buffer b's next use
            bool ok = true;
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const Unit w = unit_of(a, u);
                const int nsub = min(2, a.PT - 2 * w.pu);
                for (int f = w.f0; f < w.f1 && ok; ++f, pi += a.KT)
                    for (int sub = 0; sub < nsub && ok; ++sub)
                        for (int k = 0; k < a.KT; ++k) {
                            const int pu = pi + k, ps = pu % kPSlots;
                            if (!(ok = wait(tempty + buf, ((tph >> buf) & 1u) ^ 1u))) break;
                            tph ^= 1u << buf;
                            if ((sub == 0 && !wait(pfull + ps, (pu / kPSlots) & 1u)) ||
                                !wait(xfull + xs, xph)) {
                                ok = false;
                                break;
                            }
                            fence_after();
                            const int nk = min(kKT, a.Spad - k * kKT) >> 4;
                            const uint64_t xd = sdesc(smem_u32(ring_x + xs * kXBytes));
                            const uint64_t pd = sdesc(smem_u32(ring_p + ps * kPBytes));
                            const uint32_t dacc = tmem + buf * 256;
                            // hi lo, lo hi, then hi hi
#pragma unroll
                            for (int pass = 0; pass < 3; ++pass) {
                                const uint64_t xa = xd + (pass == 1 ? kTileBytes >> 4 : 0);
                                const uint64_t pa = pd + (pass == 0 ? 2 * kTileBytes >> 4 : 0);
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    if (j < nk)
                                        mma_f16kind(dacc, xa + 2 * j, pa + 2 * j, a.idesc,
                                                    (pass | j) ? 1u : 0u);
                            }
                            mma_commit(smem_u32(done + buf));
                            buf ^= 1u;
                            if (++xs == kXSlots) {
                                xs = 0;
                                xph ^= 1u;
                            }
                        }
            }
            // all MMAs issued by this thread complete before TMEM is released
            mma_commit(smem_u32(drain));
            const long long w0 = clock64();
            while (!mbar_try(smem_u32(drain), 0) && clock64() - w0 < kWaitCycles) {
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ------------------------------------------------ slot release
        if (elect_one()) {
            int xs = 0, pi = 0;
            uint32_t dph = 0, buf = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
                const Unit w = unit_of(a, u);
                const int nsub = min(2, a.PT - 2 * w.pu);
                for (int f = w.f0; f < w.f1 && ok; ++f, pi += a.KT)
                    for (int sub = 0; sub < nsub && ok; ++sub)
                        for (int k = 0; k < a.KT; ++k) {
                            if (!(ok = wait(done + buf, (dph >> buf) & 1u))) break;
                            dph ^= 1u << buf;
                            mbar_arrive(smem_u32(xempty + xs));
                            if (sub + 1 == nsub) mbar_arrive(smem_u32(pempty + (pi + k) % kPSlots));
                            mbar_arrive(smem_u32(tempty + buf));
                            xs = xs + 1 == kXSlots ? 0 : xs + 1;
                            buf ^= 1u;
                        }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue
        const int q = warp & 3;                  // TMEM lane quarter: patterns 16q .. 16q + 15
        const int zq = (warp - kEpi0) >> 2;      // axis columns 32 zq .. 32 zq + 31
        const float invN = 1.0f / (float)a.N;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + zq * 32;
        const bool two = a.KT == 2;
        float ud[2][16];
#pragma unroll
        for (int j = 0; j < 16; ++j) ud[0][j] = ud[1][j] = 0.f;
        uint32_t dph = 0, buf = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < n_units && ok; u += gridDim.x) {
            const Unit w = unit_of(a, u);
            const int nsub = min(2, a.PT - 2 * w.pu);
            int since = 0;                       // frequencies since the last flush
            for (int f = w.f0; f < w.f1; ++f) {
                const float wf = (f == 0 || 2 * f == a.N) ? 1.f : 2.f;
#pragma unroll
                for (int sub = 0; sub < 2; ++sub) {
                    if (sub >= nsub) break;
                    for (int k = 0; k < a.KT; ++k) {
                        const uint32_t b = buf ^ (uint32_t)k;
                        if (!wait(done + b, (dph >> b) & 1u)) {
                            ok = false;
                            break;
                        }
                        dph ^= 1u << b;
                    }
                    if (!ok) break;
                    fence_after();
                    const uint32_t tb = tq + buf * 256, t2 = tq + (buf ^ 1u) * 256;
                    // 8 patterns (16 lanes) x 16 axes at a time
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t o = ((uint32_t)(c >> 1) << 20) + 16u * (c & 1);
                        uint32_t V[16], W[16];               // (Xr, Xi) . Pr, (Xr, Xi) . Pi
                        ACOM_TMEM_LD16x256_X2(tb + o, V);
                        ACOM_TMEM_LD16x256_X2(tb + o + 128, V + 8);
                        if (two) {
                            ACOM_TMEM_LD16x256_X2(t2 + o, W);
                            ACOM_TMEM_LD16x256_X2(t2 + o + 128, W + 8);
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j) W[j] = 0u;
                        }
                        ACOM_TMEM_WAIT32(V, W);
                        if (c == 3) {
                            fence_before();
                            __syncwarp();
                            if (lane == 0) {
                                mbar_arrive(smem_u32(tempty + buf));
                                if (two) mbar_arrive(smem_u32(tempty + (buf ^ 1u)));
                            }
                        }
                        if (two)
#pragma unroll
                            for (int j = 0; j < 16; j += 2) add_pair2(V[j], V[j + 1], W[j], W[j + 1]);
#pragma unroll
                        for (int n = 0; n < 2; ++n) {
                            float* d = ud[sub] + 8 * (c >> 1) + 4 * (c & 1) + 2 * n;
                            accumulate_pair2(V[4 * n], V[4 * n + 1], V[4 * n + 2], V[4 * n + 3],
                                             V[8 + 4 * n], V[8 + 4 * n + 1], V[8 + 4 * n + 2],
                                             V[8 + 4 * n + 3], wf, d[0], d[1]);
                        }
                    }
                    if (!two) buf ^= 1u;
                }
                if (!ok) break;
                if (++since < flush && f + 1 < w.f1) continue;
                // the group's sum onto the earlier ones (this thread's own values)
                const bool first_group = f + 1 - since == w.f0;
                since = 0;
#pragma unroll
                for (int sub = 0; sub < 2; ++sub)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int b = (2 * w.pu + sub) * kNP + 8 * (2 * q + h) + (lane >> 2);
                        const float sc = b < a.nb ? invN * a.inv_pscale / a.xscale[b] : 0.f;
#pragma unroll
                        for (int n = 0; n < 4; ++n)
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const int z = w.zt * kM + zq * 32 + 8 * n + 2 * (lane & 3) + e;
                                if (b < a.nb && z < a.Z) {
                                    float* at = bound_at(a, w, b, z);
                                    const float v = ud[sub][h * 8 + 2 * n + e] * sc;
                                    *at = first_group ? v : *at + v;
                                }
                                ud[sub][h * 8 + 2 * n + e] = 0.f;
                            }
                    }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols)
                     : "memory");
    }
}

// ---- CTA pairs: a cluster of two CTAs computes each MMA together (cta_group::2,
// M = 256): CTA rank r holds pattern tile 2 p + r of the unit's two pattern
// tiles (its A rows) and half of the axis tile's B operand (rank 0 the real
// rows, rank 1 the imaginary rows); rank 0's two threads issue every MMA (even
// frequencies into TMEM buffer 0, odd into 1), whose accumulators land in both
// CTAs' tensor memory, lanes = the CTA's own patterns, columns = all 256 B
// rows, exactly as for a single CTA.  Both CTAs' copies complete on rank 0's full
// barriers (each issuer has its own per ring slot, so every full barrier has
// one consumer); commits arrive on both CTAs' barriers; both epilogues release
// rank 0's accumulator barrier.  A stage is one K tile of X and of the CTA's
// half of B (16 KB each).
constexpr int kPairStages = 6;
constexpr int kPairStageBytes = 2 * kTileBytes;

template <bool F8>
__global__ void __launch_bounds__(kThreads, 1)
k_contract_bound_pair(const __grid_constant__ CUtensorMap map_p,
                      const __grid_constant__ CUtensorMap map_x, TcArgs a) {
    constexpr int kSt = kPairStages;
    constexpr int kSB = kPairStageBytes;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment of the operand ring
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* ring = base;
    uint64_t* bars = reinterpret_cast<uint64_t*>(ring + kSt * kSB);
    uint64_t* full = bars;                      // [kIssuers][kSt]
    uint64_t* empty = bars + kIssuers * kSt;    // [kSt]
    uint64_t* tfull = empty + kSt;              // [kIssuers]
    uint64_t* tempty = tfull + kIssuers;        // [kIssuers]
    uint64_t* drain = tempty + kIssuers;        // [kIssuers]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + kIssuers);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;
    // the abort flag of the other CTA: a timeout stops both CTAs
    const uint32_t peer_abort = mapa_rank(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u);
    if (threadIdx.x == 0) {
        // a full barrier completes on the arrivals of the leading CTA's two
        // producers and the bytes of every copy of its stage
        for (int s = 0; s < kIssuers * kSt; ++s) mbar_init(smem_u32(full + s), 2);
        for (int s = 0; s < kSt; ++s) mbar_init(smem_u32(empty + s), 1);
        for (int b = 0; b < kIssuers; ++b) {
            mbar_init(smem_u32(tfull + b), 1);
            mbar_init(smem_u32(tempty + b), 2 * kEpiWarps);
            mbar_init(smem_u32(drain + b), 1);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_p)));
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)));
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    fence_before();
    cluster_sync_all();      // both CTAs' barriers exist before any copy or arrival
    fence_after();
    const uint32_t tmem = *tmem_slot;
    // units: axis tile x pair of pattern tiles, the CTAs taking a pattern tile each
    const int n_units = a.ts.units();
    const int u0 = (int)(blockIdx.x >> 1), ustep = (int)(gridDim.x >> 1);
    auto set_abort = [&]() { st_cluster_u32(peer_abort, 1u); };

    if (warp == 0 || warp == kProdP) {
        // ------------------------------------------------ TMA producers: warp 0
        // the pattern operand, warp kProdP the plan operand of every stage
        const bool xprod = warp == 0;
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            // per issuer and slot: the parity of the owner's next full phase;
            // the last stage issued into each slot and its owner, for the drain
            uint32_t fpar[kIssuers] = {0u, 0u};
            uint32_t issued_mask = 0, last_par = 0, last_own = 0;
            int fcount = 0;
            bool ok = true;
            for (int u = u0; u < n_units && ok; u += ustep) {
                const Unit w = unit_of(a, u);
                const int pt = 2 * w.pu + (int)rank;
                for (int f = w.f0; f < w.f1 && ok; ++f, ++fcount) {
                    // a CTA loads the real (rank 0) or imaginary rows of the axis tile
                    const int prow = f * a.Zrows + w.zt * 256 + 128 * (int)rank;
                    const int xrow = (f * a.PTs + pt) * 128;
                    const int own = fcount & 1;
                    for (int kt = 0; kt < a.KT; ++kt) {
                        if (!mbar_wait(smem_u32(empty + stage), phase ^ 1u, abort_flag, a.err,
                                       a.wait_cycles)) {
                            ok = false;
                            break;
                        }
                        const uint32_t fb = smem_u32(full + own * kSt + stage);
                        unsigned char* sbuf = ring + stage * kSB;
                        const int kbase = a.k0 + kt * (F8 ? kKT8 : kKT);
                        // every copy completes on the leading CTA's barrier, which
                        // expects both CTAs' bytes of its operand
                        const uint32_t fbl = mapa_rank(fb, 0);
                        if (leader) mbar_expect_tx(fb, 2 * kTileBytes);
                        if (xprod)
                            tma_load_2d_pair(smem_u32(sbuf), &map_x, kbase, xrow, fbl);
                        else
                            tma_load_2d_pair(smem_u32(sbuf + kTileBytes), &map_p, kbase, prow, fbl);
                        issued_mask |= 1u << stage;
                        const uint32_t par = (fpar[own] >> stage) & 1u;
                        last_par = (last_par & ~(1u << stage)) | (par << stage);
                        last_own = (last_own & ~(1u << stage)) | ((uint32_t)own << stage);
                        fpar[own] ^= 1u << stage;
                        if (++stage == kSt) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                }
            }
            if (!ok) {
                set_abort();
                if (leader) {
                    // let copies in flight land before the CTA's shared memory goes away
                    for (int s = 0; s < kSt; ++s)
                        if (issued_mask & (1u << s)) {
                            const uint32_t par = (last_par >> s) & 1u;
                            const int own = (last_own >> s) & 1u;
                            const long long w0 = clock64();
                            while (!mbar_try(smem_u32(full + own * kSt + s), par) &&
                                   clock64() - w0 < kWaitCycles) {
                            }
                        }
                } else {
                    // this CTA's copies complete on the other CTA's barriers: give
                    // them time to land (a copy takes microseconds)
                    const long long w0 = clock64();
                    while (clock64() - w0 < (1LL << 22)) {
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp <= kIssuers) {
        // ------------------------------------------------ MMA issuers (leading CTA)
        // issuer mi takes the frequencies with fcount % 2 == mi into TMEM
        // buffer mi; it walks the ring in the producer's order and waits only
        // on its own full barriers
        const int mi = warp - 1;
        if (lane == 0 && leader) {
            int stage = 0;
            uint32_t fpar = 0;           // bit s: parity of this issuer's next phase of slot s
            uint32_t tph = 0;
            int fcount = 0;
            bool ok = true;
            uint64_t* myfull = full + mi * kSt;
            for (int u = u0; u < n_units && ok; u += ustep) {
                const Unit w = unit_of(a, u);
                for (int f = w.f0; f < w.f1 && ok; ++f, ++fcount) {
                    if ((fcount & 1) != mi) {
                        stage = (stage + a.KT) % kSt;
                        continue;
                    }
                    if (!mbar_wait(smem_u32(tempty + mi), tph ^ 1u, abort_flag, a.err,
                                   a.wait_cycles)) {
                        ok = false;
                        break;
                    }
                    tph ^= 1u;
                    fence_after();
                    const uint32_t dacc = tmem + mi * 256;
                    for (int kt = 0; kt < a.KT; ++kt) {
                        const uint32_t spar = (fpar >> stage) & 1u;
                        fpar ^= 1u << stage;
                        const uint32_t sb = smem_u32(ring + stage * kSB);
                        // K steps of 32 bytes inside the shells (16 16-bit or 32
                        // 8-bit elements; the tail of the last tile is TMA zero
                        // fill); a step moves the descriptors' start address by
                        // 32 bytes (2 units of 16)
                        constexpr int ktel = F8 ? kKT8 : kKT;
                        const int nk = (min(ktel, a.Spad - a.k0 - kt * ktel) * (F8 ? 1 : 2) + 31) >> 5;
                        if (!mbar_wait(smem_u32(myfull + stage), spar, abort_flag, a.err,
                                       a.wait_cycles)) {
                            ok = false;
                            break;
                        }
                        fence_after();
                        const uint64_t xa = sdesc(sb), pb = sdesc(sb + kTileBytes);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (j < nk) {
                                if constexpr (F8)
                                    mma_f8kind_pair(dacc, xa + 2 * j, pb + 2 * j, a.idesc, (kt | j) ? 1u : 0u);
                                else
                                    mma_f16kind_pair(dacc, xa + 2 * j, pb + 2 * j, a.idesc, (kt | j) ? 1u : 0u);
                            }
                        mma_commit_pair_both(smem_u32(empty + stage));     // frees the stage in both CTAs
                        if (++stage == kSt) stage = 0;
                    }
                    if (ok) mma_commit_pair_both(smem_u32(tfull + mi));    // accumulators ready
                }
            }
            if (!ok) set_abort();
            // all MMAs issued by this thread complete before TMEM is released
            mma_commit_pair(smem_u32(drain + mi));
            const long long w0 = clock64();
            while (!mbar_try(smem_u32(drain + mi), 0) && clock64() - w0 < kWaitCycles) {
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue
        const int q = warp & 3;                  // TMEM lane quarter: patterns 16q .. 16q + 15
        const int zq = (warp - kEpi0) >> 2;      // axis columns 32 zq .. 32 zq + 31
        const float invN = 1.0f / (float)a.N;
        float ud[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) ud[j] = 0.f;
        uint32_t tph[2] = {0, 0};
        int fcount = 0;
        bool ok = true;
        // the accumulator barriers live in the leading CTA
        const uint32_t tempty_l[2] = {mapa_rank(smem_u32(tempty), 0),
                                      mapa_rank(smem_u32(tempty + 1), 0)};
        for (int u = u0; u < n_units && ok; u += ustep) {
            const Unit w = unit_of(a, u);
            const int pt = 2 * w.pu + (int)rank;
            for (int f = w.f0; f < w.f1; ++f, ++fcount) {
                const int buf = fcount & 1;
                if (!mbar_wait(smem_u32(tfull + buf), tph[buf], abort_flag, a.err, a.wait_cycles)) {
                    ok = false;
                    break;
                }
                tph[buf] ^= 1u;
                fence_after();
                const float wf = (f == 0 || 2 * f == a.N) ? 1.f : 2.f;
                const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + buf * 256 + zq * 32;
                // two halves of 8 patterns (16 lanes each); the second half's
                // loads are in flight while the first is reduced
                uint32_t R0[16], I0[16], R1[16], I1[16];
                ACOM_TMEM_LD16x256_X4(tb, R0);                          // (Xr, Xi) . Pr
                ACOM_TMEM_LD16x256_X4(tb + 128, I0);                    // (Xr, Xi) . Pi
                ACOM_TMEM_WAIT32(R0, I0);
                ACOM_TMEM_LD16x256_X4(tb + (16u << 16), R1);
                ACOM_TMEM_LD16x256_X4(tb + (16u << 16) + 128, I1);
                ACOM_ACCUMULATE(R0, I0, ud, wf);
                ACOM_TMEM_WAIT32(R1, I1);
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(tempty_l[buf]);
                ACOM_ACCUMULATE(R1, I1, ud + 8, wf);
            }
            if (!ok) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int b = pt * kNP + 8 * (2 * q + h) + (lane >> 2);
                // FP16 spectra carry power-of-two scales: divide them out
                const float sc = (a.xscale && b < a.nb)
                                     ? invN * a.inv_pscale / (a.xscale[b] * a.xs_mul)
                                     : invN * a.inv_pscale;
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int z = w.zt * kM + zq * 32 + 8 * n + 2 * (lane & 3) + e;
                        if (b < a.nb && z < a.Z) *bound_at(a, w, b, z) = ud[h * 8 + 2 * n + e] * sc;
                        ud[h * 8 + 2 * n + e] = 0.f;
                    }
            }
        }
        if (!ok && lane == 0) set_abort();
    }
    fence_before();
    cluster_sync_all();      // the leading CTA's MMAs and every copy are done in both CTAs
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols)
                     : "memory");
    }
}

constexpr size_t pair_smem_bytes() {
    return 1024 + (size_t)kPairStages * kPairStageBytes +
           8 * ((kIssuers + 1) * kPairStages + 3 * kIssuers) + 16;
}

}  // namespace tc

// ---------------------------------------------------------------------------
// host side: tensor maps and launch
// ---------------------------------------------------------------------------

static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

static bool get_encoder() {
    if (g_encode) return true;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
        return false;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return true;
}

// 2-D operand map: rows x cols (cols contiguous), boxes of 128 bytes x box_rows
// rows (64 16-bit or 128 8-bit columns), 128-byte swizzle; boxes reaching
// past the last column are zero-filled.  kind: 0 BF16, 1 FP16, 2 E4M3 (as
// bytes).
acom_status make_bf16_map(void* map_storage, const void* base, uint64_t rows, uint64_t cols,
                          int kind, int box_rows) {
    if (!get_encoder()) return set_error(ACOM_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    const uint64_t eb = kind == 2 ? 1 : 2;
    if ((cols * eb) % 16 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0)
        return set_error(ACOM_ERR_INVALID_ARG, "tensor map: stride or base not 16-byte aligned");
    CUtensorMap* m = reinterpret_cast<CUtensorMap*>(map_storage);
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * eb};
    if (box_rows < 8 || box_rows > 256 || box_rows % 8 != 0)
        return set_error(ACOM_ERR_INVALID_ARG, "tensor map: unsupported box");
    const cuuint32_t box[2] = {(cuuint32_t)(kind == 2 ? tc::kKT8 : tc::kKT), (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapDataType dt = kind == 2   ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                   : kind == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                               : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    CUresult r = g_encode(m, dt, 2, const_cast<void*>(base), dims,
                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(ACOM_ERR_CUDA, "cuTensorMapEncodeTiled failed");
    return ACOM_OK;
}

size_t tensor_map_bytes() { return sizeof(CUtensorMap); }

// Budget of the contraction's pipeline waits (acom_set_device_wait_limit);
// 0: the default of about 2 s.  Process-global.
static long long g_wait_cycles = 0;
void set_wait_cycles(long long cycles) { g_wait_cycles = cycles > 0 ? cycles : 0; }

// The tiles of full waves run whole.  The tiles of the last, partial wave (all
// tiles of a small batch) are split over the frequencies into as many groups as
// fill the SMs: a CTA runs a tile's frequencies in turn, so a wave of few tiles
// would take as long as a full one.  1-degree plan: one pattern (8 tiles, 19
// groups) 174 -> 27 us; 4,095 patterns (256 tiles, the last 104 too many to
// split) 676 -> 515 us, from the larger tile.
TileSplit tc_split(const acom_plan_s* p, int nb, int tile_order, bool split) {
    TileSplit ts;
    ts.zmajor = tile_order == 1 ? 1 : 0;
    ts.ZT = p->Zp / tc::kM;
    ts.PTu = (nb + 2 * tc::kNP - 1) / (2 * tc::kNP);
    ts.lb = ts.lz = 7;
    ts.set(sm_count(), sm_count(), p->F, split);
    return ts;
}

void launch_contract_bound_tc(const acom_plan_s* p, const void* map_x, int pt_stride, int nb,
                              const TileSplit& ts, float* U, float* extra, cudaStream_t st,
                              const float* xscale, int cta_pairs) {
    tc::TcArgs a;
    a.ts = ts;
    a.F = p->F;
    a.N = p->N;
    a.Z = p->Z;
    a.nb = nb;
    a.ZT = ts.ZT;
    a.PT = (nb + tc::kNP - 1) / tc::kNP;
    a.PTs = pt_stride;
    const bool f8 = p->precision == ACOM_PREC_FP8;
    const int ktel = f8 ? tc::kKT8 : tc::kKT;
    // the K range starts at the plan's first non-zero shell (a multiple of 16);
    // KT stages of `sub` K tiles each per frequency
    a.k0 = p->k0;
    auto stages = [&](int sub) { return (p->Spad - p->k0 + ktel * sub - 1) / (ktel * sub); };
    a.Spad = p->Spad;
    a.Zrows = 2 * p->Zp;
    a.U = U;
    a.extra = extra;
    a.err = p->err;
    // E4M3 is format 0 for A and B, the same bits as F16
    a.idesc = p->precision == ACOM_PREC_BF16 ? tc::kIdescBF16 : tc::kIdescF16;
    a.xscale = xscale;
    a.xs_mul = f8 ? kFp8Shift : 1.0f;
    a.inv_pscale = 1.0f / p->pscale;
    a.wait_cycles = g_wait_cycles > 0 ? g_wait_cycles : tc::kWaitCycles;
    const int nsm = sm_count();
    const int n_units = ts.units();
    if (n_units <= 0) return;
    const CUtensorMap& mx = *reinterpret_cast<const CUtensorMap*>(map_x);
    if (cta_pairs && nsm >= 2) {
        // CTA pairs: M = 256 (the pair's two pattern tiles), each CTA loading
        // half of the 256 B rows (128-row boxes)
        a.idesc = (a.idesc & ~(0x1Fu << 24)) | ((256u >> 4) << 24);
        a.KT = stages(1);
        const size_t smem = tc::pair_smem_bytes();
        auto kern = f8 ? tc::k_contract_bound_pair<true> : tc::k_contract_bound_pair<false>;
        set_max_dynamic_smem((const void*)kern, smem);
        const int clusters = n_units < nsm / 2 ? n_units : nsm / 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * clusters, 1, 1);
        cfg.blockDim = dim3(tc::kThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        prof_begin(kKContractBf16, st);
        cudaLaunchKernelEx(&cfg, kern, *reinterpret_cast<const CUtensorMap*>(p->map_p128), mx, a);
        prof_end(kKContractBf16, st);
        return;
    }
    a.KT = stages(tc::kSub);
    const size_t smem = tc::tc_smem_bytes();
    auto kern = f8 ? tc::k_contract_bound_tc<true> : tc::k_contract_bound_tc<false>;
    set_max_dynamic_smem((const void*)kern, smem);
    prof_begin(kKContractBf16, st);
    kern<<<n_units < nsm ? n_units : nsm, tc::kThreads, smem, st>>>(
        *reinterpret_cast<const CUtensorMap*>(p->map_p), mx, a);
    prof_end(kKContractBf16, st);
}

// Shells of the split operands, 0 when the plan keeps the CUDA cores: where the error
// against FP64 is not clearly below the FP32 kernel's.  More than two K tiles need more
// than four hi hi steps per accumulation (eight on all-positive spectra: 4.8e-7 against
// 2.4e-7).  With few bins the FP32 kernel's sum over the few frequencies rounds as little
// as the truncation does: up to 0.99 of its error at 100 bins (1.46e-7 against 1.46e-7), 0.94
// at 72, 0.87 at 144, 0.81 at 160, and at most 0.72 from 180 bins on.
int split_shells(const acom_plan_s* p) {
    const int K = (p->S - p->k0 + 15) / 16 * 16;
    const bool smaller_error = K > 0 && K <= 2 * tc::kKT && p->N >= 180;
    return p->precision == ACOM_PREC_FP32 && smaller_error ? K : 0;
}

void launch_contract_bound_split(const acom_plan_s* p, const void* map_x, int pt_stride, int nb,
                                 const TileSplit& ts, float* U, float* extra, cudaStream_t st,
                                 const float* xscale) {
    tc::TcArgs a{};
    a.ts = ts;
    a.F = p->F;
    a.N = p->N;
    a.Z = p->Z;
    a.nb = nb;
    a.ZT = ts.ZT;
    a.PT = (nb + tc::kNP - 1) / tc::kNP;
    a.PTs = pt_stride;
    a.Spad = p->ks;
    a.KT = (p->ks + tc::kKT - 1) / tc::kKT;
    a.Zrows = 2 * p->Zp;
    a.U = U;
    a.extra = extra;
    a.err = p->err;
    a.idesc = tc::kIdescF16;
    a.xscale = xscale;
    a.inv_pscale = 1.0f / fp16_plan_scale(p->N);
    a.wait_cycles = g_wait_cycles > 0 ? g_wait_cycles : tc::kWaitCycles;
    const int n_units = ts.units();
    if (n_units <= 0) return;
    const size_t smem = tc::tc_smem_bytes();
    set_max_dynamic_smem((const void*)tc::k_contract_bound_split, smem);
    prof_begin(kKContract, st);
    tc::k_contract_bound_split<<<std::min(n_units, sm_count()), tc::kThreads, smem, st>>>(
        *reinterpret_cast<const CUtensorMap*>(p->map_ps),
        *reinterpret_cast<const CUtensorMap*>(map_x), a, (p->F + 3) / 4);
    prof_end(kKContract, st);
}

__device__ __forceinline__ void split_half(float x, __half& hi, __half& lo) {
    hi = __float2half_rn(x);
    lo = __float2half_rn(x - __half2float(hi));
}

// plan rows -> [F][Zp / 128][256][2 K], hi then lo of scale times the spectra on the
// shells from k0 on; a warp per row
__global__ void k_plan_split(const float* __restrict__ Pr, const float* __restrict__ Pi, int Zp, int F,
                             int Spad, int k0, int K, float scale, __half* __restrict__ dst) {
    const int lane = threadIdx.x & 31;
    const int64_t orow = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int ZT = Zp / 128;
    if (orow >= (int64_t)F * ZT * 256) return;
    const int row = (int)(orow % 256), zt = (int)(orow / 256 % ZT), f = (int)(orow / 256 / ZT);
    const float* src = (row < 128 ? Pr : Pi) + ((int64_t)(zt * 128 + (row & 127)) * F + f) * Spad + k0;
    __half* d = dst + orow * 2 * K;
    for (int s = lane; s < K; s += 32) split_half(scale * src[s], d[s], d[K + s]);
}

void launch_plan_split(const acom_plan_s* p, cudaStream_t st) {
    const int64_t rows = (int64_t)p->F * p->Zp * 2;
    prof_begin(kKMisc, st);
    k_plan_split<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(
        p->Pr, p->Pi, p->Zp, p->F, p->Spad, p->k0, p->ks, fp16_plan_scale(p->N),
        reinterpret_cast<__half*>(p->Ps));
    prof_end(kKMisc, st);
}

// the patterns' shell-major rows -> [F][PTs][128][2 K] (16-row groups: 8 patterns'
// real rows, their imaginary rows), hi then lo of 2^e X^, through 32 x 32 tiles in
// shared memory; rows outside the pattern's mask as zeros
__global__ void __launch_bounds__(256)
k_rows_to_split(const float* __restrict__ sre, const float* __restrict__ sim,
                const uint32_t* __restrict__ rmask, const float* __restrict__ xscale, int F, int Spad,
                int k0, int K, int PTs, __half* __restrict__ dst) {
    __shared__ float tr[32][33], ti[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t item = blockIdx.x;
    const int f0 = blockIdx.y * 32, Fs = shell_row_stride(F), MW = Spad >> 5;
    const float sc = xscale[item];
    const int64_t row0 = (item >> 6) * 128 + ((item & 63) >> 3) * 16 + (item & 7);
    for (int s0 = 0; s0 < K; s0 += 32) {
        for (int r = warp; r < 32; r += 8) {
            const int s = k0 + s0 + r;
            const bool in = s0 + r < K && f0 + lane < Fs && (rmask[item * MW + (s >> 5)] >> (s & 31) & 1u);
            const int64_t o = (item * Spad + s) * (int64_t)Fs + f0 + lane;
            tr[r][lane] = in ? sre[o] : 0.f;
            ti[r][lane] = in ? sim[o] : 0.f;
        }
        __syncthreads();
        for (int r = warp; r < 32 && f0 + r < F; r += 8) {
            if (s0 + lane < K) {
                __half* d = dst + ((int64_t)(f0 + r) * PTs * 128 + row0) * 2 * K + s0 + lane;
                split_half(sc * tr[lane][r], d[0], d[K]);
                d += (int64_t)16 * K;                    // 8 rows on: the imaginary parts
                split_half(sc * ti[lane][r], d[0], d[K]);
            }
        }
        __syncthreads();
    }
}

void launch_rows_to_split(const acom_plan_s* p, const float* sre, const float* sim,
                          const uint32_t* rmask, const float* xscale, int items, int PTs, void* dst,
                          cudaStream_t st) {
    if (items <= 0) return;
    prof_begin(kKMisc, st);
    k_rows_to_split<<<dim3((unsigned)items, (unsigned)((p->F + 31) / 32)), 256, 0, st>>>(
        sre, sim, rmask, xscale, p->F, p->Spad, p->k0, p->ks, PTs, reinterpret_cast<__half*>(dst));
    prof_end(kKMisc, st);
}

// FP32 spectra [Zp][F][Spad] (real and imaginary arrays) -> the merged
// tensor-core operand [F][Zp / 128][256][Spad]: per frequency and 128-axis
// tile, the 128 real rows then the 128 imaginary rows, BF16 / FP16 / E4M3 of
// scale x (a power of two, exact in FP32).
template <class T>
__device__ __forceinline__ T to_half_type(float x);
template <>
__device__ __forceinline__ __nv_bfloat16 to_half_type<__nv_bfloat16>(float x) {
    return __float2bfloat16_rn(x);
}
template <>
__device__ __forceinline__ __half to_half_type<__half>(float x) {
    return __float2half_rn(x);
}
template <>
__device__ __forceinline__ __nv_fp8_e4m3 to_half_type<__nv_fp8_e4m3>(float x) {
    return __nv_fp8_e4m3(x);           // round to nearest, saturating to +-448
}

// One pass from the raster's rows to every layout of the plan (launch_plan_layouts):
// a CTA takes 32 frequencies of one axis, 32 shells at a time through shared memory,
// so each array is read or written once in whole lines.  Bound by memory: 903 axes x
// 150 shells x 181 frequencies 0.2 GB in, 0.6 GB out.  It replaced a scaling pass over
// both layouts, the raster's 8-byte frequency-major stores, three passes for the
// norms, the mask and the operand, and 0.95 GB of clearing: after the reflections the
// plan's build took 0.98 ms of the GPU and now 0.35.  A warp loads its four rows of the
// next tile together while this one is stored (one row at a time, each load waited
// through the mask's vote: 276 us, now 200).  T void: no operand.
template <class T>
__global__ void __launch_bounds__(256)
k_plan_layouts(const float* __restrict__ sumsq, int Z, int ZT, int F, int Spad,
               float* __restrict__ sre, float* __restrict__ sim, float* __restrict__ re,
               float* __restrict__ im, T* __restrict__ op, float scale,
               uint32_t* __restrict__ smask, float* __restrict__ fmax) {
    __shared__ float tr[32][33], ti[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int z = blockIdx.x, f0 = blockIdx.y * 32, Fs = shell_row_stride(F);
    const bool real_axis = z < Z;
    const float ss = real_axis ? sumsq[z] : 0.f;
    const float a = ss > 0.f ? rsqrtf(ss) : 0.f;
    float nrm[4] = {0.f, 0.f, 0.f, 0.f};      // of frequencies f0 + warp + 8 j, lanes over shells
    const bool in_row = f0 + lane < Fs;
    float u[4], v[4];                         // the next tile's rows warp + 8 j, loads in flight
    auto load = [&](int s0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t o = ((int64_t)z * Spad + s0 + warp + 8 * j) * Fs + f0 + lane;
            const bool get = real_axis && in_row;
            u[j] = get ? sre[o] : 0.f;
            v[j] = get ? sim[o] : 0.f;
        }
    };
    load(0);
    for (int s0 = 0; s0 < Spad; s0 += 32) {
        uint32_t rows = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = warp + 8 * j;
            const float x = u[j] * a, y = v[j] * a;
            tr[r][lane] = x;
            ti[r][lane] = y;
            if (in_row) {
                const int64_t o = ((int64_t)z * Spad + s0 + r) * Fs + f0 + lane;
                sre[o] = x;
                sim[o] = y;
            }
            if (__any_sync(0xffffffffu, x != 0.f || y != 0.f)) rows |= 1u << r;
        }
        if (rows && lane == 0) atomicOr(smask + (int64_t)z * (Spad >> 5) + (s0 >> 5), rows);
        if (s0 + 32 < Spad) load(s0 + 32);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int f = f0 + warp + 8 * j;
            if (f < F) {
                const float x = tr[lane][warp + 8 * j], y = ti[lane][warp + 8 * j];
                const int64_t o = ((int64_t)z * F + f) * Spad + s0 + lane;
                re[o] = x;
                im[o] = y;
                nrm[j] = fmaf(x, x, fmaf(y, y, nrm[j]));
                if constexpr (!std::is_void<T>::value) {
                    T* d = op + (((int64_t)f * ZT + (z >> 7)) * 256 + (z & 127)) * Spad + s0 + lane;
                    d[0] = to_half_type<T>(scale * x);
                    d[(int64_t)128 * Spad] = to_half_type<T>(scale * y);
                }
            }
        }
        __syncthreads();
    }
    // max over axes of the norm over shells, times 1.0001 for its rounding: non-negative
    // floats order like their bit patterns
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float n = nrm[j];
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        const int f = f0 + warp + 8 * j;
        if (lane == 0 && f < F) atomicMax(reinterpret_cast<int*>(fmax) + f, __float_as_int(sqrtf(n) * 1.0001f));
    }
}

template <class T>
static void run_plan_layouts(const acom_plan_s* p, const float* sumsq, cudaStream_t st) {
    const dim3 grid((unsigned)p->Zp, (unsigned)((p->F + 31) / 32));
    k_plan_layouts<T><<<grid, 256, 0, st>>>(sumsq, p->Z, p->Zp / 128, p->F, p->Spad, p->Psr, p->Psi,
                                            p->Pr, p->Pi, reinterpret_cast<T*>(p->Pb), p->pscale,
                                            p->smask, p->pfmax);
}

void launch_plan_layouts(const acom_plan_s* p, const float* sumsq, cudaStream_t st) {
    cudaMemsetAsync(p->smask, 0, sizeof(uint32_t) * (size_t)p->Zp * (p->Spad / 32), st);
    cudaMemsetAsync(p->pfmax, 0, sizeof(float) * (size_t)p->F, st);
    prof_begin(kKScale, st);
    if (!p->Pb)
        run_plan_layouts<void>(p, sumsq, st);
    else if (tc_kind(p->precision) == 2)
        run_plan_layouts<__nv_fp8_e4m3>(p, sumsq, st);
    else if (tc_kind(p->precision) == 1)
        run_plan_layouts<__half>(p, sumsq, st);
    else
        run_plan_layouts<__nv_bfloat16>(p, sumsq, st);
    prof_end(kKScale, st);
}

template <class T>
__global__ void k_plan_to_operand(const float* __restrict__ Pr, const float* __restrict__ Pi,
                                  int Zp, int F, int Spad, T* __restrict__ dst, float scale) {
    // one warp per operand row (f, zt, row): row < 128 takes the real part of
    // axis zt 128 + row, row >= 128 the imaginary part of axis zt 128 + row - 128;
    // lanes over the shells, four at a time (Spad is a multiple of 32)
    const int lane = threadIdx.x & 31;
    const int64_t orow = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int ZT = Zp / 128;
    if (orow >= (int64_t)F * ZT * 256) return;
    const int row = (int)(orow % 256);
    const int64_t t = orow / 256;
    const int zt = (int)(t % ZT), f = (int)(t / ZT);
    const int z = zt * 128 + (row & 127);
    const float4* src = reinterpret_cast<const float4*>((row < 128 ? Pr : Pi) +
                                                        ((int64_t)z * F + f) * Spad);
    T* d = dst + orow * Spad;
    for (int q = lane; q < Spad / 4; q += 32) {
        const float4 v = src[q];
        d[4 * q] = to_half_type<T>(scale * v.x);
        d[4 * q + 1] = to_half_type<T>(scale * v.y);
        d[4 * q + 2] = to_half_type<T>(scale * v.z);
        d[4 * q + 3] = to_half_type<T>(scale * v.w);
    }
}

void launch_plan_to_operand(const float* Pr, const float* Pi, int Zp, int F, int Spad, void* dst,
                            cudaStream_t st, int kind, float scale) {
    const int64_t rows = (int64_t)F * (Zp / 128) * 256;        // one warp per row
    const unsigned blocks = (unsigned)((rows + 7) / 8);
    prof_begin(kKMisc, st);
    if (kind == 2)
        k_plan_to_operand<__nv_fp8_e4m3><<<blocks, 256, 0, st>>>(
            Pr, Pi, Zp, F, Spad, reinterpret_cast<__nv_fp8_e4m3*>(dst), scale);
    else if (kind == 1)
        k_plan_to_operand<__half><<<blocks, 256, 0, st>>>(Pr, Pi, Zp, F, Spad,
                                                           reinterpret_cast<__half*>(dst), scale);
    else
        k_plan_to_operand<__nv_bfloat16><<<blocks, 256, 0, st>>>(
            Pr, Pi, Zp, F, Spad, reinterpret_cast<__nv_bfloat16*>(dst), 1.0f);
    prof_end(kKMisc, st);
}

// FP16 operand rows -> E4M3 rows times mul (a power of two, exact), 8 per thread.
__global__ void k_half_to_e4m3(const __half* __restrict__ src, uint8_t* __restrict__ dst,
                               int64_t n8, float mul) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint4 v = reinterpret_cast<const uint4*>(src)[i];
        const __half2* h = reinterpret_cast<const __half2*>(&v);
        uint16_t o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 f = __half22float2(h[j]);
            f.x *= mul;
            f.y *= mul;
            o[j] = (uint16_t)__nv_cvt_float2_to_fp8x2(f, __NV_SATFINITE, __NV_E4M3);
        }
        reinterpret_cast<uint2*>(dst)[i] = *reinterpret_cast<const uint2*>(o);
    }
}

void launch_half_to_e4m3(const void* src, void* dst, int64_t n, float mul, cudaStream_t st) {
    const int64_t n8 = n / 8;
    if (n8 <= 0) return;
    const int blocks = (int)std::min<int64_t>((n8 + 255) / 256, 152 * 32);
    prof_begin(kKMisc, st);
    k_half_to_e4m3<<<blocks, 256, 0, st>>>(reinterpret_cast<const __half*>(src),
                                            reinterpret_cast<uint8_t*>(dst), n8, mul);
    prof_end(kKMisc, st);
}

}  // namespace acom
