// Device code of the swap-potential step: cell-sorted Verlet list build,
// the per-centre S pass, the force pass fused with the integrator, and the
// persistent cooperative kernel that runs many time steps per launch.
//
// Method (Ciarella & Ellenbroek, section "The swap potential"):
//   two-body term  v(r) = 4 eps [(sigma/r)^(2n) - (sigma/r)^n]       (Eq. 2b)
//   normalised     vh(r) = 1 (r <= r_min), -v(r)/eps (r > r_min)       (Eq. pot)
//   three-body     v3_ijk = lambda eps vh_ij vh_ik, centre i           (Eq. 3bp)
// With a = sqrt(lambda eps) and S_i = sum_k a_ik vh_ik over the reactive
// partners of i, the three-body energy of centre i is
//   sum_{j<k} a_ij a_ik vh_ij vh_ik = 1/2 sum_j a_ij vh_ij (S_i - a_ij vh_ij)
// and dU3/dvh_ij = a_ij [(S_i - a_ij vh_ij) + (S_j - a_ij vh_ij)], so the
// triplet sum costs O(neighbours) once S is known for every particle: one
// pass forms S, the next forms every pair force from S_i and S_j.  Beyond
// r_min, vh' = -v'/eps_hat, so the total force of a reactive pair is the
// two-body force times (1 - dU3/dvh_ij / eps_hat).
//
// This file is compiled several times: with SWP_BATCHED 0 into namespace
// swp::single (the single-system step kernel and the exchange kernels; see
// swp_launch.cuh) and with SWP_BATCHED 1 into one namespace per block shape
// of the batched kernel (SWP_BATCH_NS, SWP_BATCH_THREADS threads per block,
// SWP_BATCH_MINB blocks per SM in its launch bounds; see swp_batch_impl.cuh),
// so that the code a group of one block or a group of fewer blocks than
// thermo quantities needs costs the single-system kernel nothing.

#include <type_traits>

#include "swp_internal.h"

#ifndef SWP_BATCHED
#error "define SWP_BATCHED (0 or 1) before including swp_kernels.cuh"
#endif

// With SWP_BATCHED 0 and SWP_WIDE 1 it is compiled into namespace swp::wide:
// the single-system step kernel with 1024-thread blocks (two-barrier step
// only), which bonded networks run, whose gathers' latency is hidden better
// with more warps, and unbonded FP32 systems of 769 to 1,024 particles per block,
// which are one row per thread there.  That copy leaves out the resident step and
// the exchange kernels.
#undef SWP_HAS_RESIDENT
#if !SWP_BATCHED && !SWP_WIDE
#define SWP_HAS_RESIDENT 1
#else
#define SWP_HAS_RESIDENT 0
#endif

namespace swp {
#if SWP_BATCHED
#if !defined(SWP_BATCH_NS) || !defined(SWP_BATCH_THREADS) || !defined(SWP_BATCH_MINB)
#error "define SWP_BATCH_NS, SWP_BATCH_THREADS and SWP_BATCH_MINB with SWP_BATCHED 1"
#endif
namespace SWP_BATCH_NS {
#elif SWP_WIDE
namespace wide {
#else
namespace single {
#endif

constexpr bool kBatched = SWP_BATCHED != 0;
// The list rebuild is kept out of line in the batched kernel: inlined, its
// register needs spread into the step loop (whose per-system descriptors come
// from shared memory there, not the parameter bank) and cost spills.
#undef SWP_COLD
#if SWP_BATCHED
#define SWP_COLD __noinline__
#else
#define SWP_COLD
#endif
// Threads per block.  The batched kernel reads every system's descriptors from
// shared memory rather than the constant bank; its block shapes trade
// registers per thread (spills at 1024 threads, 64 registers) against warps
// per SM, and SwapBatch.autotune times them on the batch at hand.  The
// single-system kernel runs 768 threads in FP32 (80 registers: its resident step
// keeps a thread's row, the integrator's state and the pair arithmetic in
// registers at once) and 512 in FP64 (128 registers: eight warps fill the FP64
// pipe, and spills cost more than more warps bring).  FP64 batches and networks
// exist with 1,024 threads only.
#if SWP_BATCHED
constexpr int kThreads = SWP_BATCH_THREADS;
constexpr int kMinBlocks = SWP_BATCH_MINB;
#elif SWP_WIDE
constexpr int kThreads = kBlockWide;
#else
constexpr int kThreads = SWP_BLOCK;
#endif

// ---------------------------------------------------------------------------
// Group of blocks that advances one system: the whole grid for a single
// system; in a batched launch, the blocks given to that system (possibly one).
// Every phase partitions its work over the group, and grid barriers are
// barriers over the group.
#if SWP_BATCHED
static __shared__ int s_grp[2];  // [0] this block's rank in the group, [1] group size
__device__ __forceinline__ int g_rank() { return s_grp[0]; }
__device__ __forceinline__ int g_size() { return s_grp[1]; }
#else
__device__ __forceinline__ int g_rank() { return blockIdx.x; }
__device__ __forceinline__ int g_size() { return gridDim.x; }
#endif

// ---------------------------------------------------------------------------
// Small helpers

__device__ __forceinline__ long long gtimer_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int ld_relaxed(const int* p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// IEEE operations with one rounding each and no contraction, for the
// distance decisions that must be reproducible bit for bit.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }

__device__ __forceinline__ int packed_of(float w) { return __float_as_int(w); }
__device__ __forceinline__ int packed_of(double w) { return (int)__double_as_longlong(w); }
__device__ __forceinline__ float pack_w(int v, float) { return __int_as_float(v); }
__device__ __forceinline__ double pack_w(int v, double) { return __longlong_as_double((long long)v); }

// Packed tag/type bits of a position snapshot.
__device__ __forceinline__ int pos_bits(const int4& p) { return p.w; }
__device__ __forceinline__ int pos_bits(const dbl4& p) { return packed_of(p.w); }

// Fixed point <-> arithmetic precision.  FP32: through 32-bit halves (the
// 64-bit conversions are slow on this part).  q = hi 2^32 + lo with hi and lo
// converted exactly whenever q carries at most 24 significant bits (every
// float position does), so a float position round-trips exactly; otherwise
// the result is within one float ulp.  The displacement x 2^48 is split at
// 2^24: both halves are exact integers in float for |x| >= 2^-25.
__device__ __forceinline__ float fix_to_real(long long q, float)
{
    const float hi = (float)(int)(q >> 32);
    const float lo = __uint2float_rn((unsigned)(q & 0xffffffffll));
    return fmaf(hi, 0x1p32f, lo) * 0x1p-48f;
}
__device__ __forceinline__ double fix_to_real(long long q, double) { return __ll2double_rn(q) * kInvFix; }
__device__ __forceinline__ long long real_to_fix(float x)
{
    const float y = x * 0x1p24f;
    const float h = truncf(y);
    const int hi = (int)h;
    const int lo = __float2int_rn((y - h) * 0x1p24f);
    return (long long)hi * 16777216ll + lo;
}
__device__ __forceinline__ long long real_to_fix(double x) { return __double2ll_rn(x * kFix); }

__device__ __forceinline__ const PairP<float>* uni_params(const RunArgs& a, float) { return a.uf; }
__device__ __forceinline__ const PairP<double>* uni_params(const RunArgs& a, double) { return a.ud; }

// Selects the run constant of the arithmetic precision.
__device__ __forceinline__ float pick(float, float f, double) { return f; }
__device__ __forceinline__ double pick(double, float, double d) { return d; }

template <typename P4>
__device__ __forceinline__ int type_of(const P4& p) { return pos_bits(p) & ((1 << kTypeBits) - 1); }

// Snapshot coordinate c of fixed-point coordinate q: FP32, the 32-bit box
// fraction floor(q fmul / 2^64); FP64, the coordinate itself.
__device__ __forceinline__ int snap_coord(long long q, int c, const Dev<float>& d)
{
    return (int)__umul64hi((unsigned long long)q, d.fmul[c]);
}
__device__ __forceinline__ double snap_coord(long long q, int, const Dev<double>&) { return fix_to_real(q, 0.0); }
__device__ __forceinline__ int snap_bits(int b, const Dev<float>&) { return b; }
__device__ __forceinline__ double snap_bits(int b, const Dev<double>&) { return pack_w(b, 0.0); }

// FP32 minimum-image displacement of box fractions a -> b along c: the
// wrap-around difference of the fractions (exact), converted and scaled with
// one rounding each.
__device__ __forceinline__ float frac_delta(int a, int b, int c, const Dev<float>& d)
{
    return __fmul_rn(__int2float_rn((int)((unsigned)b - (unsigned)a)), d.fscale[c]);
}

__device__ __forceinline__ float frac_dist2(const int4& pi, const int4& pj, const Dev<float>& d, float& dx,
                                            float& dy, float& dz)
{
    dx = frac_delta(pi.x, pj.x, 0, d);
    dy = frac_delta(pi.y, pj.y, 1, d);
    dz = frac_delta(pi.z, pj.z, 2, d);
    float s = mul_rn(dx, dx);
    s = add_rn(s, mul_rn(dy, dy));
    s = add_rn(s, mul_rn(dz, dz));
    return s;
}

// Squared minimum-image distance of j from i, in the decision precision;
// returns dx = x_j - x_i (wrapped) for the force evaluation.
template <typename Real, typename R4>
__device__ __forceinline__ Real dist2(const R4& pi, const R4& pj, const Dev<Real>& d, Real& dx,
                                      Real& dy, Real& dz)
{
    dx = sub_rn(pj.x, pi.x);
    dy = sub_rn(pj.y, pi.y);
    dz = sub_rn(pj.z, pi.z);
    if (dx > d.hL[0]) dx = sub_rn(dx, d.L[0]);
    else if (dx < -d.hL[0]) dx = add_rn(dx, d.L[0]);
    if (dy > d.hL[1]) dy = sub_rn(dy, d.L[1]);
    else if (dy < -d.hL[1]) dy = add_rn(dy, d.L[1]);
    if (dz > d.hL[2]) dz = sub_rn(dz, d.L[2]);
    else if (dz < -d.hL[2]) dz = add_rn(dz, d.L[2]);
    Real s = mul_rn(dx, dx);
    s = add_rn(s, mul_rn(dy, dy));
    s = add_rn(s, mul_rn(dz, dz));
    return s;
}

// The same squared distance for a pair already in the list (|x_j - x_i| wraps
// at most once and the wrapped distance is below the list radius, a third of
// the box): k = rint(dx / L) is then the wrap of the branchy form above and
// dx - k L is the same single rounding, so d2 is bit-identical.
__device__ __forceinline__ float wrap_rint(float dx, float L, float iL) { return fmaf(-L, rintf(dx * iL), dx); }
__device__ __forceinline__ double wrap_rint(double dx, double L, double iL) { return fma(-L, rint(dx * iL), dx); }

template <typename Real, typename R4>
__device__ __forceinline__ Real dist2_listed(const R4& pi, const R4& pj, const Dev<Real>& d, Real& dx,
                                             Real& dy, Real& dz)
{
    dx = wrap_rint(sub_rn(pj.x, pi.x), d.L[0], d.iL[0]);
    dy = wrap_rint(sub_rn(pj.y, pi.y), d.L[1], d.iL[1]);
    dz = wrap_rint(sub_rn(pj.z, pi.z), d.L[2], d.iL[2]);
    Real s = mul_rn(dx, dx);
    s = add_rn(s, mul_rn(dy, dy));
    s = add_rn(s, mul_rn(dz, dz));
    return s;
}

// FP32 snapshots: one rule for every distance (the fraction difference is
// already the minimum image).
__device__ __forceinline__ float dist2(const int4& pi, const int4& pj, const Dev<float>& d, float& dx, float& dy,
                                       float& dz)
{
    return frac_dist2(pi, pj, d, dx, dy, dz);
}
__device__ __forceinline__ float dist2_listed(const int4& pi, const int4& pj, const Dev<float>& d, float& dx,
                                              float& dy, float& dz)
{
    return frac_dist2(pi, pj, d, dx, dy, dz);
}

template <typename Real>
__device__ __forceinline__ Real ipow(Real b, int e)
{
    // the common exponents n = 10 and n = 6 (e = n/2) by their short chains;
    // e is uniform over a warp, so the branch costs no divergence
    if (e == 5) {
        Real b2 = b * b;
        return b2 * b2 * b;
    }
    if (e == 3) return b * b * b;
    Real r = Real(1);
    while (e) {
        if (e & 1) r *= b;
        e >>= 1;
        if (e) b *= b;
    }
    return r;
}

// FP32: the hardware reciprocal approximation (PTX rcp.approx, relative error
// below 2^-22): it feeds only the values of the potential and forces, never a
// decision, and its error is far inside the FP32 force tolerance.
__device__ __forceinline__ float recip(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

// (sigma/r)^n from s2 = (sigma/r)^2.  X says what the run's exponents are
// (RunArgs::expo): kExpoStd n = 10 for reactive pairs (REACT) and n = 6 for the
// others, kExpoEven any even n, kExpoAny any n.  FP32 code is free of branches
// but for kExpoAny's odd n, so that the pairs a thread works on overlap: with a
// loop over the bits of n (n = 100), or merely a test for n = 10, they went one
// after the other and one pair of a lone warp took 600 to 900 cycles.  The
// products are those of ipow in the same order: the same bits.  (FP64 is bound
// by the number of multiplications.)
template <int X, bool REACT, typename Real>
__device__ __forceinline__ Real pair_power(const PairP<Real>& p, Real s2)
{
    if (sizeof(Real) == 8) {
        Real x = ipow(s2, p.nhalf);
        if (p.odd) x *= sqrt(s2);
        return x;
    }
    if (X == kExpoStd) {
        const Real b2 = s2 * s2;
        return REACT ? b2 * b2 * s2 : b2 * s2;
    }
    const int e = p.nhalf;  // at most 64
    Real b = s2, r = e & 1 ? s2 : Real(1);
#pragma unroll
    for (int k = 1; k < 7; k++) {
        b *= b;
        r = e >> k & 1 ? r * b : r;
    }
    if (X == kExpoAny && p.odd) r *= sqrt(s2);
    return r;
}

// Eq. 2b at squared distance r2: v and f = -(dv/dr)/r.
template <int X, bool REACT, typename Real>
__device__ __forceinline__ void lj_eval(const PairP<Real>& p, Real r2, Real& v, Real& f)
{
    Real ir2 = recip(r2);
    Real s2 = p.sig2 * ir2;
    Real x = pair_power<X, REACT>(p, s2);
    Real x2 = x * x;
    v = p.four_eps * (x2 - x);
    f = p.four_eps * p.n_real * (Real(2) * x2 - x) * ir2;
}

// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; r++) {
        unsigned hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        unsigned hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// Three standard normals for (seed, step, tag): counter (tag, step lo,
// step hi, 1), key (seed lo, seed hi), Box-Muller on (u0,u1) and (u2,u3).
// FP32: the hardware logarithm and sine/cosine (absolute error about 1e-6 on
// these arguments, far below what the noise amplitude sqrt((1 - c^2) kT/m)
// lets through to a trajectory), at a fifth of the accurate functions' cost.
__device__ __forceinline__ void normals3(unsigned long long seed, long long step, unsigned tag,
                                         float z[3])
{
    uint4 w = philox4x32_10(make_uint4(tag, (unsigned)step, (unsigned)((unsigned long long)step >> 32), 1u),
                            make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
    const float s32 = 2.3283064365386963e-10f;
    const float two_pi = 6.28318530717958648f;
    float u0 = (__uint2float_rn(w.x) + 0.5f) * s32;
    float u1 = (__uint2float_rn(w.y) + 0.5f) * s32;
    float u2 = (__uint2float_rn(w.z) + 0.5f) * s32;
    float u3 = (__uint2float_rn(w.w) + 0.5f) * s32;
    float ra = sqrtf(-2.0f * __logf(u0));
    float rb = sqrtf(-2.0f * __logf(u2));
    float sn, cs;
    __sincosf(two_pi * u1, &sn, &cs);
    z[0] = ra * cs;
    z[1] = ra * sn;
    z[2] = rb * __cosf(two_pi * u3);
}

__device__ __forceinline__ void normals3(unsigned long long seed, long long step, unsigned tag,
                                         double z[3])
{
    uint4 w = philox4x32_10(make_uint4(tag, (unsigned)step, (unsigned)((unsigned long long)step >> 32), 1u),
                            make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
    const double s32 = 2.3283064365386962890625e-10;
    double u0 = ((double)w.x + 0.5) * s32;
    double u1 = ((double)w.y + 0.5) * s32;
    double u2 = ((double)w.z + 0.5) * s32;
    double u3 = ((double)w.w + 0.5) * s32;
    double ra = sqrt(-2.0 * log(u0));
    double rb = sqrt(-2.0 * log(u2));
    double sn, cs;
    sincospi(2.0 * u1, &sn, &cs);
    z[0] = ra * cs;
    z[1] = ra * sn;
    z[2] = rb * cospi(2.0 * u3);
}

// ---------------------------------------------------------------------------
// Grid barrier for the cooperative launch: split arrive / wait, every wait
// bounded in time; on expiry the status word gets kStatusTimeout and every
// block leaves the kernel.

struct BarState {
    unsigned long long target;  // valid in thread 0
};

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Set (thread 0 of one block) when the launch must withhold that block's
// arrival at its first grid barrier (a test of the bounded waits).
static __shared__ int s_withhold;

// Arrival: the block's writes are ordered before a release add on the
// counter (after the block-wide __syncthreads, thread 0's release is
// cumulative over them).  Generation g completes at count g * (group size).
// With pub_dst set, thread 0 first folds the block's shared maximum *pub_src
// into the global maximum *pub_dst (and clears it), so the other blocks see
// it after their wait.
__device__ __forceinline__ void bar_arrive(Ctl* ctl, BarState& b, unsigned* pub_dst = nullptr,
                                           unsigned* pub_src = nullptr)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        if (pub_dst) {
            const unsigned m = *pub_src;
            if (m) atomicMax(pub_dst, m);
            *pub_src = 0u;
        }
        if (kBatched && g_size() == 1) return;  // a group of one block: __syncthreads is the barrier
        b.target += g_size();
        if (s_withhold)
            s_withhold = 0;  // this arrival is withheld: every wait of the barrier runs out
        else
            asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(&ctl->barrier), "l"(1ull) : "memory");
    }
}

// Wait: acquire polling, bounded in time.  Every arrival is a release add on
// the counter, and later adds continue its release sequence, so the load that
// first sees the target synchronises with every arrival: the other blocks'
// writes are visible to this block after the __syncthreads.  (Relaxed polling
// followed by an acquire fence measured 0.4 us slower per step.)
__device__ __forceinline__ bool bar_wait(Ctl* ctl, const BarState& b, long long timeout_ns,
                                         int where, int* s_ok)
{
    if (kBatched && g_size() == 1) {
        __syncthreads();
        return true;
    }
    if (threadIdx.x == 0) {
        int ok = 1;
        int spins = 0;
        long long t0 = 0;
        while (ld_acquire_u64(&ctl->barrier) < b.target) {
            if (++spins < 64) continue;
            if (spins == 64) t0 = gtimer_ns();
            if (ld_relaxed(&ctl->status) & kStatusTimeout) {
                ok = 0;
                break;
            }
            if (gtimer_ns() - t0 > timeout_ns) {
                atomicOr(&ctl->status, kStatusTimeout);
                ctl->timeout_at = where;
                ok = 0;
                break;
            }
            __nanosleep(32);
        }
        *s_ok = ok;
    }
    __syncthreads();
    if (*s_ok == 0) asm volatile("cp.async.wait_all;" ::: "memory");  // leave no copy in flight
    return *s_ok != 0;
}

// ---------------------------------------------------------------------------
// Block reductions

// Compensated FP32 summation (Knuth's TwoSum; the double-float addition of
// Dekker and Bailey): a pair (hi, lo) carries about 44 significant bits, so
// the block sums below lose nothing beyond the per-thread FP32 terms.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bv = __fsub_rn(s, a);
    const float av = __fsub_rn(s, bv);
    e = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
}

__device__ __forceinline__ void df_add(float& hi, float& lo, float bh, float bl)
{
    float s, e;
    two_sum(hi, bh, s, e);
    e = __fadd_rn(e, __fadd_rn(lo, bl));
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// Block sums of the per-thread thermo accumulators (energies, virial, bond
// count), written to out[q] (the block's partial of the pass; block partials
// are summed over blocks in FP64, run_reduce_thermo).
//
// FP32 two-barrier passes: a warp folds its lanes' terms after every 32
// particles (a shuffle tree, at most five roundings of the sum of magnitudes),
// lane q carries quantity q in FP64, and the warps meet in s_wacc in FP64
// (block_sums_from_rows), so the error does not grow with the system size.
//
// FP64 passes: every thread's terms, staged in shared memory and summed by one
// warp per quantity over the threads that had any (block_sums_from_threads;
// with 13 particles on a block the sums over every thread's zeros were a tenth
// of a step).
//
// The resident step: one row per thread, the warps' shuffle-tree sums in
// s_wpart; warp q then sums quantity q over the block's warps compensated
// (double-float).
static __shared__ double s_wacc[32][kNQA];
static __shared__ float s_wpart[kNQA][32];

template <typename T>
__device__ __forceinline__ T warp_sum(T x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// s_wpart[q][warp] = the warp's sum of x (every lane of the warp calls it).
__device__ __forceinline__ void warp_part(float x, int q)
{
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) s_wpart[q][threadIdx.x >> 5] = x;
}

// Sums s_wpart over the block's warps into out (and out2, when given).  The
// caller orders the s_wpart writes before and the next ones after
// (block_sums_from_warps: two __syncthreads).
__device__ __forceinline__ void warp_sums_to(double* out, double* out2)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int q = warp; q < kNQ; q += nw) {  // quantity q by warp q mod nw (blocks of fewer warps)
        if (q >= kNQA) {
            if (lane == 0) {
                out[q] = 0.0;
                if (out2) out2[q] = 0.0;
            }
            continue;
        }
        float hi = lane < nw ? s_wpart[q][lane] : 0.0f, lo = 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
            df_add(hi, lo, h2, l2);
        }
        if (lane == 0) {
            const double tot = (double)hi + (double)lo;
            out[q] = tot;
            if (out2) out2[q] = tot;
        }
    }
}

__device__ __forceinline__ void block_sums_from_warps(double* out, double* out2)
{
    __syncthreads();
    warp_sums_to(out, out2);
    __syncthreads();
}

// Sums s_wacc over the first nact warps (those that had particles; 0: none) into
// out (and out2, when given).
__device__ __forceinline__ void block_sums_from_rows(int nact, double* out, double* out2)
{
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int q = warp; q < kNQ; q += nw) {
        double x = lane < nact && q < kNQA ? s_wacc[lane][q] : 0.0;
        if (q < kNQA)
            for (int o = 1; o < nact; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) {
            out[q] = x;
            if (out2) out2[q] = x;
        }
    }
    __syncthreads();
}

// FP64: the sums of stage[q][thread] over the first nact threads (the others'
// terms are zero).
__device__ __forceinline__ void block_sums_from_threads(const double* stage, int nact, double* out, double* out2)
{
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, B = blockDim.x, nw = (B + 31) >> 5;
    for (int q = warp; q < kNQ; q += nw) {
        double x = 0.0;
        if (q < kNQA) {
            for (int k = lane; k < nact; k += 32) x += stage[q * B + k];
            x = warp_sum(x);
        }
        if (lane == 0) {
            out[q] = x;
            if (out2) out2[q] = x;
        }
    }
    __syncthreads();
}

// Exclusive scan of one int per thread over the block (block 0 only).
__device__ __forceinline__ int block_excl_scan(int v, int* sh, int* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int s = (lane < nw) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) sh[lane] = s;  // inclusive warp totals
    }
    __syncthreads();
    int base = warp > 0 ? sh[warp - 1] : 0;
    *total = sh[nw - 1];
    __syncthreads();
    return base + x - v;
}

// ---------------------------------------------------------------------------
// Neighbour-list rebuild phases: bin by cell, counting sort with a
// deterministic order inside each cell (by old slot), every per-particle array
// moved into the sorted order, then one row per particle from the 27-cell
// stencil.  Five grid barriers.  (With the counts of a block's cells summed in a
// phase of their own, the members of a cell sorted in global memory by one thread
// and the arrays then gathered one load after the other, the phases before the
// row build took 17 us at 1,200 particles and 82 us at 1M; now 13 and 49.)

template <typename Real>
__device__ __forceinline__ void cell_coords(const Dev<Real>& d, const typename Dev<Real>::R4& p,
                                            int& cx, int& cy, int& cz)
{
    cx = (int)(p.x * d.inv_cw[0]);
    cy = (int)(p.y * d.inv_cw[1]);
    cz = (int)(p.z * d.inv_cw[2]);
    cx = min(max(cx, 0), d.nc[0] - 1);
    cy = min(max(cy, 0), d.nc[1] - 1);
    cz = min(max(cz, 0), d.nc[2] - 1);
}

// FP32 snapshots: the cell of a box fraction u is floor(u nc / 2^32), exact.
__device__ __forceinline__ void cell_coords(const Dev<float>& d, const int4& p, int& cx, int& cy, int& cz)
{
    cx = min((int)__umulhi((unsigned)p.x, (unsigned)d.nc[0]), d.nc[0] - 1);
    cy = min((int)__umulhi((unsigned)p.y, (unsigned)d.nc[1]), d.nc[1] - 1);
    cz = min((int)__umulhi((unsigned)p.z, (unsigned)d.nc[2]), d.nc[2] - 1);
}

// Block b owns the contiguous chunk [b*ch, (b+1)*ch) of cells (ranks) in the scan.
template <typename Real>
__device__ __forceinline__ int chunk_cells(const Dev<Real>& d) { return (d.ncell + g_size() - 1) / g_size(); }

// Counts the cells' particles and the chunks' (through chunk: g_size() ints of
// shared memory); both counts start at zero (k_set_state, ph_chunk_scan, ph_move).
template <typename Real>
__device__ void ph_bin(const Dev<Real>& d, int pc, int* chunk)
{
    const int G = g_size(), ch = chunk_cells(d);
    __syncthreads();  // what the memory held before has been read (r_flush)
    for (int b = threadIdx.x; b < G; b += blockDim.x) chunk[b] = 0;
    __syncthreads();
    for (int p0 = g_rank() * blockDim.x; p0 < d.n; p0 += G * blockDim.x) {  // block-uniform
        const int p = p0 + threadIdx.x;
        int b = -1;
        if (p < d.n) {
            int cx, cy, cz;
            cell_coords(d, d.pos[pc][p], cx, cy, cz);
            const int r = __ldg(&d.cell_rank[(cz * d.nc[1] + cy) * d.nc[0] + cx]);
            d.perm[p] = r;  // the cell of old slot p
            atomicAdd(&d.cell_cnt[r], 1);
            b = r / ch;
        }
        // slots are nearly in cell order: a warp has one or two chunks
        const unsigned m = __match_any_sync(0xffffffffu, b);
        if (b >= 0 && (threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(&chunk[b], __popc(m));
    }
    __syncthreads();
    for (int b = threadIdx.x; b < G; b += blockDim.x)
        if (chunk[b]) atomicAdd(&d.bsum[b], chunk[b]);
}

// Exclusive scan of the cell counts: each block adds up the chunks before its
// own, scans its cells, writes cell_start and cell_fill, and zeroes the counts it
// consumed (so the next build starts from zero without a separate pass).
__device__ __forceinline__ int block_sum_int(int v, int* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < nw; w++) t += sh[w];
    __syncthreads();
    return t;
}

template <typename Real>
__device__ void ph_chunk_scan(const Dev<Real>& d, int* sh)
{
    const int ch = chunk_cells(d);
    const int beg = min(g_rank() * ch, d.ncell), end = min(beg + ch, d.ncell);
    int v = 0;
    for (int b = threadIdx.x; b < g_rank(); b += blockDim.x) v += d.bsum[b];
    int base = block_sum_int(v, sh);
    // scan the chunk in pieces of blockDim.x cells
    for (int c0 = beg; c0 < end; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const int cnt = c < end ? d.cell_cnt[c] : 0;
        int total;
        int ex = block_excl_scan(cnt, sh, &total);
        if (c < end) {
            d.cell_start[c] = base + ex;
            d.cell_fill[c] = base + ex;
            d.cell_cnt[c] = 0;
        }
        base += total;
    }
    if (end == d.ncell && beg < end && threadIdx.x == 0) d.cell_start[d.ncell] = base;
}

// The members of every cell, in any order (after the fill counters).
template <typename Real>
__device__ void ph_scatter(const Dev<Real>& d, int t, int nt)
{
    for (int p = t; p < d.n; p += nt) d.cell_fill[d.ncell + atomicAdd(&d.cell_fill[d.perm[p]], 1)] = p;
}

// Moves every particle to its new slot: its cell's first, plus the members of
// the cell with a smaller old slot.  All loads of a particle come before its
// stores.
template <typename Real>
__device__ void ph_move(const Dev<Real>& d, int pc, int ac, int t, int nt)
{
    const int n = d.n;
    const int* member = d.cell_fill + d.ncell;
    if (g_rank() == 0)
        for (int b = threadIdx.x; b < g_size(); b += blockDim.x) d.bsum[b] = 0;  // every block has read them
    for (int p = t; p < n; p += nt) {
        const int r = d.perm[p];
        const typename Dev<Real>::P4 pp = d.pos[pc][p];
        const typename Dev<Real>::R4 v = d.vel[ac][p];
        long long x[3];
        int im[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            x[c] = d.xq[ac][c * n + p];
            im[c] = d.img[ac][c * n + p];
        }
        const int s = d.cell_start[r], e = d.cell_start[r + 1];
        int q = s;
        for (int k = s; k < e; k += 4) {
            int m[4];
#pragma unroll
            for (int u = 0; u < 4; u++) m[u] = k + u < e ? member[k + u] : n;
#pragma unroll
            for (int u = 0; u < 4; u++) q += m[u] < p;
        }
        d.pos[pc ^ 1][q] = pp;
        if (d.has_bonds) d.slot_of_tag[pos_bits(pp) >> kTypeBits] = q;
        d.vel[ac ^ 1][q] = v;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            d.xq[ac ^ 1][c * n + q] = x[c];
            d.img[ac ^ 1][c * n + q] = im[c];
        }
    }
}

// Every block's dynamic shared memory; the regions of its users (the list build,
// the passes, the resident step) sit at compile-time offsets, so that every
// access is a direct shared-memory access.
extern __shared__ __align__(32) unsigned char g_dyn[];

// ---------------------------------------------------------------------------
// Block ownership and the neighbour list.
//
// Block b of a G-block launch owns the contiguous (Morton-ordered, hence
// spatially compact) particle range [b*Pb, min((b+1)*Pb, n)), Pb = ceil(n/G),
// processed in sub-chunks of at most blockDim.x particles.  The neighbour
// entries of a sub-chunk are stored contiguously in the block's region of the
// list buffer: first the reactive rows of all its particles, then the other
// rows; entry e holds the partner slot ent_j[e], and pinfo[p] = (first reactive
// entry, n_reactive, first other entry, n_other).  Entry positions are
// unsigned 32-bit.
//
// FP32: one thread works through one particle's rows.  The threads of a
// sub-chunk take its particles in descending order of (n_reactive, n_other),
// so that the 32 rows of a warp have alike lengths (perm[q0 + t] = particle of
// thread t, tinfo[q0 + t] = its pinfo); rows are stored in that order, each
// padded with the particle's own slot to a multiple of four entries, so that a
// thread loads its partners four at a time.
// FP64: rows in particle order without padding, ent_o[e] = the owner's index
// inside its sub-chunk (one lane works on one entry).

template <typename Real>
__device__ __forceinline__ void block_range(const Dev<Real>& d, int& b0, int& b1)
{
    const int Pb = (d.n + g_size() - 1) / g_size();
    b0 = min(g_rank() * Pb, d.n);
    b1 = min(b0 + Pb, d.n);
}

// Stable counting sort, largest key first, of one item per thread (key in
// [0, 255], -1: no item): returns the item's rank.  Equal keys keep the thread
// order.  wh: scratch of blockDim / 32 x 256 u16 counts; hist: 256 ints; sh:
// block_excl_scan's scratch; blockDim >= 256.
static __device__ int rank_desc(int key, unsigned short* wh, int* hist, int* sh)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, NW = blockDim.x >> 5;
    __syncthreads();  // a previous call's readers are done with wh and hist
    for (int k = t; k < NW * 256; k += blockDim.x) wh[k] = 0;
    __syncthreads();
    // the warp's lanes with this key, and how many come before this lane
    const unsigned m = __match_any_sync(0xffffffffu, key);
    const int before = __popc(m & ((1u << lane) - 1u));
    if (key >= 0 && before == 0) wh[warp * 256 + key] = (unsigned short)__popc(m);
    __syncthreads();
    // per key: the counts of the warps before each warp, and the key's total
    if (t < 256) {
        int run = 0;
        for (int w = 0; w < NW; w++) {
            const int c = wh[w * 256 + t];
            wh[w * 256 + t] = (unsigned short)run;
            run += c;
        }
        hist[t] = run;
    }
    __syncthreads();
    // keys in descending order: the first rank of key b is the count above it
    const int b = 255 - t;
    int tot;
    const int ex = block_excl_scan(t < 256 ? hist[b] : 0, sh, &tot);
    if (t < 256) hist[b] = ex;  // every thread read hist before the scan's barriers
    __syncthreads();
    return key >= 0 ? hist[key] + wh[warp * 256 + key] + before : 0;
}

// Shared-memory scratch of the list build.
struct BuildStage {
    static constexpr int kCap = 24;  // partners a thread holds before they are placed
    static constexpr size_t B = kThreads;
    static constexpr size_t O_HITS = 0;                       // [kCap][B] partner slots: reactive from the front, others from the back
    static constexpr size_t O_CNT = O_HITS + kCap * B * 4;    // [B] int2 row lengths, then row starts, by particle
    static constexpr size_t O_SIZE = O_CNT + B * 8;           // [B] int2 row sizes, then places, by thread order
    static constexpr size_t O_WH = O_SIZE + B * 8;            // rank_desc's scratch
    static constexpr size_t O_HIST = O_WH + B / 32 * 512;
    static constexpr size_t kBytes = O_HIST + 1024;
};

// Whether candidate pj lies inside the list radius of pi.  FP64: FP32 distances
// decide all but the pairs within 2^-18 of the box of the radius, so that the
// FP64 pipe, 19 cycles per warp instruction, sees hardly any candidate (with 8
// FP64 instructions for every one the rows of 20,000 particles took 132 us, now 27).
__device__ __forceinline__ bool in_list(const Dev<float>& d, const PairP<float>& p, const int4& pi, const int4& pj)
{
    float dx, dy, dz;
    return dist2(pi, pj, d, dx, dy, dz) < p.rlist2;
}
__device__ __forceinline__ float float_dist2(const Dev<double>& d, const dbl4& pi, const dbl4& pj);
__device__ __forceinline__ bool in_list(const Dev<double>& d, const PairP<double>& p, const dbl4& pi, const dbl4& pj)
{
    const float r2 = float_dist2(d, pi, pj);
    if (r2 >= p.list_out2) return false;
    if (r2 < p.list_in2) return true;
    double dx, dy, dz;
    return dist2(pi, pj, d, dx, dy, dz) < p.rlist2;
}

// One lane's share [c0, c1) of the 27 stencil cells of particle i (cell cx, cy,
// cz): hit(q, reactive) for every partner q inside the list radius, in stencil
// order.  The next cell's range is loaded while the present one's candidates
// are tested, two at a time.
template <typename Real, typename F>
__device__ __forceinline__ void sweep_cells(const Dev<Real>& d, const PairP<Real>* row, const typename Dev<Real>::P4* pos,
                                            const typename Dev<Real>::P4& pi, int i, int cx, int cy, int cz, int c0,
                                            int c1, F&& hit)
{
    typedef typename Dev<Real>::P4 P4;
    auto range = [&](int c, int& s, int& e) {
        int x = cx + c % 3 - 1, y = cy + (c / 3) % 3 - 1, z = cz + c / 9 - 1;
        x = x < 0 ? x + d.nc[0] : (x >= d.nc[0] ? x - d.nc[0] : x);
        y = y < 0 ? y + d.nc[1] : (y >= d.nc[1] ? y - d.nc[1] : y);
        z = z < 0 ? z + d.nc[2] : (z >= d.nc[2] ? z - d.nc[2] : z);
        const int r = __ldg(&d.cell_rank[(z * d.nc[1] + y) * d.nc[0] + x]);
        s = d.cell_start[r];
        e = d.cell_start[r + 1];
    };
    auto test = [&](int q, const P4& pj) {
        const PairP<Real>& p = row[type_of(pj)];
        if (q != i && in_list(d, p, pi, pj)) hit(q, p.kind == KIND_SWAP);
    };
    int s = 0, e = 0;
    if (c0 < c1) range(c0, s, e);
    for (int c = c0; c < c1; c++) {
        const int s0 = s, e0 = e;
        if (c + 1 < c1) range(c + 1, s, e);
        for (int q = s0; q < e0; q += 2) {
            const bool two = q + 1 < e0;
            const P4 pa = pos[q], pb = pos[two ? q + 1 : q];
            test(q, pa);
            if (two) test(q + 1, pb);
        }
    }
}

// Builds the block's rows (last rebuild phase).  G lanes (a power of two, as
// many as the block's particles leave) share a particle: each tests the
// candidates of its share of the 27 stencil cells and keeps the partners it
// finds in shared memory; the sub-chunk's rows are then placed and written, in
// stencil order whatever G is.  (Rows longer than the lanes can hold: the
// cells are gone through once more to write them.)  One warp per cell with the
// candidates across the lanes, in a counting and a writing sweep, spent 540
// warp instructions per particle, most of them on handing out candidates and
// on ballots: 2.8 -> 1.0 ms per build at 2M beads.
// Returns the block's entry count per particle (rounded up), the row length a
// capacity check needs.
template <typename Real>
__device__ int ph_build_rows(const Dev<Real>& d, const PairP<Real>* tab, int pc, int* sh, int* overflow)
{
    typedef typename Dev<Real>::P4 P4;
    typedef BuildStage BS;
    constexpr bool kRows = sizeof(Real) == 4;  // sorted and padded rows
    const P4* pos = d.pos[pc];
    int* hits = (int*)(g_dyn + BS::O_HITS);
    int2* cnt = (int2*)(g_dyn + BS::O_CNT);
    int2* size = (int2*)(g_dyn + BS::O_SIZE);
    const int t = threadIdx.x, B = blockDim.x;
    int b0, b1;
    block_range(d, b0, b1);
    const int Pb = (d.n + g_size() - 1) / g_size();
    // the block's region: list_stride entries per particle (max_nn and the padding)
    long long base = (long long)g_rank() * Pb * d.list_stride;
    long long used = 0;  // entries without padding
    for (int q0 = b0; q0 < b1; q0 += B) {
        const int P = min(B, b1 - q0);
        int lg = 0;
        while (lg < 5 && (P << (lg + 1)) <= B) lg++;
        const int G = 1 << lg, g = t & (G - 1), pl = t >> lg;
        const bool has = pl < P;
        const int i = q0 + (has ? pl : 0);
        const P4 pi = pos[i];
        const PairP<Real>* row = tab + type_of(pi) * d.ntypes;
        int cx, cy, cz;
        cell_coords(d, pi, cx, cy, cz);
        const int c0 = has ? 27 * g / G : 0, c1 = has ? 27 * (g + 1) / G : 0;
        int nr = 0, nw = 0;
        sweep_cells(d, row, pos, pi, i, cx, cy, cz, c0, c1, [&](int q, bool react) {
            if (nr + nw < BS::kCap) hits[(react ? nr : BS::kCap - 1 - nw) * B + t] = q;
            nr += react;
            nw += !react;
        });
        // the lane's place in its particle's rows, and the rows' lengths
        int er = nr, ew = nw;
        for (int o = 1; o < G; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, er, o, G), b = __shfl_up_sync(0xffffffffu, ew, o, G);
            if (g >= o) {
                er += a;
                ew += b;
            }
        }
        const int tr = __shfl_sync(0xffffffffu, er, G - 1, G), tw = __shfl_sync(0xffffffffu, ew, G - 1, G);
        er -= nr;
        ew -= nw;
        if (has && g == 0) cnt[pl] = make_int2(tr, tw);
        const bool again = __syncthreads_or(nr + nw > BS::kCap);
        // places: the reactive rows of the sub-chunk, then the others, in thread order
        const int2 c = t < P ? cnt[t] : make_int2(0, 0);
        int rk = t;
        if (kRows)
            rk = rank_desc(t < P ? (min(c.x, 15) << 4 | min(c.y, 15)) : -1, (unsigned short*)(g_dyn + BS::O_WH),
                           (int*)(g_dyn + BS::O_HIST), sh);
        if (kRows && ((q0 - b0) / B & 1)) rk = P - 1 - rk;  // every warp gets long and short rows in turn
        const int pad = kRows ? 3 : 0;
        if (t < P) size[rk] = make_int2((c.x + pad) & ~pad, (c.y + pad) & ~pad);
        __syncthreads();
        const int2 z = t < P ? size[t] : make_int2(0, 0);
        int Er, Ew, Ec;
        const int offr = block_excl_scan(z.x, sh, &Er);
        const int offw = block_excl_scan(z.y, sh, &Ew);
        block_excl_scan(c.x + c.y, sh, &Ec);
        if (t < P) size[t] = make_int2(offr, offw);
        __syncthreads();
        used += Ec;
        const bool fits = used <= (long long)Pb * d.max_nn;
        if (fits) {
            if (t < P) {
                const int2 o = size[rk];
                const int ro = (int)(unsigned)(base + o.x), wo = (int)(unsigned)(base + Er + o.y);
                const int4 inf = make_int4(ro, c.x, wo, c.y);
                d.pinfo[q0 + t] = inf;
                if constexpr (kRows) {
                    d.tinfo[q0 + rk] = inf;
                    d.perm[q0 + rk] = q0 + t;
                }
                cnt[t] = make_int2(ro, wo);
            }
            __syncthreads();
            if (has) {
                const unsigned ro = (unsigned)cnt[pl].x, wo = (unsigned)cnt[pl].y;
                unsigned kr = ro + er, kw = wo + ew;
                auto put = [&](unsigned& k, int q) {
                    d.ent_j[k] = q;
                    if constexpr (!kRows) d.ent_o[k] = (unsigned short)pl;
                    k++;
                };
                if (!again) {
                    for (int k = 0; k < nr; k++) put(kr, hits[k * B + t]);
                    for (int k = 0; k < nw; k++) put(kw, hits[(BS::kCap - 1 - k) * B + t]);
                } else {
                    sweep_cells(d, row, pos, pi, i, cx, cy, cz, c0, c1,
                                [&](int q, bool react) { put(react ? kr : kw, q); });
                }
                if (kRows && g == G - 1) {
                    while (kr & 3u) put(kr, i);  // rows start at multiples of four
                    while (kw & 3u) put(kw, i);
                }
            }
        } else if (t == 0) {
            *overflow = 1;
        }
        base += Er + Ew;
        __syncthreads();  // cnt, size and hits are free
    }
    const int np = b1 - b0;
    return np > 0 ? (int)((used + np - 1) / np) : 0;
}

// ---------------------------------------------------------------------------
// UNI: every reactive type pair has the same coefficients (ps) and so has
// every other interacting pair (pw); they are then read from the
// kernel-parameter constant bank instead of the shared-memory table, which
// costs neither a lookup nor registers.
template <typename Real, bool UNI>
__device__ __forceinline__ const PairP<Real>& pair_of(const PairP<Real>* tab, int ti, int tj, int nt,
                                                    const PairP<Real>& uni)
{
    return UNI ? uni : tab[ti * nt + tj];
}

// The two-barrier passes: nothing in a pass waits for another warp, so that one
// warp's gathers overlap the arithmetic of the others.
//
// FP32 (s_pass_rows, f_pass_rows): one thread per particle, in the order of
// the build (alike rows in a warp).  A thread loads its partners four at a
// time and gathers them together.  An entry-parallel version (one lane per
// entry, results through shared memory to the owners) spent 2,900 warp
// instructions per 32 particles and step, this one 1,700; block barriers around
// 768-particle waves before that: mix of 1M particles 197 ->
// 125 us per step, 20-step launches with a list build in each.
//
// FP64 (s_pass_waves, f_pass_waves): the bound is the FP64 pipe, which takes 19
// cycles per warp instruction on the whole SM however many of its lanes are on
// (24 warps; one warp alone 64).  So every FP64 instruction is given as many
// lanes as there are, and pairs that cannot contribute none: the block sorts
// out a wave of entries with FP32 distances (conservative, see may_reach: half
// of the listed pairs lie in the skin), lines up the rest, evaluates them one
// per thread, and the owners sum the rows.  The reactive pairs' values of the S
// pass are kept in shared memory for the force pass where they fit.  (Every
// listed entry evaluated, twice if reactive, took
// 57 us per step of 20,000 particles and 31 of 2,000, this takes 28 and 20.)

constexpr int kBeyond = 1 << 15;  // FP64: marks a lined-up entry, a kept pair outside r_min

// Shared-memory staging of the passes: slot t holds thread t's particle (FP32,
// in the threads' order) or particle t of the sub-chunk (FP64).
template <typename Real>
struct Stage {
    typedef typename Dev<Real>::R4 R4;
    typedef typename Dev<Real>::P4 P4;
    static constexpr bool kWaves = sizeof(Real) == 8;
    static constexpr int kWave = !kWaves ? 0 : kThreads > 512 ? 2048 : 3072;  // entries of a wave
    static constexpr size_t B = kThreads;
    static constexpr size_t O_POS = 0;                                  // [B] P4 positions
    static constexpr size_t O_VEL = O_POS + B * sizeof(P4);             // [B] R4 velocities
    static constexpr size_t O_XQ = O_VEL + B * sizeof(R4);              // [3B] fixed-point positions
    static constexpr size_t O_INFO = O_XQ + 3 * B * sizeof(long long);  // [B] int4 list ranges
    static constexpr size_t O_S = O_INFO + B * sizeof(int4);            // [B] S
    static constexpr size_t O_IDX = O_S + B * sizeof(Real);             // FP32: [B] particle slots
    static constexpr size_t O_W = O_IDX + (kWaves ? 0 : B * 4);         // FP64: [3][kWave] entry results
    static constexpr size_t O_LIST = O_W + (size_t)kWave * 24;          // [kWave] int2 entries lined up (entry of the
                                                                        // wave | owner << 16, partner)
    static constexpr size_t O_KEEP = O_LIST + (size_t)kWave * 8;        // [6][kKeep] reactive pairs' values
    static constexpr int kKeep = !kWaves ? 0 : (int)((212 * 1024 - O_KEEP) / 48);
    static constexpr size_t kPassBytes = O_KEEP + (size_t)kKeep * 48;
    static_assert(kWave <= kBeyond, "an entry of the wave in 15 bits");
    static_assert(!kWaves || kPassBytes - O_W >= kNQA * B * 8, "the thermo terms fit behind the particles' state");
    static constexpr size_t kBytes = kPassBytes > BuildStage::kBytes ? kPassBytes : BuildStage::kBytes;

    static __device__ __forceinline__ P4* pos() { return (P4*)(g_dyn + O_POS); }
    static __device__ __forceinline__ R4* vel() { return (R4*)(g_dyn + O_VEL); }
    static __device__ __forceinline__ long long* xq() { return (long long*)(g_dyn + O_XQ); }
    static __device__ __forceinline__ int4* info() { return (int4*)(g_dyn + O_INFO); }
    static __device__ __forceinline__ Real* S() { return (Real*)(g_dyn + O_S); }
    static __device__ __forceinline__ int* idx() { return (int*)(g_dyn + O_IDX); }
    static __device__ __forceinline__ Real* w() { return (Real*)(g_dyn + O_W); }
    static __device__ __forceinline__ int2* list() { return (int2*)(g_dyn + O_LIST); }
    static __device__ __forceinline__ Real* keep() { return (Real*)(g_dyn + O_KEEP); }
};

// Asynchronous global -> shared copies (no register staging).
__device__ __forceinline__ void cp_async(void* smem, const void* gmem, int bytes)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if (bytes == 16)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
    else if (bytes == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename R4>
__device__ __forceinline__ void cp_async_r4(R4* smem, const R4* gmem)
{
    if (sizeof(R4) == 16) {
        cp_async(smem, gmem, 16);
    } else {
        cp_async(smem, gmem, 16);
        cp_async((char*)smem + 16, (const char*)gmem + 16, 16);
    }
}

// ---------------------------------------------------------------------------
// S pass: S_i = sum over reactive partners k inside r_cut of a vh(r_ik).

// One reactive entry's term of S_i: a vh(r_ij) inside r_cut, else 0 (evaluated
// for every listed pair and selected by the cut-off decision, see entry_force).
template <typename Real, bool UNI, int X>
__device__ __forceinline__ Real s_term(const Dev<Real>& d, const PairP<Real>* tab, const PairP<Real>& ps,
                                       const typename Dev<Real>::P4& pi, const typename Dev<Real>::P4& pj)
{
    const PairP<Real>& p = pair_of<Real, UNI>(tab, type_of(pi), type_of(pj), d.ntypes, ps);
    Real dx, dy, dz;
    const Real r2 = dist2_listed(pi, pj, d, dx, dy, dz);
    Real v, f;
    lj_eval<X, true>(p, r2, v, f);
    const Real vh = r2 > p.rmin2 ? (p.vshift - v) * p.inv_epshat : Real(1);
    return r2 < p.rc2 ? mul_rn(p.a, vh) : Real(0);
}

// Brings the first line of each of a thread's rows into L2 (the rows of a warp
// are neighbours) while the warp works on other entries.
__device__ __forceinline__ void prefetch_row(const Dev<float>& d, int first)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(&d.ent_j[(unsigned)first]));
}

__device__ __forceinline__ int4 load_four(const Dev<float>& d, int first, int k)
{
    return __ldcs((const int4*)&d.ent_j[(unsigned)first + (unsigned)k]);  // streamed: keep L2 for the snapshots
}

// The 1024-thread shapes (64 registers) gather two partners at a time and load the
// next row's ranges late: with four at a time and the ranges held through the row
// they spilled (2M-bead network, 10 steps 2.36 -> 2.30 ms; sweep of 96 systems, 50
// steps 6.81 -> 6.61 ms).
constexpr bool kLean = kThreads >= 1024;

// FP32.  staged: the block has one sub-chunk and the shared copies of its
// positions and list ranges are current (kept by the previous force pass), so
// they are not loaded again; its S values also stay in shared memory for the
// force pass.
template <bool UNI, int X>
__device__ void s_pass_rows(const Dev<float>& d, const PairP<float>* tab, int pc, const PairP<float>& ps, bool staged)
{
    typedef Stage<float> SM;
    const int4* pos = d.pos[pc];
    int b0, b1;
    block_range(d, b0, b1);
    const int t = threadIdx.x;
    const bool single = b1 - b0 <= kThreads;
    if (t >= b1 - b0) return;
    // what the thread's next row needs is loaded while it works on the present one
    int4 ti, pi;
    int i;
    if (staged) {
        ti = SM::info()[t];
        i = SM::idx()[t];
        pi = SM::pos()[t];
    } else {
        ti = d.tinfo[b0 + t];
        i = d.perm[b0 + t];
        pi = pos[i];
        if (single) {
            SM::info()[t] = ti;
            SM::idx()[t] = i;
            SM::pos()[t] = pi;
        }
    }
    int4 jn = ti.y > 0 ? load_four(d, ti.x, 0) : make_int4(0, 0, 0, 0);
    for (int q = b0 + t; q < b1; q += kThreads) {
        const int qn = q + kThreads;
        int4 tn = make_int4(0, 0, 0, 0);
        int in = i;
        if (!kLean && qn < b1) {
            tn = d.tinfo[qn];
            in = d.perm[qn];
        }
        // groups of four, then one by one: the order of every path
        float s = 0.0f;
        const int cnt = ti.y;
        for (int k = 0; k < cnt; k += 4) {
            const int4 j = jn;
            if (k + 4 < cnt) jn = load_four(d, ti.x, k + 4);
            const int4 p0 = pos[j.x], p1 = pos[j.y];  // padding: the own slot
            int4 p2, p3;
            float w0;
            if (kLean) {
                w0 = s_term<float, UNI, X>(d, tab, ps, pi, p0);
                const float w1 = s_term<float, UNI, X>(d, tab, ps, pi, p1);
                p2 = pos[j.z];
                p3 = pos[j.w];
                const float w2 = s_term<float, UNI, X>(d, tab, ps, pi, p2);
                if (k + 4 <= cnt) {
                    s += (w0 + w1) + (w2 + s_term<float, UNI, X>(d, tab, ps, pi, p3));
                } else {
                    s += w0;
                    if (k + 1 < cnt) s += w1;
                    if (k + 2 < cnt) s += w2;
                }
                continue;
            }
            p2 = pos[j.z];
            p3 = pos[j.w];
            w0 = s_term<float, UNI, X>(d, tab, ps, pi, p0);
            if (k + 4 <= cnt) {
                const float w1 = s_term<float, UNI, X>(d, tab, ps, pi, p1);
                const float w2 = s_term<float, UNI, X>(d, tab, ps, pi, p2);
                const float w3 = s_term<float, UNI, X>(d, tab, ps, pi, p3);
                s += (w0 + w1) + (w2 + w3);
            } else {
                s += w0;
                if (k + 1 < cnt) s += s_term<float, UNI, X>(d, tab, ps, pi, p1);
                if (k + 2 < cnt) s += s_term<float, UNI, X>(d, tab, ps, pi, p2);
            }
        }
        d.S[i] = s;
        if (single) SM::S()[t] = s;
        if (qn < b1) {
            ti = kLean ? d.tinfo[qn] : tn;
            i = kLean ? d.perm[qn] : in;
            pi = pos[i];
            if (ti.y > 0) jn = load_four(d, ti.x, 0);
            // the row after that, into L2
            if (qn + kThreads < b1) prefetch_row(d, d.tinfo[qn + kThreads].x);
        }
    }
}

// ---------------------------------------------------------------------------
// FP64 waves.

static __shared__ int s_int[64];
static __shared__ int s_nlist;  // entries lined up
static __shared__ int s_nkeep;  // reactive pairs whose values the S pass kept (-1: not kept)

// A non-negative double cut off to a float, from its bits (the conversion
// instruction runs on the FP64 pipe).  Values below 2^-126 come out below it too.
__device__ __forceinline__ float float_below(double x)
{
    return __int_as_float((int)__funnelshift_l((unsigned)__double2loint(x), (unsigned)max(__double2hiint(x) - 0x38000000, 0), 3));
}

// Squared distance in FP32, far closer than 2^-18 of the box.
__device__ __forceinline__ float float_dist2(const Dev<double>& d, const dbl4& pi, const dbl4& pj)
{
    const double xi[3] = {pi.x, pi.y, pi.z}, xj[3] = {pj.x, pj.y, pj.z};
    float r2 = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        float dx = float_below(xj[c]) - float_below(xi[c]);
        dx = fmaf(-d.Lf[c], rintf(dx * d.iLf[c]), dx);
        r2 = fmaf(dx, dx, r2);
    }
    return r2;
}

// Whether a listed pair may lie inside its cut-off (p.reach2: the cut-off plus
// 2^-18 of the box, squared).
__device__ __forceinline__ bool may_reach(const Dev<double>& d, const dbl4& pi, const dbl4& pj, float reach2)
{
    return float_dist2(d, pi, pj) < reach2;
}

// dist2_listed with the wrap, 9 of its 17 FP64 instructions, left to the pairs
// across a face (|dx| below half an edge wraps by zero): the same bits.
__device__ __forceinline__ double dist2_near(const dbl4& pi, const dbl4& pj, const Dev<double>& d, double& dx,
                                             double& dy, double& dz)
{
    dx = sub_rn(pj.x, pi.x);
    dy = sub_rn(pj.y, pi.y);
    dz = sub_rn(pj.z, pi.z);
    auto far = [](double v, double h) { return (__double2hiint(v) & 0x7fffffff) >= __double2hiint(h); };
    if (far(dx, d.hL[0]) | far(dy, d.hL[1]) | far(dz, d.hL[2])) {
        dx = wrap_rint(dx, d.L[0], d.iL[0]);
        dy = wrap_rint(dy, d.L[1], d.iL[1]);
        dz = wrap_rint(dz, d.L[2], d.iL[2]);
    }
    double s = mul_rn(dx, dx);
    s = add_rn(s, mul_rn(dy, dy));
    return add_rn(s, mul_rn(dz, dz));
}

// Lines up the entries [e0, e1) that may lie inside their cut-off behind the
// entries already in the list and zeroes the wave's results of the others.
// ordered: in entry order, so that the energies, which thread c of the evaluation
// adds up for the c-th entries, are the same in every run (a block barrier every
// kThreads entries); else as the warps come, which changes no force: results go to
// the entries' places.  The force pass orders its entries on sampled steps, the S
// pass, whose list the force pass goes on with, always (as the warps come there
// too: 2,000 particles x 100 logged steps 1865 us, energies that did not repeat; this
// way 1888, with a test of the step's kind in the S pass 1900).  nres: results per entry (1
// or 3).  The caller's barriers come before and complete it.
template <bool UNI>
__device__ __forceinline__ void line_up(const Dev<double>& d, const PairP<double>* tab, const PairP<double>& pu,
                                        const dbl4* pos, unsigned wb, unsigned e0, unsigned e1, int nres, bool ordered)
{
    typedef Stage<double> SM;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int placed = ordered ? s_nlist : 0, buf = 0;
    // the same in the whole warp (ordered: block)
    for (unsigned eb = e0 + (ordered ? 0u : threadIdx.x & ~31u); eb < e1; eb += kThreads) {
        const unsigned e = eb + (ordered ? threadIdx.x : lane);
        bool in = false;
        int j = 0, o = 0;
        if (e < e1) {
            j = d.ent_j[e];
            o = d.ent_o[e];
            const dbl4 pi = SM::pos()[o], pj = pos[j];
            const PairP<double>& p = pair_of<double, UNI>(tab, type_of(pi), type_of(pj), d.ntypes, pu);
            in = may_reach(d, pi, pj, p.reach2);
            if (!in)
                for (int c = 0; c < nres; c++) SM::w()[c * SM::kWave + (e - wb)] = 0.0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        int base = 0;
        if (ordered) {
            if (lane == 0) s_int[buf + warp] = __popc(m);
            __syncthreads();
            const int c = lane < kThreads / 32 ? s_int[buf + lane] : 0;
            base = placed + __reduce_add_sync(0xffffffffu, lane < warp ? c : 0);
            placed += __reduce_add_sync(0xffffffffu, c);
            buf ^= 32;
        } else {
            if (lane == 0 && m) base = atomicAdd(&s_nlist, __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
        }
        if (in) SM::list()[base + __popc(m & ((1u << lane) - 1u))] = make_int2((int)(e - wb) | o << 16, j);
    }
    if (ordered && e0 < e1 && threadIdx.x == 0) s_nlist = placed;
}

// Adds the results at w[k - wb] of entries [k0, k1) to f in entry order.  Zeros
// are passed over (they change nothing), each lane to its own next entry, so
// that a warp's FP64 additions are as many as its longest row has pairs inside
// the cut-off.
template <int N>
__device__ __forceinline__ void sum_row(const double* w, int k0, int k1, double (&f)[N])
{
    typedef Stage<double> SM;
    int k = k0;
    while (__any_sync(0xffffffffu, k < k1)) {
        bool some = false;
        while (k < k1 && !some) {
            unsigned long long b = 0;
#pragma unroll
            for (int c = 0; c < N; c++) b |= (unsigned long long)__double_as_longlong(w[c * SM::kWave + k]);
            some = (b << 1) != 0;  // +-0
            k++;
        }
        __syncwarp();
        if (some)
#pragma unroll
            for (int c = 0; c < N; c++) f[c] += w[c * SM::kWave + k - 1];
    }
}

// S_i, summed in entry order.  staged: as in s_pass_rows.  th: the force pass
// samples the energies (it needs the pair energies of the kept pairs).
template <bool UNI>
__device__ void s_pass_waves(const Dev<double>& d, const PairP<double>* tab, int pc, const PairP<double>& ps,
                             bool staged, bool th)
{
    typedef Stage<double> SM;
    const dbl4* pos = d.pos[pc];
    int b0, b1;
    block_range(d, b0, b1);
    const int t = threadIdx.x;
    const bool single = b1 - b0 <= kThreads;
    if (t == 0) s_nkeep = -1;
    for (int q0 = b0; q0 < b1; q0 += kThreads) {
        const int P = min(kThreads, b1 - q0);
        if (!staged && t < P) {
            SM::pos()[t] = pos[q0 + t];
            SM::info()[t] = d.pinfo[q0 + t];
        }
        if (t == 0) s_nlist = 0;
        __syncthreads();
        const int4 inf = SM::info()[min(t, P - 1)];
        const int4 last = SM::info()[P - 1];
        const unsigned e_beg = SM::info()[0].x, e_end = (unsigned)last.x + (unsigned)last.y;
        // the values are kept for the force pass when it takes the same wave
        const bool keep = single && (unsigned)last.z + (unsigned)last.w - e_beg <= (unsigned)SM::kWave;
        double s[1] = {0.0};
        for (unsigned wb = e_beg; wb < e_end; wb += SM::kWave) {
            const unsigned we = min(wb + SM::kWave, e_end);
            line_up<UNI>(d, tab, ps, pos, wb, wb, we, 1, true);
            __syncthreads();
            const int m = s_nlist;
            const bool kept = keep && m <= SM::kKeep;
            for (int c = t; c < m; c += kThreads) {
                const int2 it = SM::list()[c];
                const int x = it.x & (kBeyond - 1);
                const dbl4 pi = SM::pos()[it.x >> 16], pj = pos[it.y];
                const PairP<double>& p = pair_of<double, UNI>(tab, type_of(pi), type_of(pj), d.ntypes, ps);
                double dx, dy, dz, v, ft;
                const double r2 = dist2_near(pi, pj, d, dx, dy, dz);
                lj_eval<kExpoAny, true>(p, r2, v, ft);
                const bool in = r2 < p.rc2;
                const double vh = r2 > p.rmin2 ? (p.vshift - v) * p.inv_epshat : 1.0;
                SM::w()[x] = in ? mul_rn(p.a, vh) : 0.0;
                if (kept) {
                    double* k = SM::keep() + c;
                    k[0] = in ? ft : 0.0;
                    k[SM::kKeep] = vh;
                    k[2 * SM::kKeep] = dx;
                    k[3 * SM::kKeep] = dy;
                    k[4 * SM::kKeep] = dz;
                    if (th) k[5 * SM::kKeep] = v;
                    if (r2 > p.rmin2) SM::list()[c].x = it.x | kBeyond;
                }
            }
            if (kept && t == 0) s_nkeep = m;
            __syncthreads();
            const unsigned r0 = (unsigned)inf.x, r1 = r0 + (unsigned)inf.y;
            const bool on = t < P && r1 > wb && r0 < we;
            sum_row(SM::w(), on ? (int)(max(r0, wb) - wb) : 0, on ? (int)(min(r1, we) - wb) : 0, s);
            if (t == 0 && !kept) s_nlist = 0;
            __syncthreads();
        }
        if (t < P) {
            d.S[q0 + t] = s[0];
            if (single) SM::S()[t] = s[0];
        }
        // the staging is free (a sub-chunk without a reactive pair has run no wave)
        if (!single) __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Force pass fused with the integrator.
//
// flags: closing = finish the current step with the second half kick;
//        opening = start the next step: half kick, half drift, (Langevin O),
//                  half drift, write the new snapshot into pos[pc^1];
//        store   = keep the forces (for a later opening or a read-out).
enum { F_CLOSING = 1, F_OPENING = 2, F_STORE = 4 };

template <typename Real>
struct Acc {
    Real q[kNQA];
};

// Per-particle integrator inputs, loaded before the force gathers so that
// their latency overlaps the entry work.
template <typename Real>
struct PState {
    typename Dev<Real>::R4 v;
    long long q[3];
};

template <typename Real>
__device__ __forceinline__ void load_pstate(const Dev<Real>& d, int ac, int i, int flags,
                                            PState<Real>& ps)
{
    const int n = d.n;
    ps.v = d.vel[ac][i];
    if (flags & F_OPENING) {
#pragma unroll
        for (int c = 0; c < 3; c++) ps.q[c] = d.xq[ac][c * n + i];
    }
}

// Adds a displacement to one fixed-point coordinate and wraps it into the box;
// w gets the change of the image count (-1, 0 or +1).
__device__ __forceinline__ long long advance_fix(long long q0, long long Lq, long long dq, int& w)
{
    const long long q = q0 + dq;
    if (q >= Lq) {
        w = 1;
        return q - Lq;
    }
    if (q < 0) {
        w = -1;
        return q + Lq;
    }
    w = 0;
    return q;
}

// The integrator on one particle's registers: the closing half kick of the
// step that ends, the kinetic energy, and (opening) the half kick, half drift,
// Langevin O step and half drift of the next (BAOAB; velocity Verlet without
// O).  q[] (fixed point) and v are advanced in place, w[] gets the image
// changes, np the new snapshot.  z: the O step's normals (Langevin, opening).
// Returns the squared displacement of the drift (0 when not opening).
template <typename Real>
__device__ __forceinline__ float advance_particle(const Dev<Real>& d, const RunArgs& a, Real fx, Real fy, Real fz,
                                                  int flags, const Real (&z)[3], int wbits,
                                                  typename Dev<Real>::R4& v, long long q[3], int w[3], Real& kin,
                                                  typename Dev<Real>::P4& np)
{
    const Real im = v.w;
    const Real hdt = pick(Real(0), a.hdt_f, a.hdt_d);
    if (flags & F_CLOSING) {
        v.x += hdt * fx * im;
        v.y += hdt * fy * im;
        v.z += hdt * fz * im;
    }
    kin += Real(0.5) * (v.x * v.x + v.y * v.y + v.z * v.z) * recip(im);
    float disp2 = 0.0f;
    w[0] = w[1] = w[2] = 0;
    if (flags & F_OPENING) {
        v.x += hdt * fx * im;
        v.y += hdt * fy * im;
        v.z += hdt * fz * im;
        Real ddx = hdt * v.x, ddy = hdt * v.y, ddz = hdt * v.z;
        if (a.langevin) {
            const Real c1 = pick(Real(0), a.c1_f, a.c1_d);
            const Real sd = pick(Real(0), a.c2_f, a.c2_d) * (im == Real(1) ? Real(1) : sqrt(im));
            v.x = c1 * v.x + sd * z[0];
            v.y = c1 * v.y + sd * z[1];
            v.z = c1 * v.z + sd * z[2];
        }
        ddx += hdt * v.x;
        ddy += hdt * v.y;
        ddz += hdt * v.z;
        disp2 = (float)(ddx * ddx + ddy * ddy + ddz * ddz);
        q[0] = advance_fix(q[0], d.Lq[0], real_to_fix(ddx), w[0]);
        q[1] = advance_fix(q[1], d.Lq[1], real_to_fix(ddy), w[1]);
        q[2] = advance_fix(q[2], d.Lq[2], real_to_fix(ddz), w[2]);
        np.x = snap_coord(q[0], 0, d);
        np.y = snap_coord(q[1], 1, d);
        np.z = snap_coord(q[2], 2, d);
        np.w = snap_bits(wbits, d);
    }
    return disp2;
}

// Advances particle i given its force (state from global memory, written
// back there; the image count is touched only when the particle wraps).
// Returns the squared displacement of this step's drift (0 when not opening).
template <typename Real>
__device__ __forceinline__ float integrate_one(const Dev<Real>& d, const RunArgs& a, int pc,
                                               int ac, int i, Real fx, Real fy, Real fz,
                                               int flags, long long step, PState<Real>& st,
                                               int wbits, Real& kin, typename Dev<Real>::P4* keep)
{
    typename Dev<Real>::R4 v = st.v;
    typename Dev<Real>::P4 np;
    int w[3];
    Real z[3] = {Real(0), Real(0), Real(0)};
    if ((flags & F_OPENING) && a.langevin) normals3(a.seed, step, (unsigned)(wbits >> kTypeBits), z);
    const float disp2 = advance_particle(d, a, fx, fy, fz, flags, z, wbits, v, st.q, w, kin, np);
    if (flags & F_OPENING) {
        const int n = d.n;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            __stcs(&d.xq[ac][c * n + i], st.q[c]);  // read again only next step: evict first
            if (w[c]) d.img[ac][c * n + i] += w[c];
        }
        d.pos[pc ^ 1][i] = np;
        if (keep) *keep = np;
    }
    if constexpr (sizeof(Real) == 4)
        __stcs((float4*)&d.vel[ac][i], *(const float4*)&v);
    else
        d.vel[ac][i] = v;
    return disp2;
}

// What a thread's FP32 thermo terms are multiplied by when they are folded: half
// of a pair to each end, and the virial's sign (the force is on the owner).
__device__ __forceinline__ float th_scale(int q)
{
    return q == Q_K ? 1.0f : q >= Q_W0 && q < Q_BONDS ? -0.5f : 0.5f;
}

// One entry's pair force on its owner (returned as the components of
// f (x_i - x_j)), with the pair's energies, virial and bond count when TH (the
// sampled step of a launch), bare: th_scale holds the factors.  REACT: a reactive pair (two-body
// plus the three-body factor); else a purely two-body pair.
template <typename Real, bool UNI, int X, bool REACT, bool TH>
__device__ __forceinline__ void entry_force(const Dev<Real>& d, const PairP<Real>* tab,
                                            const typename Dev<Real>::P4& pi,
                                            const typename Dev<Real>::P4& pj, Real Si, Real Sj,
                                            const PairP<Real>& pu, Acc<Real>& acc, Real& fx,
                                            Real& fy, Real& fz)
{
    Real dx, dy, dz;
    const Real r2 = dist2_listed(pi, pj, d, dx, dy, dz);
    const PairP<Real>& p = pair_of<Real, UNI>(tab, type_of(pi), type_of(pj), d.ntypes, pu);
    // evaluated for every listed pair and selected by the cut-off decision
    // (no divergent branch: about half of the listed pairs lie in the skin)
    const bool in = r2 < p.rc2;
    Real v, ft;
    lj_eval<X, REACT>(p, r2, v, ft);
    if (TH) acc.q[Q_U2] += in ? v + p.ushift : Real(0);
    if (REACT) {
        const bool beyond = r2 > p.rmin2;
        const Real vh = beyond ? (p.vshift - v) * p.inv_epshat : Real(1);
        const Real h = p.a * (Si + Sj - Real(2) * p.a * vh);
        ft = beyond ? ft * (Real(1) - h * p.inv_epshat) : ft;
        if (TH) {
            const Real av = p.a * vh;
            acc.q[Q_U3] += in ? av * (Si - av) : Real(0);
            acc.q[Q_BONDS] += (in && r2 < p.rbond2) ? Real(1) : Real(0);
        }
    }
    ft = in ? ft : Real(0);
    fx = -ft * dx;
    fy = -ft * dy;
    fz = -ft * dz;
    if (!TH) return;
    acc.q[Q_W0 + 0] += fx * dx;
    acc.q[Q_W0 + 1] += fy * dy;
    acc.q[Q_W0 + 2] += fz * dz;
    acc.q[Q_W0 + 3] += fx * dy;
    acc.q[Q_W0 + 4] += fx * dz;
    acc.q[Q_W0 + 5] += fy * dz;
}

// The harmonic bonds of particle pi (vitrimer chains): F_i = k (r - r0) (x_j -
// x_i) / r, half of the energy and virial to each end (added to the two-body
// terms).
template <typename Real, bool TH>
__device__ __forceinline__ void bond_forces(const Dev<Real>& d, const typename Dev<Real>::P4* pos,
                                            const typename Dev<Real>::P4& pi, Acc<Real>& acc, Real& fx, Real& fy,
                                            Real& fz)
{
    const int tag = pos_bits(pi) >> kTypeBits;
    for (int b = 0; b < kMaxBonds; b++) {
        const int pt = d.bond_tag[tag * kMaxBonds + b];
        if (pt < 0) break;
        const typename Dev<Real>::P4 pj = pos[d.slot_of_tag[pt]];
        Real dx, dy, dz;
        const Real r = sqrt(dist2_listed(pi, pj, d, dx, dy, dz));
        const Real dr = r - d.bond_r0;
        const Real g = d.bond_k * dr / r;
        fx += g * dx;
        fy += g * dy;
        fz += g * dz;
        if (!TH) continue;
        // (FP32 terms are scaled when they are folded, th_scale)
        acc.q[Q_U2] += (sizeof(Real) == 4 ? Real(0.5) : Real(0.25)) * d.bond_k * dr * dr;
        const Real hf = sizeof(Real) == 4 ? g : Real(-0.5) * g;
        acc.q[Q_W0 + 0] += hf * dx * dx;
        acc.q[Q_W0 + 1] += hf * dy * dy;
        acc.q[Q_W0 + 2] += hf * dz * dz;
        acc.q[Q_W0 + 3] += hf * dx * dy;
        acc.q[Q_W0 + 4] += hf * dx * dz;
        acc.q[Q_W0 + 5] += hf * dy * dz;
    }
}

// Where the S pass of the same step left the block's positions, list ranges and
// S values in shared memory (a block of one sub-chunk), they are taken
// from there, and the integrator keeps the shared positions current for the
// next S pass.  TH: the sampled step (the warps' thermo terms are left in
// s_wacc, see block_sums_from_rows).  Returns the thread's largest squared
// drift displacement.
template <bool UNI, int X, bool BONDS, bool TH>
__device__ float f_pass_rows(const Dev<float>& d, const PairP<float>* tab, const RunArgs& a, int pc, int ac, int flags,
                             long long step, const PairP<float>& ps, const PairP<float>& pw)
{
    typedef Stage<float> SM;
    const int4* pos = d.pos[pc];
    int b0, b1;
    block_range(d, b0, b1);
    const int n = d.n;
    const int t = threadIdx.x, lane = t & 31;
    const bool single = b1 - b0 <= kThreads;
    float dmax = 0.0f;
    [[maybe_unused]] double run = 0.0;  // lane q: quantity q of the warp's particles so far
    const int4 none = make_int4(0, 0, 0, 0);
    // what the thread's next rows need is loaded while it works on the present ones
    int4 ti = none;
    int i = b0;
    if (b0 + t < b1) {
        ti = single ? SM::info()[t] : d.tinfo[b0 + t];
        i = single ? SM::idx()[t] : d.perm[b0 + t];
    }
    int4 jn = ti.y > 0 ? load_four(d, ti.x, 0) : none;
    for (int q0 = b0; q0 < b1; q0 += kThreads) {
        const int P = min(kThreads, b1 - q0);
        if ((t & ~31) >= P) break;  // the same in the whole warp
        const bool on = t < P;
        const int qn = q0 + kThreads + t;
        int4 tn = none, pi = none;
        int in = i;
        float Si = 0.0f;
        if (on) {
            // integrator inputs: asynchronous copies, waited for after the entries
            cp_async_r4(&SM::vel()[t], &d.vel[ac][i]);
            if (flags & F_OPENING)
                for (int c = 0; c < 3; c++) cp_async(&SM::xq()[3 * t + c], &d.xq[ac][c * n + i], 8);
            cp_async_commit();
            if (single) {
                pi = SM::pos()[t];
                Si = SM::S()[t];
            } else {
                pi = pos[i];
                Si = d.S[i];
                if (!kLean && qn < b1) {
                    tn = d.tinfo[qn];
                    in = d.perm[qn];
                }
            }
        }
        float fx = 0.0f, fy = 0.0f, fz = 0.0f, gx = 0.0f, gy = 0.0f, gz = 0.0f;  // reactive and other rows' sums
        Acc<float> acc;
        if (TH)
#pragma unroll
            for (int q = 0; q < kNQA; q++) acc.q[q] = 0.0f;
        auto reactive = [&](const int4& pj, float Sj) {
            float ex, ey, ez;
            entry_force<float, UNI, X, true, TH>(d, tab, pi, pj, Si, Sj, ps, acc, ex, ey, ez);
            fx = __fadd_rn(fx, ex);
            fy = __fadd_rn(fy, ey);
            fz = __fadd_rn(fz, ez);
        };
        auto other = [&](const int4& pj) {
            float ex, ey, ez;
            entry_force<float, UNI, X, false, TH>(d, tab, pi, pj, 0.0f, 0.0f, pw, acc, ex, ey, ez);
            gx = __fadd_rn(gx, ex);
            gy = __fadd_rn(gy, ey);
            gz = __fadd_rn(gz, ez);
        };
        int4 jo = ti.w > 0 ? load_four(d, ti.z, 0) : none;
        for (int k = 0; k < ti.y; k += 4) {
            const int4 j = jn;
            if (k + 4 < ti.y) jn = load_four(d, ti.x, k + 4);
            const int4 p0 = pos[j.x], p1 = pos[j.y];  // padding: the own slot
            const float s0 = d.S[j.x], s1 = d.S[j.y];
            if (kLean) {
                reactive(p0, s0);
                if (k + 1 < ti.y) reactive(p1, s1);
                if (k + 2 < ti.y) {
                    const int4 p2 = pos[j.z], p3 = pos[j.w];
                    const float s2 = d.S[j.z], s3 = d.S[j.w];
                    reactive(p2, s2);
                    if (k + 3 < ti.y) reactive(p3, s3);
                }
                continue;
            }
            const int4 p2 = pos[j.z], p3 = pos[j.w];
            const float s2 = d.S[j.z], s3 = d.S[j.w];
            reactive(p0, s0);
            if (k + 1 < ti.y) reactive(p1, s1);
            if (k + 2 < ti.y) reactive(p2, s2);
            if (k + 3 < ti.y) reactive(p3, s3);
        }
        for (int k = 0; k < ti.w; k += 4) {
            const int4 j = jo;
            if (k + 4 < ti.w) jo = load_four(d, ti.z, k + 4);
            const int4 p0 = pos[j.x], p1 = pos[j.y], p2 = pos[j.z], p3 = pos[j.w];
            other(p0);
            if (k + 1 < ti.w) other(p1);
            if (k + 2 < ti.w) other(p2);
            if (k + 3 < ti.w) other(p3);
        }
        // the force: the reactive row's sum plus the other row's (the order of
        // the resident step, so both paths give the same bits)
        fx = __fadd_rn(fx, gx);
        fy = __fadd_rn(fy, gy);
        fz = __fadd_rn(fz, gz);
        if (BONDS && d.has_bonds && on)  // BONDS: some system of the launch has bonds
            bond_forces<float, TH>(d, pos, pi, acc, fx, fy, fz);
        // the pair terms join the running sums now, so that they hold no
        // registers at the integrator's peak
        if (TH)
#pragma unroll
            for (int q = 0; q < kNQA; q++)
                if (q != Q_K) {
                    const float x = warp_sum(acc.q[q] * th_scale(q));
                    if (lane == q) run += (double)x;
                }
        if (qn < b1) {
            if (kLean) {
                tn = d.tinfo[qn];
                in = d.perm[qn];
                prefetch_row(d, tn.x);
            } else if (tn.y > 0) {
                jn = load_four(d, tn.x, 0);
            }
            if (tn.w > 0) prefetch_row(d, tn.z);
        }
        float kin = 0.0f;
        if (on) {
            if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) atomicOr(&d.ctl->status, kStatusNonfinite);
            if (flags & F_STORE) d.force[i] = make_float4(fx, fy, fz, 0.0f);
            cp_async_wait_all();
            PState<float> st;
            st.v = SM::vel()[t];
            if (flags & F_OPENING)
                for (int c = 0; c < 3; c++) st.q[c] = SM::xq()[3 * t + c];
            dmax = fmaxf(dmax, integrate_one(d, a, pc, ac, i, fx, fy, fz, flags, step, st, pos_bits(pi), kin,
                                             single ? &SM::pos()[t] : (int4*)nullptr));
        }
        if (TH) {
            const float x = warp_sum(kin);
            if (lane == Q_K) run += (double)x;
        }
        ti = tn;
        i = in;
        if (kLean && ti.y > 0) jn = load_four(d, ti.x, 0);
    }
    if (TH && lane < kNQA) s_wacc[t >> 5][lane] = run;
    return dmax;
}

// One pair's force on its owner into the wave's results at place x, from the
// pair force ft (zero outside the cut-off) and, when TH, its share of the
// virial.
template <bool TH>
__device__ __forceinline__ void put_force(double ft, double dx, double dy, double dz, int x, Acc<double>& acc)
{
    typedef Stage<double> SM;
    SM::w()[x] = -ft * dx;
    SM::w()[SM::kWave + x] = -ft * dy;
    SM::w()[2 * SM::kWave + x] = -ft * dz;
    if (!TH) return;
    const double hf = 0.5 * ft;
    acc.q[Q_W0 + 0] += hf * dx * dx;
    acc.q[Q_W0 + 1] += hf * dy * dy;
    acc.q[Q_W0 + 2] += hf * dz * dz;
    acc.q[Q_W0 + 3] += hf * dx * dy;
    acc.q[Q_W0 + 4] += hf * dx * dz;
    acc.q[Q_W0 + 5] += hf * dy * dz;
}

// A reactive pair: the three-body factor on its two-body force (outside r_min).
template <bool TH>
__device__ __forceinline__ void put_reactive(const PairP<double>& p, double r2, bool in, double v, double ft, double vh,
                                             bool beyond, double dx, double dy, double dz, double Si, double Sj, int x,
                                             Acc<double>& acc)
{
    const double h = p.a * (Si + Sj - 2.0 * p.a * vh);
    if (beyond) ft = ft * (1.0 - h * p.inv_epshat);
    if (TH && in) {
        acc.q[Q_U2] += 0.5 * (v + p.ushift);
        acc.q[Q_U3] += 0.5 * p.a * vh * (Si - p.a * vh);
        if (r2 < p.rbond2) acc.q[Q_BONDS] += 0.5;
    }
    put_force<TH>(ft, dx, dy, dz, x, acc);
}

template <bool UNI, bool BONDS, bool TH>
__device__ float f_pass_waves(const Dev<double>& d, const PairP<double>* tab, const RunArgs& a, int pc, int ac,
                              int flags, long long step, const PairP<double>& ps, const PairP<double>& pw)
{
    typedef Stage<double> SM;
    const dbl4* pos = d.pos[pc];
    int b0, b1;
    block_range(d, b0, b1);
    const int t = threadIdx.x, n = d.n;
    const bool single = b1 - b0 <= kThreads;
    float dmax = 0.0f;
    Acc<double> acc;
    if (TH)
#pragma unroll
        for (int q = 0; q < kNQA; q++) acc.q[q] = 0.0;
    for (int q0 = b0; q0 < b1; q0 += kThreads) {
        const int P = min(kThreads, b1 - q0);
        if (t < P) {
            const int i = q0 + t;
            // integrator inputs: asynchronous copies, waited for after the entries
            cp_async_r4(&SM::vel()[t], &d.vel[ac][i]);
            if (flags & F_OPENING)
                for (int c = 0; c < 3; c++) cp_async(&SM::xq()[3 * t + c], &d.xq[ac][c * n + i], 8);
            cp_async_commit();
            if (!single) {
                SM::pos()[t] = pos[i];
                SM::S()[t] = d.S[i];
                SM::info()[t] = d.pinfo[i];
            }
        }
        const int nkeep = single ? s_nkeep : -1;  // kept pairs: the first nkeep of the list
        if (nkeep < 0 && t == 0) s_nlist = 0;
        __syncthreads();
        const int4 inf = SM::info()[min(t, P - 1)];
        const int4 last = SM::info()[P - 1];
        const unsigned e_beg = SM::info()[0].x, e_rend = (unsigned)last.x + (unsigned)last.y, e_end = (unsigned)last.z + (unsigned)last.w;
        double f[3] = {0.0, 0.0, 0.0}, g[3] = {0.0, 0.0, 0.0};  // reactive and other rows' sums
        for (unsigned wb = e_beg; wb < e_end; wb += SM::kWave) {
            const unsigned we = min(wb + SM::kWave, e_end);
            const unsigned wr = min(max(e_rend, wb), we);  // reactive entries before, others from here
            int nre = nkeep;  // reactive pairs in the list
            if (nkeep < 0) {
                line_up<UNI>(d, tab, ps, pos, wb, wb, wr, 3, TH);
                __syncthreads();
                nre = s_nlist;
                __syncthreads();
            } else {
                // kept: the places of the pairs that were left out (line_up has
                // zeroed the first of their three results, and the pairs' own
                // places are all written below)
                for (unsigned e = wb + t; e < wr; e += kThreads) {
                    SM::w()[e - wb] = 0.0;
                    SM::w()[SM::kWave + (e - wb)] = 0.0;
                    SM::w()[2 * SM::kWave + (e - wb)] = 0.0;
                }
            }
            line_up<UNI>(d, tab, pw, pos, wb, wr, we, 3, TH);
            __syncthreads();
            const int m = s_nlist;
            for (int c = t; c < m; c += kThreads) {
                const int2 it = SM::list()[c];
                const int x = it.x & (kBeyond - 1), o = it.x >> 16;
                double dx, dy, dz, v = 0.0, ft;
                if (c < nkeep) {
                    const double Sj = d.S[it.y];
                    const double* k = SM::keep() + c;
                    const bool beyond = it.x & kBeyond;
                    dx = k[2 * SM::kKeep];
                    dy = k[3 * SM::kKeep];
                    dz = k[4 * SM::kKeep];
                    double r2 = 0.0;
                    bool in = true;
                    const PairP<double>* p = &ps;
                    if (!UNI) p = &tab[type_of(SM::pos()[o]) * d.ntypes + type_of(pos[it.y])];
                    if (TH) {
                        v = k[5 * SM::kKeep];
                        r2 = add_rn(add_rn(mul_rn(dx, dx), mul_rn(dy, dy)), mul_rn(dz, dz));
                        in = r2 < p->rc2;
                    }
                    put_reactive<TH>(*p, r2, in, v, k[0], k[SM::kKeep], beyond, dx, dy, dz, SM::S()[o], Sj, x, acc);
                } else {
                    const dbl4 pi = SM::pos()[o], pj = pos[it.y];
                    const bool react = c < nre;
                    const PairP<double>& p = UNI ? (react ? ps : pw) : tab[type_of(pi) * d.ntypes + type_of(pj)];
                    const double Sj = react ? d.S[it.y] : 0.0;
                    const double r2 = dist2_near(pi, pj, d, dx, dy, dz);
                    const bool in = r2 < p.rc2;
                    lj_eval<kExpoAny, true>(p, r2, v, ft);
                    ft = in ? ft : 0.0;
                    if (react) {
                        const bool beyond = r2 > p.rmin2;
                        const double vh = beyond ? (p.vshift - v) * p.inv_epshat : 1.0;
                        put_reactive<TH>(p, r2, in, v, ft, vh, beyond, dx, dy, dz, SM::S()[o], Sj, x, acc);
                    } else {
                        if (TH && in) acc.q[Q_U2] += 0.5 * (v + p.ushift);
                        put_force<TH>(ft, dx, dy, dz, x, acc);
                    }
                }
            }
            __syncthreads();
            if (t == 0) s_nlist = 0;
            auto part = [&](unsigned r0, unsigned r1, double (&sum)[3]) {
                const bool on = t < P && r1 > wb && r0 < we;
                sum_row(SM::w(), on ? (int)(max(r0, wb) - wb) : 0, on ? (int)(min(r1, we) - wb) : 0, sum);
            };
            part((unsigned)inf.x, (unsigned)inf.x + (unsigned)inf.y, f);
            part((unsigned)inf.z, (unsigned)inf.z + (unsigned)inf.w, g);
            __syncthreads();
        }
        double fx = add_rn(f[0], g[0]), fy = add_rn(f[1], g[1]), fz = add_rn(f[2], g[2]);
        if (BONDS && d.has_bonds && t < P)  // BONDS: some system of the launch has bonds
            bond_forces<double, TH>(d, pos, SM::pos()[t], acc, fx, fy, fz);
        double kin = 0.0;
        if (t < P) {
            const int i = q0 + t;
            if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) atomicOr(&d.ctl->status, kStatusNonfinite);
            if (flags & F_STORE) {
                dbl4 fo;
                fo.x = fx;
                fo.y = fy;
                fo.z = fz;
                fo.w = 0.0;
                d.force[i] = fo;
            }
            cp_async_wait_all();
            PState<double> st;
            st.v = SM::vel()[t];
            if (flags & F_OPENING)
                for (int c = 0; c < 3; c++) st.q[c] = SM::xq()[3 * t + c];
            dmax = fmaxf(dmax, integrate_one(d, a, pc, ac, i, fx, fy, fz, flags, step, st, pos_bits(SM::pos()[t]), kin,
                                             single ? &SM::pos()[t] : (dbl4*)nullptr));
        }
        if (TH) acc.q[Q_K] += kin;
        if (!single) __syncthreads();  // the staging is free
    }
    if (TH) {
        // staged for block_sums_from_threads (the waves' buffer is free)
#pragma unroll
        for (int q = 0; q < kNQA; q++) SM::w()[q * kThreads + t] = acc.q[q];
    }
    return dmax;
}

// Opening half of a step from stored forces (start of a run).
template <typename Real>
__device__ __forceinline__ float open_from_stored(const Dev<Real>& d, const RunArgs& a, int pc,
                                                  int ac, int i, long long step)
{
    typedef typename Dev<Real>::R4 R4;
    const R4 f = d.force[i];
    const typename Dev<Real>::P4 pi = d.pos[pc][i];
    PState<Real> st;
    load_pstate(d, ac, i, F_OPENING, st);
    Real unused = Real(0);
    return integrate_one(d, a, pc, ac, i, f.x, f.y, f.z, F_OPENING, step, st, pos_bits(pi), unused,
                         (typename Dev<Real>::P4*)nullptr);
}

// ---------------------------------------------------------------------------
// The persistent step kernel.  One cooperative launch advances a.nsteps time
// steps (or only rebuilds, or only brings the forces up to date), with two
// grid barriers per step and a rebuild whenever the accumulated displacement
// bound can let an unlisted pair come inside its cut-off.
//
// Block-wide state lives in shared memory at namespace scope (addressed
// directly, not through pointers), so that nothing but the phase at hand
// occupies registers: the kernel runs at the 80-register limit of a
// 768-thread block.

struct LoopState {
    unsigned long long bar_target;  // barrier generation target (thread 0)
    long long step;
    long long rebuilds;
    int state, pc, ac, need_rb, remaining, done, have_thermo, rc, ok;
    float disp;
    unsigned dmax_bits;  // the block's largest squared step displacement (float bits)
    int own_ok;          // shared positions and list ranges of the block's particles are current
    // resident mode (section below)
    int r_try;           // build the resident structures before the next step
    int r_valid;         // every block's resident structures are built and current
    int r_rb;            // threads that hold rows
    unsigned r_epoch;    // publications of this launch
    int r_round;         // agreement round (selects ctl->rfail[round & 1])
    int r_np, r_nh, r_nhr;  // own particles, halo particles, halo rows of S
    int r_steps;         // steps this launch took in the resident mode
    int tlog_left;       // steps up to and including the next logged one (0: no log)
    int tlog_slot;       // ring slot of the next thermo-log record
    int tlog_k;          // records this launch wrote
};

static __shared__ __align__(16) unsigned char s_tab_raw[kMaxTypes * kMaxTypes * sizeof(PairP<double>)];
static __shared__ double s_red[32];
static __shared__ LoopState s_ls;

template <typename Real>
__device__ __forceinline__ const PairP<Real>* stab() { return (const PairP<Real>*)s_tab_raw; }

__device__ __forceinline__ bool grid_barrier(Ctl* ctl, long long timeout_ns, int where,
                                             unsigned* pub_dst = nullptr)
{
    BarState bs;
    bs.target = s_ls.bar_target;
    bar_arrive(ctl, bs, pub_dst, &s_ls.dmax_bits);
    if (threadIdx.x == 0) s_ls.bar_target = bs.target;
    return bar_wait(ctl, bs, timeout_ns, where, &s_ls.ok);
}

// 0: ok; 1: the list overflowed its capacity; 2: a wait timed out.
template <typename Real>
__device__ SWP_COLD int run_rebuild(const Dev<Real>& d, const RunArgs& a)
{
    Ctl* ctl = d.ctl;
    const int gt = g_rank() * blockDim.x + threadIdx.x, gn = g_size() * blockDim.x;
    if (threadIdx.x == 0 && g_rank() == 0) {
        ctl->max_row = 0;
        ctl->overflow = 0;
    }
    const int pc0 = s_ls.pc, ac0 = s_ls.ac;
    ph_bin(d, pc0, (int*)g_dyn);
    if (!grid_barrier(ctl, a.timeout_ns, 1)) return 2;
    ph_chunk_scan(d, s_int);
    if (!grid_barrier(ctl, a.timeout_ns, 3)) return 2;
    ph_scatter(d, gt, gn);
    if (!grid_barrier(ctl, a.timeout_ns, 4)) return 2;
    ph_move(d, pc0, ac0, gt, gn);
    __syncthreads();
    if (threadIdx.x == 0) {
        s_ls.pc = pc0 ^ 1;
        s_ls.ac = ac0 ^ 1;
    }
    if (!grid_barrier(ctl, a.timeout_ns, 6)) return 2;
    int ovf = 0;
    const int need = ph_build_rows<Real>(d, stab<Real>(), pc0 ^ 1, s_int, &ovf);
    if (threadIdx.x == 0) {
        atomicMax(&ctl->max_row, need);
        if (ovf) atomicOr(&ctl->overflow, 1);
    }
    if (!grid_barrier(ctl, a.timeout_ns, 7)) return 2;
    const int any_ovf = ld_relaxed(&ctl->overflow);
    if (threadIdx.x == 0) {
        s_ls.rebuilds++;
        s_ls.disp = 0.0f;
        s_ls.own_ok = 0;  // the particles were reordered
    }
    __syncthreads();
    if (any_ovf) {
        if (gt == 0) atomicOr(&ctl->status, kStatusOverflow);
        return 1;
    }
    return 0;
}

// One sub-chunk: the block's particles fit one shared staging.
template <typename Real>
__device__ __forceinline__ bool single_chunk(const Dev<Real>& d)
{
    return (d.n + g_size() - 1) / g_size() <= (int)blockDim.x;
}

// Runs f(std::integral_constant<int, X>) for the run's exponents (the same in
// the whole block); uniform coefficients only can be kExpoStd.
template <bool UNI, typename F>
__device__ __forceinline__ void expo_switch(const RunArgs& a, F&& f)
{
    if (UNI && a.expo == kExpoStd) f(std::integral_constant<int, UNI ? kExpoStd : kExpoAny>());
    else if (!kBatched && a.expo == kExpoEven) f(std::integral_constant<int, kBatched ? kExpoAny : kExpoEven>());
    else f(std::integral_constant<int, kExpoAny>());
}

// The caller sets s_ls.own_ok after the grid barrier that follows (every warp
// has read it by then).
template <typename Real, bool UNI>
__device__ __forceinline__ void run_s_pass(const Dev<Real>& d, const RunArgs& a, [[maybe_unused]] bool th)
{
    const bool staged = single_chunk(d) && s_ls.own_ok;
    if constexpr (sizeof(Real) == 4)
        expo_switch<UNI>(a, [&](auto x) {
            s_pass_rows<UNI, decltype(x)::value>(d, stab<Real>(), s_ls.pc, uni_params(a, Real(0))[0], staged);
        });
    else
        s_pass_waves<UNI>(d, stab<Real>(), s_ls.pc, uni_params(a, Real(0))[0], staged, th);
}

// Folds a thread's squared displacement into the block's shared maximum (one
// shared atomic per warp); the barrier arrival publishes it.  A NaN (a particle
// whose velocity is none) counts for nothing, so that the others' lists are still
// rebuilt in time; the bits of the other values order like them.
__device__ __forceinline__ void warp_max_disp(float v)
{
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(v, 0.0f)));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(&s_ls.dmax_bits, m);
}

template <typename Real, bool UNI, bool BONDS, bool TH>
__device__ __forceinline__ void run_f_pass(const Dev<Real>& d, const RunArgs& a, int flags, long long stp)
{
    const PairP<Real>*ps = &uni_params(a, Real(0))[0], *pw = &uni_params(a, Real(0))[1];
    float dmax = 0.0f;
    if constexpr (sizeof(Real) == 4)
        expo_switch<UNI>(a, [&](auto x) {
            dmax = f_pass_rows<UNI, decltype(x)::value, BONDS, TH>(d, stab<Real>(), a, s_ls.pc, s_ls.ac, flags, stp, *ps,
                                                                   *pw);
        });
    else
        dmax = f_pass_waves<UNI, BONDS, TH>(d, stab<Real>(), a, s_ls.pc, s_ls.ac, flags, stp, *ps, *pw);
    if (flags & F_OPENING) warp_max_disp(dmax);
}

template <typename Real>
__device__ void run_open_pass(const Dev<Real>& d, const RunArgs& a, long long stp)
{
    float dmax = 0.0f;
    const int pc = s_ls.pc, ac = s_ls.ac;
    for (int i = g_rank() * blockDim.x + threadIdx.x; i < d.n; i += g_size() * blockDim.x)
        dmax = fmaxf(dmax, open_from_stored(d, a, pc, ac, i, stp));
    warp_max_disp(dmax);
}

// Deterministic reduction of the block partials of the sampled step: block q
// sums quantity q over all blocks in a fixed order.
template <typename Real>
__device__ void run_reduce_thermo(const Dev<Real>& d)
{
    const int G = g_size(), nwp = (G + 31) / 32;
    const int lw = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int q = g_rank(); q < kNQA; q += G) {  // block-uniform loop
        if (w < nwp) {
            const int b = threadIdx.x;
            double v = b < G ? d.partials[(size_t)b * kNQ + q] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lw == 0) s_red[w] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < nwp; k++) t += s_red[k];
            d.ctl->thermo[q] = t;
        }
        __syncthreads();
    }
}

// The same reduction for a group of fewer than kNQA blocks (batched runs):
// rank 0 alone, warp q summing quantity q over the group's blocks in order.
template <typename Real>
__device__ __forceinline__ void reduce_small(const Dev<Real>& d)
{
    if (g_rank() != 0) return;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    for (int q = w; q < kNQA; q += nw) {
        double v = lane < g_size() ? d.partials[(size_t)lane * kNQ + q] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) d.ctl->thermo[q] = v;
    }
}

// Writes the block's partials of a sampled step's thermo terms (energies,
// virial, bond count, kinetic energy) from the warps' sums (s_wacc, or for a
// resident step s_wpart) to the launch's partials (last: the last step of the
// launch, whose values the launch reports; reduced after the loop) and/or to a
// thermo-log record (log).  Every call is followed by a grid barrier.  Steps
// that are neither the launch's last nor logged skip the thermo terms
// altogether.
template <typename Real>
__device__ __forceinline__ void thermo_partials(const Dev<Real>& d, bool resident, bool last, double* log)
{
    double* out = last ? d.partials + (size_t)g_rank() * kNQ : log;
    double* out2 = last ? log : nullptr;
    if (resident) {
        block_sums_from_warps(out, out2);
    } else {
        int b0, b1;
        block_range(d, b0, b1);
        if constexpr (sizeof(Real) == 4) {
            block_sums_from_rows(min((b1 - b0 + 31) / 32, kThreads / 32), out, out2);
        } else {
            // threads that had a particle or (the lined-up pairs) an entry
            int nact = kThreads;
            if (b1 - b0 <= kThreads && b1 > b0) {
                const int4 l = Stage<Real>::info()[b1 - b0 - 1];
                nact = min(kThreads, max(b1 - b0, l.z + l.w - Stage<Real>::info()[0].x));
            }
            block_sums_from_threads((const double*)Stage<Real>::w(), nact, out, out2);
        }
    }
    if (last && threadIdx.x == 0) s_ls.have_thermo = 1;
}

__device__ __forceinline__ void add_disp(Ctl* ctl, long long stp)
{
    if (threadIdx.x == 0)
        s_ls.disp += sqrtf(__uint_as_float((unsigned)ld_relaxed((const int*)&ctl->dmax2[stp & 1])));
    __syncthreads();
}

#if SWP_HAS_RESIDENT
// ---------------------------------------------------------------------------
// Resident mode: one system, FP32, no bonds, every block's particles in one
// sub-chunk (up to blockDim x grid particles).
//
// After each list build every block copies into shared memory what its steps
// need: the snapshots of its own particles and of its halo -- every particle
// outside the block that is a list partner of an own particle, plus every
// reactive partner of those that are reactive partners of an own particle --
// the own rows, and the reactive rows of that first halo shell (each the
// owner's row, in the owner's order), all with partners as 16-bit local
// indices.  A step then reads the halo's new snapshots once, forms S for the own
// particles and for the reactive halo from shared memory (a halo row is its
// owner's row, evaluated in the same order with the same operations, so both
// blocks hold bit-identical S), and the pair forces and the integrator with no
// further global gather.  Forces and trajectories are bit-identical to the
// two-barrier path (same per-entry operations, same summation orders); only
// the thermo partials are grouped differently.
//
// Steps follow one another by the data itself, without a grid barrier: a block
// publishes each own snapshot as one 16-byte store whose top bit tells the
// step (its parity over the writes of that buffer), and the blocks that hold
// the particle in their halo read it until the bit is the expected one.  What
// all blocks have to agree on, the displacement bound that asks for a list
// build, comes along late: one thread posts the block's largest displacement and
// its arrival once the block has read its halo, and waits for every block's while
// the others work on S and the forces; the step is thrown away before the integrator
// if the list turns out to have to be rebuilt first.
//
// The order of the accesses.  A snapshot is a relaxed 16-byte store and load of one
// size and place, and carries its own step.  A block posts publication k after it has
// read its halo of k, and writes publication k + 1 (into the buffer of k - 1) once it
// has seen all post k.  The arrival is a release add, after a block barrier that all
// the block's reads come before, and the wait ends with an acquire fence ahead of
// the block barrier that all its writes come after: every read of publication k - 1
// happens before the write over it, and the maximum is read after every block's part
// of it.  (Posted ahead of the halo, whose reads then ran beside it, the release waited
// for the block's own stores on their way out: 512 particles x 64 steps 386 us, 4,099 x
// 100 769, 100,000 x 100 logged 1,541; behind it 368, 721, 1,465; relaxed throughout and
// ahead of the halo, without the order above being promised, 380, 757, 1,500.  A slot
// per block that every block reads took three times as long as one counter: the
// readers crowd the lines that are being written.)
// With a grid barrier per step (arrival, poll, then the halo copies, nine block
// barriers in all) a step of 512 particles took 7.3 us (6.2 this way, 4.1 with
// the branch-free powers of pair_power), one of 100,000 14.8 (14.2, 12.4).

struct RStage {
    static constexpr int kL = 3072;    // local particles: own (at most blockDim), then halo
    static constexpr int kES = 16384;  // entries of the rows of S, warp-major (padded to each warp's longest)
    static constexpr int kEF = 12288;  // entries of the own rows (force pass), laid out the same way
    static constexpr int kHash = 4096; // open-addressing table of halo slots (while building)
    static constexpr int kRounds = (kL + kBlock - 1) / kBlock;  // rows of S per thread, at most
    static constexpr size_t O_LPOS = 0;                             // [kL] int4 snapshots (own, then halo)
    static constexpr size_t O_LS = O_LPOS + (size_t)kL * 16;        // [kL] float S
    static constexpr size_t O_HSLOT = O_LS + (size_t)kL * 4;        // [kL] int global slot of halo particle h
    static constexpr size_t O_SENT = O_HSLOT + (size_t)kL * 4;      // [kES] u16 local partners of the rows of S
    static constexpr size_t O_FENT = O_SENT + (size_t)kES * 2;      // [kEF] u16 local partners of the own rows
    static constexpr size_t O_SDESC = O_FENT + (size_t)kEF * 2;     // [kL] int2 row of S: (lane's first entry, centre | n << 16)
    static constexpr size_t O_FDESC = O_SDESC + (size_t)kL * 8;     // [kBlock] int4 by thread: (first entry of its
                                                                    // reactive row, of its other row, nr | nw << 16,
                                                                    // centre of each (16 bits each, 0xffff: none))
    static constexpr size_t O_FW = O_FDESC + (size_t)kBlock * 16;   // [3][kBlock] float other-row forces by centre
    // the own particles' state, by row position, kept here between list builds
    // (global memory is brought up to date by r_flush)
    static constexpr size_t O_VEL = O_FW + (size_t)kBlock * 12;     // [kBlock] float4 velocities
    static constexpr size_t O_XQ = O_VEL + (size_t)kBlock * 16;     // [3 kBlock] fixed-point positions
    static constexpr size_t O_IMG = O_XQ + (size_t)kBlock * 24;     // [3 kBlock] image counts
    static constexpr size_t kBytes = O_IMG + (size_t)kBlock * 12;
    // While building, the own-state area holds the hash table (keys, values),
    // the sorts' histograms and the warp-block lengths; O_SENT holds the reactive
    // first shell's table indices, O_FENT the force rows' per-warp counts, O_LS
    // the centres of the rows of S by position.
    static constexpr size_t B_KEY = O_VEL, B_VAL = B_KEY + (size_t)kHash * 4, B_HIST = B_VAL + (size_t)kHash * 4,
                            B_WL = B_HIST + 3 * 256 * 4, B_END = B_WL + ((size_t)(kRounds + 2) * 33) * 4;
    static_assert(B_END <= kBytes, "build scratch fits the own-state area");
    static_assert(kES <= 65536 && kEF <= 65536 && kL <= 65536, "16-bit local indices and offsets");
    static_assert(kBlock % 32 == 0 && kBlock / 32 <= 32, "whole warps, at most 32");
    static_assert(kBlock >= 768 && kEF >= kBlock / 32 * 512, "force-row sort scratch in O_FENT");
    static_assert(kHash > kL + kBlock, "the halo's table never fills up");
    static_assert(kES >= 2 * kHash, "the reactive first shell's table indices in O_SENT");

    static __device__ __forceinline__ int4* lpos() { return (int4*)(g_dyn + O_LPOS); }
    static __device__ __forceinline__ float* lS() { return (float*)(g_dyn + O_LS); }
    static __device__ __forceinline__ int* hslot() { return (int*)(g_dyn + O_HSLOT); }
    static __device__ __forceinline__ unsigned short* sent() { return (unsigned short*)(g_dyn + O_SENT); }
    static __device__ __forceinline__ unsigned short* fent() { return (unsigned short*)(g_dyn + O_FENT); }
    static __device__ __forceinline__ int2* sdesc() { return (int2*)(g_dyn + O_SDESC); }
    static __device__ __forceinline__ int4* fdesc() { return (int4*)(g_dyn + O_FDESC); }
    static __device__ __forceinline__ float* fw() { return (float*)(g_dyn + O_FW); }
    static __device__ __forceinline__ float4* vel() { return (float4*)(g_dyn + O_VEL); }
    static __device__ __forceinline__ long long* xq() { return (long long*)(g_dyn + O_XQ); }
    static __device__ __forceinline__ int* img() { return (int*)(g_dyn + O_IMG); }
};
static_assert(RStage::kBytes <= 227 * 1024 - 12 * 1024, "the resident layout fits beside the static shared memory");

__device__ __forceinline__ unsigned r_hash(int q) { return ((unsigned)q * 2654435761u) >> 20; }

static __shared__ int s_nh, s_nhr;  // halo particles, halo rows of S (while building)

// Inserts slot q into the table (if absent; a new one gets the next local index
// after the P own particles); its place, or -1 when there is no room.  val:
// bit 0 reactive partner of an own particle, then the rank in the halo.  Once the
// halo is too large nothing is inserted any more, so that the table, larger than the
// halo by more than the block's threads, never fills up: with every insertion going
// round a full table a build that failed took 8 ms (50,000 particles, r_cut 3.3: 30
// steps 21,100 us, now 1,440).
__device__ __forceinline__ int r_insert(int* key, int* val, int q, int P)
{
    if (*(volatile int*)&s_nh > RStage::kL - P) return -1;
    unsigned h = r_hash(q) & (RStage::kHash - 1);
    for (int probe = 0; probe < RStage::kHash; probe++) {
        const int old = atomicCAS(&key[h], -1, q);
        if (old == -1) {
            const int r = atomicAdd(&s_nh, 1);
            if (P + r >= RStage::kL) return -1;
            RStage::hslot()[r] = q;
            atomicOr(&val[h], r << 1);
        }
        if (old == -1 || old == q) return (int)h;
        h = (h + 1) & (RStage::kHash - 1);
    }
    return -1;
}

// Local index of global slot q: own particles first (q - b0), then the halo.
__device__ __forceinline__ int r_lid(const int* key, const int* val, int q, int b0, int b1, int P)
{
    if (q >= b0 && q < b1) return q - b0;
    unsigned h = r_hash(q) & (RStage::kHash - 1);
    for (int probe = 0; probe < RStage::kHash && key[h] != q; probe++) h = (h + 1) & (RStage::kHash - 1);
    return P + (val[h] >> 1);
}

// Four entries of a row as local indices (padding: the row's own particle, in
// the block or the halo like every partner).
__device__ __forceinline__ void r_put_four(const Dev<float>& d, const int* key, const int* val, int b0, int b1, int P,
                                           const int4& j, unsigned short* out, int n)
{
    const int q[4] = {j.x, j.y, j.z, j.w};
#pragma unroll
    for (int u = 0; u < 4; u++)
        if (u < n) out[32 * u] = (unsigned short)r_lid(key, val, q[u], b0, b1, P);
}

// 256 counts -> the first rank of every key, keys in descending order (one warp).
__device__ __forceinline__ void warp_desc_starts(int* hist)
{
    const int lane = threadIdx.x & 31;
    int c[8], sum = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        c[i] = hist[255 - 8 * lane - i];
        sum += c[i];
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    x -= sum;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        hist[255 - 8 * lane - i] = x;
        x += c[i];
    }
}

// Adds the lanes with a key (-1: none) to counts[key], one atomic per key and
// warp; the lane's place among them.
__device__ __forceinline__ int warp_count(int key, int* counts)
{
    const int lane = threadIdx.x & 31;
    const unsigned m = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (key >= 0 && lane == leader) base = atomicAdd(&counts[key], __popc(m));
    return __shfl_sync(0xffffffffu, base, leader) + __popc(m & ((1u << lane) - 1u));
}

// Lengths of n warp blocks (32 rows each) -> their first entries, in order; the
// total goes behind them (one warp).
__device__ __forceinline__ void warp_block_starts(int* wl, int n)
{
    const int lane = threadIdx.x & 31;
    int base = 0;
    for (int b = 0; b < n; b += 32) {
        const int L = b + lane < n ? 32 * wl[b + lane] : 0;
        int x = L;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (b + lane < n) wl[b + lane] = base + x - L;
        base += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) wl[n] = base;
}

// Builds the block's resident structures from the global list and the
// snapshots pos[pc].  Returns 1 when they fit (the same answer in every
// thread of the block); 0 leaves nothing the step relies on.  Halo particles
// and rows of S are numbered in the order in which threads find them: nothing
// that is summed depends on it.  (With block-wide scans and sorts for the
// numbering, one-thread layouts and one entry loaded at a time this took 26 us
// at 4 particles per block and 50 us at 660, in every launch and after every list
// build; now 11 and 28.)
static __device__ int r_localize(const Dev<float>& d, int pc, int ac)
{
    typedef RStage RS;
    constexpr int RR = RS::kRounds;
    int4* lpos = RS::lpos();
    int* key = (int*)(g_dyn + RS::B_KEY);
    int* val = (int*)(g_dyn + RS::B_VAL);
    int* hist = (int*)(g_dyn + RS::B_HIST);  // rows of S; reactive and other force rows
    int* wl = (int*)(g_dyn + RS::B_WL);      // warp blocks of the rows of S; of the two kinds of force rows
    int *wlr = wl + RR * 32 + 1, *wlo = wlr + 33;
    int* hr = (int*)RS::sent();   // table place of the k-th reactive first-shell particle
    int* cen = (int*)RS::lS();    // centre (local index) of the row at each position
    const int t = threadIdx.x, B = blockDim.x, lane = t & 31, warp = t >> 5, nw = B >> 5;
    int b0, b1;
    block_range(d, b0, b1);
    const int P = b1 - b0;
    if (B != kBlock || P > B) return 0;
    for (int h = t; h < RS::kHash; h += B) {
        key[h] = -1;
        val[h] = 0;
    }
    if (t == 0) s_nh = s_nhr = 0;
    int4 inf = make_int4(0, 0, 0, 0);
    if (t < P) inf = d.pinfo[b0 + t];
    __syncthreads();
    int fail = inf.y > 255 || inf.w > 255;
    // 1. first shell: the partners of the own rows outside the block (lanes that
    // the particles leave share a row, four entries at a time)
    {
        int lg = 0;
        while (lg < 5 && (P << (lg + 1)) <= B) lg++;
        const int i = t >> lg, g = t & ((1 << lg) - 1);
        if (i < P) {
            const int4 f = d.pinfo[b0 + i];
            const int cr = (f.y + 3) >> 2, cw = (f.w + 3) >> 2;
            for (int c = g; c < cr + cw; c += 1 << lg) {
                const bool react = c < cr;
                const int4 j = load_four(d, react ? f.x : f.z, 4 * (react ? c : c - cr));
                const int q[4] = {j.x, j.y, j.z, j.w};
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    if (q[u] >= b0 && q[u] < b1) continue;  // padding is the own slot
                    const int h = r_insert(key, val, q[u], P);
                    if (h < 0) fail = 1;
                    else if (react && !(atomicOr(&val[h], 1) & 1)) hr[atomicAdd(&s_nhr, 1)] = h;
                }
            }
        }
    }
    if (__syncthreads_or(fail)) return 0;
    // 2. second shell: the reactive partners of the reactive first shell (whose S
    // is formed here too)
    const int Hr = s_nhr;
    {
        int lg = 0;
        while (lg < 3 && (Hr << (lg + 1)) <= B) lg++;
        for (int k = t >> lg; k < Hr; k += B >> lg) {
            const int4 f = d.pinfo[key[hr[k]]];
            for (int c = t & ((1 << lg) - 1); c < (f.y + 3) >> 2; c += 1 << lg) {
                const int4 j = load_four(d, f.x, 4 * c);
                const int q[4] = {j.x, j.y, j.z, j.w};
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if ((q[u] < b0 || q[u] >= b1) && r_insert(key, val, q[u], P) < 0) fail = 1;
            }
        }
    }
    // 3. rows of S (the own rows and the reactive first shell's), longest
    // first, dealt out over the RB row threads as a snake: rank s goes to round
    // s / RB, to thread s % RB in even rounds and RB - 1 - s % RB in odd ones, so
    // that a thread's second row is short when its first is long.  The force
    // pass runs two loops per thread, over a reactive row and over another
    // particle's other (purely two-body) row: reactive rows longest first
    // from warp 0, other rows longest first from the last warp, so that the
    // rows of a warp are alike in each loop and the warps' totals even out.
    const int NS = P + Hr;
    if (NS > RS::kL) return 0;  // the same in every thread
    // the rows leave the last warp free for the agreement (r_run) where they can
    const int RB = P <= B - 32 && NS <= RR * (B - 32) ? B - 32 : B;
    const int rounds = (NS + RB - 1) / RB, W32 = (P + 31) & ~31;
    int skey[RR + 1], hrow[RR];
    skey[0] = t < P ? min(inf.y, 255) : -1;
#pragma unroll
    for (int r = 0; r < RR; r++) {
        const int k = t + r * B;
        skey[r + 1] = -1;
        hrow[r] = 0;
        if (k < Hr) {
            const int4 f = d.pinfo[key[hr[k]]];
            hrow[r] = f.x;
            if (f.y > 255) fail = 1;
            skey[r + 1] = min(f.y, 255);
        }
    }
    // force rows are ranked in particle order among equal lengths (their threads
    // sum the thermo terms): counts per warp and key, reactive then other
    unsigned short* wh = RS::fent();
    for (int k = t; k < nw * 256; k += B) ((int*)wh)[k] = 0;
    for (int k = t; k < 3 * 256; k += B) hist[k] = 0;
    for (int q = t; q < rounds * RB; q += B) RS::sdesc()[q] = make_int2(0, -1);  // no row here
    if (t < W32) RS::fdesc()[t] = make_int4(0, 0, 0, -1);                        // no rows; centres 0xffff
    if (__syncthreads_or(fail)) return 0;
    const int H = s_nh;
    const int krow = t < P ? inf.y : -1, kother = t < P ? inf.w : -1;
    const unsigned mr = __match_any_sync(0xffffffffu, krow), mo = __match_any_sync(0xffffffffu, kother);
    const int br = __popc(mr & ((1u << lane) - 1u)), bo = __popc(mo & ((1u << lane) - 1u));
    if (t < P && br == 0) wh[warp * 512 + krow] = (unsigned short)__popc(mr);
    if (t < P && bo == 0) wh[warp * 512 + 256 + kother] = (unsigned short)__popc(mo);
#pragma unroll
    for (int r = 0; r <= RR; r++)
        if (r == 0 || (r - 1) * B < Hr) warp_count(skey[r], hist);
    __syncthreads();
    if (t >= 256) {
        // per key: the counts of the warps before each warp, and the key's total
        const int k = t - 256;  // 512 threads: the two kinds
        int run = 0;
        for (int w = 0; w < nw; w++) {
            const int c = wh[w * 512 + k];
            wh[w * 512 + k] = (unsigned short)run;
            run += c;
        }
        hist[t] = run;
    } else if (warp == 0) {
        warp_desc_starts(hist);
    }
    __syncthreads();
    if (warp < 2) warp_desc_starts(hist + 256 * (warp + 1));
    __syncthreads();
    // what each position needs: the centre and the row (start, count)
#pragma unroll
    for (int r = 0; r <= RR; r++) {
        if (r > 0 && (r - 1) * B >= Hr) continue;
        const int sr = warp_count(skey[r], hist);
        if (skey[r] < 0) continue;
        const int g = sr / RB, slot = sr - g * RB;
        const int q = g * RB + ((g & 1) ? RB - 1 - slot : slot);
        if (r == 0) {
            cen[q] = t;
            RS::sdesc()[q] = make_int2(inf.x, inf.y);
        } else {
            cen[q] = P + (val[hr[t + (r - 1) * B]] >> 1);
            RS::sdesc()[q] = make_int2(hrow[r - 1], skey[r]);
        }
    }
    if (t < P) {
        const int rpos = hist[256 + krow] + wh[warp * 512 + krow] + br;
        const int wrank = hist[512 + kother] + wh[warp * 512 + 256 + kother] + bo;
        const int wpos = W32 - 32 - (wrank & ~31) + (wrank & 31);  // rank chunk c -> warp W32/32 - 1 - c
        // 16-bit fields: (z, w) = (nr, nw, reactive centre, other centre)
        int4* fr = &RS::fdesc()[rpos];
        int4* fo = &RS::fdesc()[wpos];
        fr->x = inf.x;
        fo->y = inf.z;
        ((unsigned short*)&fr->z)[0] = (unsigned short)inf.y;
        ((unsigned short*)&fo->z)[1] = (unsigned short)inf.w;
        ((unsigned short*)&fr->w)[0] = (unsigned short)t;
        ((unsigned short*)&fo->w)[1] = (unsigned short)t;
    }
    __syncthreads();
    // 4. warp-major layouts: every warp block of 32 rows takes 32 x its longest
    // row; the rows of S in order (round, warp); the own rows' reactive parts,
    // then their other parts
    int2 src[RR];
#pragma unroll
    for (int r = 0; r < RR; r++) {
        src[r] = r < rounds && t < RB ? RS::sdesc()[t + r * RB] : make_int2(0, -1);
        const int L = __reduce_max_sync(0xffffffffu, max(src[r].y, 0));
        if (lane == 0) wl[r * nw + warp] = L;
    }
    const int4 fd = t < W32 ? RS::fdesc()[t] : make_int4(0, 0, 0, -1);
    const int nrc = fd.z & 0xffff, nwc = (int)((unsigned)fd.z >> 16);
    const int Lr = __reduce_max_sync(0xffffffffu, nrc), Lo = __reduce_max_sync(0xffffffffu, nwc);
    if (lane == 0) {
        wlr[warp] = Lr;
        wlo[warp] = Lo;
    }
    __syncthreads();
    if (warp == 0) warp_block_starts(wl, RR * nw);
    else if (warp < 3) warp_block_starts(warp == 1 ? wlr : wlo, nw);
    __syncthreads();
    const int ER = wlr[nw];
    if (wl[RR * nw] > RS::kES || ER + wlo[nw] > RS::kEF) return 0;  // the same in every thread
    // 5. the rows, partners as local indices
#pragma unroll
    for (int r = 0; r < RR; r++) {
        if (r >= rounds || src[r].y < 0) continue;
        const int q = t + r * RB, first = wl[r * nw + warp] + lane, n = src[r].y;
        for (int m = 0; m < n; m += 4)
            r_put_four(d, key, val, b0, b1, P, load_four(d, src[r].x, m), RS::sent() + first + 32 * m, n - m);
        RS::sdesc()[q] = make_int2(first, cen[q] | (n << 16));
    }
    if (t < W32) {
        const int first_r = wlr[warp] + lane, first_o = ER + wlo[warp] + lane;
        for (int m = 0; m < nrc; m += 4)
            r_put_four(d, key, val, b0, b1, P, load_four(d, fd.x, m), RS::fent() + first_r + 32 * m, nrc - m);
        for (int m = 0; m < nwc; m += 4)
            r_put_four(d, key, val, b0, b1, P, load_four(d, fd.y, m), RS::fent() + first_o + 32 * m, nwc - m);
        RS::fdesc()[t] = make_int4(first_r, first_o, fd.z, fd.w);
    }
    if (t < P) {
        const int4 own = d.pos[pc][b0 + t];
        lpos[t] = own;               // own snapshots by local index
        d.pos[pc ^ 1][b0 + t] = own; // top bit clear: the first publication into this buffer sets it
    }
    if (t == 0) {
        s_ls.r_rb = RB;
        s_ls.r_np = P;
        s_ls.r_nh = H;
        s_ls.r_nhr = Hr;
    }
    __syncthreads();
    // 6. the own particles' state by reactive-row position (over the table, now unused)
    if (t < P) {
        const int i = b0 + (fd.w & 0xffff), n = d.n;
        RS::vel()[t] = d.vel[ac][i];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            RS::xq()[3 * t + c] = d.xq[ac][c * n + i];
            RS::img()[3 * t + c] = d.img[ac][c * n + i];
        }
    }
    __syncthreads();
    return 1;
}

// Writes the own particles' state back to the global arrays (snapshots to set
// pc, without the step's bit; the rest to set ac): before a list build reorders
// them, and when the run ends.  Every block has read its halo of pos[pc].
__device__ __forceinline__ void r_flush(const Dev<float>& d, int pc, int ac)
{
    typedef RStage RS;
    const int t = threadIdx.x, n = d.n;
    if (t < s_ls.r_np) {
        int b0, b1;
        block_range(d, b0, b1);
        const int lid = RS::fdesc()[t].w & 0xffff, i = b0 + lid;
        d.pos[pc][i] = RS::lpos()[lid];
        d.vel[ac][i] = RS::vel()[t];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            d.xq[ac][c * n + i] = RS::xq()[3 * t + c];
            d.img[ac][c * n + i] = RS::img()[3 * t + c];
        }
    }
}

// A snapshot as one 16-byte access (single-copy atomic: a reader sees a whole
// one), through L2.
__device__ __forceinline__ int4 ld_snapshot(const int4* p)
{
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 v;\n\tld.relaxed.gpu.global.b128 v, [%2];\n\tmov.b128 {%0, %1}, v;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_int4((int)lo, (int)(lo >> 32), (int)hi, (int)(hi >> 32));
}

__device__ __forceinline__ void st_snapshot(int4* p, const int4& v)
{
    const unsigned long long lo = (unsigned)v.x | (unsigned long long)(unsigned)v.y << 32;
    const unsigned long long hi = (unsigned)v.z | (unsigned long long)(unsigned)v.w << 32;
    asm volatile("{\n\t.reg .b128 v;\n\tmov.b128 v, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], v;\n\t}" ::"l"(p), "l"(lo),
                 "l"(hi)
                 : "memory");
}

// One turn of a bounded wait: false once the time is up (or another wait's is).
struct Patience {
    int spins = 0;
    long long t0 = 0;
    __device__ __forceinline__ bool more(Ctl* ctl, long long timeout_ns, int where)
    {
        if (++spins < 64) return true;
        if (spins == 64) t0 = gtimer_ns();
        if (ld_relaxed(&ctl->status) & kStatusTimeout) return false;
        if (gtimer_ns() - t0 > timeout_ns) {
            atomicOr(&ctl->status, kStatusTimeout);
            ctl->timeout_at = where;
            return false;
        }
        return true;
    }
};

// The top bit of publication k = 1, 2, ... since the resident structures were
// built (two buffers in turn, both clear before).
__device__ __forceinline__ unsigned r_bit(int k) { return ((unsigned)(((k - 1) >> 1) & 1) ^ 1u) << 31; }

// Post and agreement of publication e = 1, 2, ... of a launch (one thread of the
// block).  The words of e's parity: arrivals, and (publication, largest squared
// displacement); both only grow, so neither is ever reset.
__device__ __forceinline__ void r_post(const Dev<float>& d, unsigned e)
{
    unsigned long long* w = d.agree + 2 * (e & 1);
    const unsigned long long mine = (unsigned long long)e << 32 | s_ls.dmax_bits;
    s_ls.dmax_bits = 0u;
    asm volatile("red.relaxed.gpu.global.max.u64 [%0], %1;" ::"l"(w + 1), "l"(mine) : "memory");
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(w), "l"(1ull) : "memory");
}

__device__ __forceinline__ void r_agree(const Dev<float>& d, const RunArgs& a, unsigned e)
{
    const unsigned long long* w = d.agree + 2 * (e & 1);
    const unsigned long long want = (unsigned long long)((e + 1) / 2) * (unsigned)g_size();
    Patience wait;
    for (;;) {
        unsigned long long n, m;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(n) : "l"(w) : "memory");
        if (n >= want) {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(m) : "l"(w + 1) : "memory");
            s_ls.disp += sqrtf(__uint_as_float((unsigned)m));
            return;
        }
        if (!wait.more(d.ctl, a.timeout_ns, 22)) {
            s_ls.ok = 0;
            return;
        }
    }
}

// S of one row (entries e[0], e[32], ...) with the two-barrier path's order of
// additions (groups of four, then one by one).
template <bool UNI, int X>
__device__ __forceinline__ float r_row_s(const Dev<float>& d, const PairP<float>* tab, const PairP<float>& ps,
                                         const int4* lpos, const unsigned short* e, int cnt, const int4& pi)
{
    float s = 0.0f;
    int k = 0;
    for (; k + 4 <= cnt; k += 4) {
        const float w0 = s_term<float, UNI, X>(d, tab, ps, pi, lpos[e[32 * k]]);
        const float w1 = s_term<float, UNI, X>(d, tab, ps, pi, lpos[e[32 * (k + 1)]]);
        const float w2 = s_term<float, UNI, X>(d, tab, ps, pi, lpos[e[32 * (k + 2)]]);
        const float w3 = s_term<float, UNI, X>(d, tab, ps, pi, lpos[e[32 * (k + 3)]]);
        s += (w0 + w1) + (w2 + w3);
    }
    for (; k < cnt; k++) s += s_term<float, UNI, X>(d, tab, ps, pi, lpos[e[32 * k]]);
    return s;
}

// The pair forces of a thread's rows: the other (purely two-body) row of one
// particle, whose sum goes to fw, and the reactive row of particle lid into f.
// TH (the sampled step): the pair terms are left summed per warp in s_wpart
// (so that the accumulators are not live through the integrator).
template <bool UNI, int X, bool TH>
__device__ __forceinline__ void r_forces(const Dev<float>& d, const RunArgs& a, int P, const int4& fd, float& fx,
                                         float& fy, float& fz)
{
    typedef RStage RS;
    const int t = threadIdx.x;
    const PairP<float>* tab = stab<float>();
    const PairP<float>& ps = a.uf[0];
    const PairP<float>& pw = a.uf[1];
    const int4* lpos = RS::lpos();
    const float* lS = RS::lS();
    float* fw = RS::fw();
    Acc<float> acc;
    if (TH)
#pragma unroll
        for (int q = 0; q < kNQA; q++) acc.q[q] = 0.0f;
    if (t < ((P + 31) & ~31)) {
        const int nr = fd.z & 0xffff, nw = (int)((unsigned)fd.z >> 16);
        const int cw = (int)((unsigned)fd.w >> 16);
        if (cw != 0xffff) {
            const unsigned short* ew = RS::fent() + fd.y;
            const int4 pc_ = lpos[cw];
            float gx = 0.0f, gy = 0.0f, gz = 0.0f;
#pragma unroll 2
            for (int k = 0; k < nw; k++) {
                const int j = ew[32 * k];
                float ex, ey, ez;
                entry_force<float, UNI, X, false, TH>(d, tab, pc_, lpos[j], 0.0f, 0.0f, pw, acc, ex, ey, ez);
                gx = __fadd_rn(gx, ex);
                gy = __fadd_rn(gy, ey);
                gz = __fadd_rn(gz, ez);
            }
            fw[cw] = gx;
            fw[kBlock + cw] = gy;
            fw[2 * kBlock + cw] = gz;
        }
        if (t < P) {
            const int lid = fd.w & 0xffff;
            const unsigned short* er = RS::fent() + fd.x;
            const int4 pi = lpos[lid];
            const float Si = lS[lid];
#pragma unroll 2
            for (int k = 0; k < nr; k++) {
                const int j = er[32 * k];
                float ex, ey, ez;
                entry_force<float, UNI, X, true, TH>(d, tab, pi, lpos[j], Si, lS[j], ps, acc, ex, ey, ez);
                fx = __fadd_rn(fx, ex);
                fy = __fadd_rn(fy, ey);
                fz = __fadd_rn(fz, ez);
            }
        }
    }
    if (TH) {
        if ((t & ~31) < P) {  // the warp holds rows (the same in all its lanes)
#pragma unroll
            for (int q = 0; q < kNQA; q++)
                if (q != Q_K) warp_part(acc.q[q] * th_scale(q), q);
        } else if ((t & 31) == 0) {
#pragma unroll
            for (int q = 0; q < kNQA; q++)
                if (q != Q_K) s_wpart[q][t >> 5] = 0.0f;
        }
    }
}

// Resident steps until the run's last one is done (1), the list has to be
// rebuilt before the next (2) or a wait ran out (0).  The loop's state is the
// same in every thread.
template <bool UNI, int X>
static __device__ int r_run(const Dev<float>& d, const RunArgs& a)
{
    typedef RStage RS;
    const int t = threadIdx.x, B = blockDim.x;
    const int P = s_ls.r_np, H = s_ls.r_nh, RB = s_ls.r_rb;
    const int NQ = (P + s_ls.r_nhr + RB - 1) / RB * RB;  // positions of the rows of S
    const bool spare = RB < B;                           // the last warp has no rows
    int b0, b1;
    block_range(d, b0, b1);
    int pc = s_ls.pc, remaining = s_ls.remaining, k = 0;
    long long step = s_ls.step;
    unsigned epoch = s_ls.r_epoch;
    int tl_left = s_ls.tlog_left, tl_slot = s_ls.tlog_slot, tl_n = 0;
    const float skin_eff = (float)a.skin_eff;
    int4* lpos = RS::lpos();
    float* lS = RS::lS();
    const int* hslot = RS::hslot();
    double* lg = nullptr;  // record of the previous step, its warps' sums not yet added up
    int result = 0;
    for (;;) {
        const bool more = remaining > 1, logged = tl_left == 1, th = !more || logged;
        // the halo's snapshots (complete at the first step)
        const int4* pos = d.pos[pc];
        const unsigned bit = r_bit(k), care = k > 0 ? 0x80000000u : 0u;
        int4 v0 = make_int4(0, 0, 0, 0), v1 = v0;
        bool w0 = t < RB && t < H, w1 = t < RB && t + RB < H;
        if (w0) v0 = ld_snapshot(&pos[hslot[t]]);
        if (w1) v1 = ld_snapshot(&pos[hslot[t + RB]]);
        if (lg) {
            __syncthreads();
            warp_sums_to(lg, nullptr);
            lg = nullptr;
        }
        int ok = 1;
        for (int h = t; w0; h += 2 * RB) {
            Patience wait;
            for (;;) {
                if (w0 && (((unsigned)v0.w ^ bit) & care) == 0) {
                    v0.w &= 0x7fffffff;
                    lpos[P + h] = v0;
                    w0 = false;
                }
                if (w1 && (((unsigned)v1.w ^ bit) & care) == 0) {
                    v1.w &= 0x7fffffff;
                    lpos[P + h + RB] = v1;
                    w1 = false;
                }
                if (!w0 && !w1) break;
                if (!wait.more(d.ctl, a.timeout_ns, 23)) {
                    ok = 0;
                    break;
                }
                if (w0) v0 = ld_snapshot(&pos[hslot[h]]);
                if (w1) v1 = ld_snapshot(&pos[hslot[h + RB]]);
            }
            w0 = ok && h + 2 * RB < H;
            w1 = ok && h + 3 * RB < H;
            if (w0) v0 = ld_snapshot(&pos[hslot[h + 2 * RB]]);
            if (w1) v1 = ld_snapshot(&pos[hslot[h + 3 * RB]]);
        }
        if (!__syncthreads_and(ok)) break;
        if (k > 0 && t == B - 32) {
            r_post(d, epoch);
            if (spare) r_agree(d, a, epoch);
        }
        int4 fd = make_int4(0, 0, 0, -1);
        float fx = 0.0f, fy = 0.0f, fz = 0.0f;
        if (t < RB) {
            const PairP<float>* tab = stab<float>();
            for (int q = t; q < NQ; q += RB) {
                const int2 dsc = RS::sdesc()[q];
                if (dsc.y < 0) continue;  // no row at this position
                const int lid = dsc.y & 0xffff;
                lS[lid] = r_row_s<UNI, X>(d, tab, a.uf[0], lpos, RS::sent() + dsc.x, (int)((unsigned)dsc.y >> 16), lpos[lid]);
            }
            asm volatile("bar.sync 1, %0;" ::"r"(RB) : "memory");  // the row threads (whole warps)
            if (t < ((P + 31) & ~31)) fd = RS::fdesc()[t];
        }
        if (th) r_forces<UNI, X, true>(d, a, P, fd, fx, fy, fz);
        else if (t < RB) r_forces<UNI, X, false>(d, a, P, fd, fx, fy, fz);
        if (!spare && k > 0 && t == B - 32) r_agree(d, a, epoch);
        // the noise of the next step's start, while the agreement is on its way
        float z[3] = {0.0f, 0.0f, 0.0f};
        const int lid = fd.w & 0xffff;
        int4 pi = make_int4(0, 0, 0, 0);
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
        long long q[3] = {0, 0, 0};
        if (t < P) {
            pi = lpos[lid];
            v = RS::vel()[t];
#pragma unroll
            for (int c = 0; c < 3; c++) q[c] = RS::xq()[3 * t + c];
            if (more && a.langevin) normals3(a.seed, step + 1, (unsigned)(pi.w >> kTypeBits), z);
        }
        __syncthreads();  // every row has read the old snapshots, fw is complete, the displacement bound is known
        if (k > 0) {
            if (!s_ls.ok) break;
            if (2.0f * s_ls.disp > skin_eff) {
                result = 2;
                break;
            }
        }
        float kin = 0.0f, dmax = 0.0f;
        if (t < P) {
            const float* fw = RS::fw();
            const int i = b0 + lid;
            // the force: the reactive row's sum plus the other row's
            fx = __fadd_rn(fx, fw[lid]);
            fy = __fadd_rn(fy, fw[kBlock + lid]);
            fz = __fadd_rn(fz, fw[2 * kBlock + lid]);
            if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) atomicOr(&d.ctl->status, kStatusNonfinite);
            if (!more) d.force[i] = make_float4(fx, fy, fz, 0.0f);
            int w[3];
            int4 np = make_int4(0, 0, 0, 0);
            dmax = advance_particle(d, a, fx, fy, fz, F_CLOSING | (more ? F_OPENING : 0), z, pi.w, v, q, w, kin, np);
            if (more) {
                int4 pub = np;
                pub.w |= (int)r_bit(k + 1);
                st_snapshot(&d.pos[pc ^ 1][i], pub);
                lpos[lid] = np;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    RS::xq()[3 * t + c] = q[c];
                    if (w[c]) RS::img()[3 * t + c] += w[c];
                }
            }
            RS::vel()[t] = v;
        }
        if (th) {
            if ((t & ~31) < P)
                warp_part(kin, Q_K);
            else if ((t & 31) == 0)
                s_wpart[Q_K][t >> 5] = 0.0f;
        }
        step++;
        remaining--;
        if (tl_left > 0) tl_left = logged ? a.tlog_every : tl_left - 1;
        if (logged) {
            lg = d.tlog + ((size_t)tl_slot * a.max_blocks + g_rank()) * kNQ;
            if (t == 0 && g_rank() == 0) {
                d.tlog_step[2 * tl_slot] = step;
                d.tlog_step[2 * tl_slot + 1] = g_size();
            }
            tl_n++;
            tl_slot = tl_slot + 1 == d.tlog_cap ? 0 : tl_slot + 1;
        }
        if (!more) {
            thermo_partials(d, true, true, lg);
            result = 1;
            break;
        }
        if (t < RB) warp_max_disp(dmax);
        k++;
        epoch++;
        pc ^= 1;
    }
    __syncthreads();
    if (t == 0) {
        const int done = s_ls.remaining - remaining;
        s_ls.step = step;
        s_ls.remaining = remaining;
        s_ls.done += done;
        s_ls.r_steps += done;
        s_ls.pc = pc;
        s_ls.r_epoch = epoch;
        s_ls.tlog_left = tl_left;
        s_ls.tlog_slot = tl_slot;
        s_ls.tlog_k += tl_n;
        s_ls.own_ok = 0;
    }
    __syncthreads();
    return result;
}

// Builds every block's resident structures and agrees on the mode: the step
// runs resident only if every block's structures fit.
static __device__ bool r_enter(const Dev<float>& d, const RunArgs& a)
{
    const int ok = r_localize(d, s_ls.pc, s_ls.ac);
    const int round = s_ls.r_round;
    if (threadIdx.x == 0 && !ok) atomicOr(&d.ctl->rfail[round & 1], 1);
    if (!grid_barrier(d.ctl, a.timeout_ns, 8)) return false;
    if (threadIdx.x == 0) {
        s_ls.r_valid = ld_relaxed(&d.ctl->rfail[round & 1]) == 0;
        s_ls.r_try = 0;  // tried again after the next list build
        s_ls.r_round = round + 1;
        s_ls.own_ok = 0;  // the build overwrote the two-barrier path's staging
        // the next round's word: every block reads this round's word before it
        // arrives at the next barrier, and the next round comes after it
        if (g_rank() == 0) d.ctl->rfail[(round + 1) & 1] = 0;
    }
    __syncthreads();
    return true;
}

#endif  // SWP_HAS_RESIDENT

// One system advanced by the group of blocks this block belongs to (g_rank /
// g_size set by the caller).  Returns false when a wait timed out (the status
// word says so).
template <typename Real, bool UNI, bool BONDS>
__device__ __forceinline__ bool run_system(const Dev<Real>& d, const RunArgs& a)
{
    // the resident mode exists for one FP32 system without bonds
    constexpr bool kRes = SWP_HAS_RESIDENT && sizeof(Real) == 4 && !BONDS;
    Ctl* ctl = d.ctl;
    PairP<Real>* tab = (PairP<Real>*)s_tab_raw;
    const int ntt = d.ntypes * d.ntypes;
    for (int t = threadIdx.x; t < ntt; t += blockDim.x) tab[t] = d.table[t];
    if (threadIdx.x == 0) {
        s_withhold = a.withhold && g_rank() == 0;
        s_ls.bar_target = 0;
        s_ls.step = ctl->step;
        s_ls.rebuilds = 0;
        s_ls.state = ctl->state;
        s_ls.pc = ctl->pos_cur;
        s_ls.ac = ctl->arr_cur;
        // the list's block partition depends on the grid: rebuild if it changed
        s_ls.need_rb = ctl->need_rebuild | a.force_rebuild | (ctl->list_grid != g_size()) |
                       (ctl->list_chunk != (int)blockDim.x);
        s_ls.remaining = a.nsteps;
        s_ls.done = 0;
        s_ls.have_thermo = 0;
        s_ls.rc = 0;
        s_ls.disp = (float)ctl->disp;
        s_ls.dmax_bits = 0u;
        s_ls.own_ok = 0;
        s_ls.r_try = (kRes && a.resident && single_chunk(d)) ? 1 : 0;
        s_ls.r_valid = 0;
        s_ls.r_rb = 0;
        s_ls.r_epoch = 0;
        s_ls.ok = 1;
        s_ls.r_round = 0;
        s_ls.r_np = s_ls.r_nh = s_ls.r_nhr = 0;
        s_ls.r_steps = 0;
        s_ls.tlog_left = 0;
        s_ls.tlog_slot = 0;
        s_ls.tlog_k = 0;
        if (a.tlog_every > 0 && d.tlog) {
            s_ls.tlog_left = a.tlog_every - (int)(s_ls.step % a.tlog_every);
            s_ls.tlog_slot = (int)(ctl->tlog_n % d.tlog_cap);
        }
        // both agreement words start clear: every round comes after a barrier
        if (kRes && g_rank() == 0) {
            ctl->rfail[0] = 0;
            ctl->rfail[1] = 0;
        }
    }
    __syncthreads();
    const float skin_eff = (float)a.skin_eff;

    if (a.build_only) {
        const int rc = run_rebuild(d, a);
        if (rc == 2) return false;
        if (threadIdx.x == 0) {
            s_ls.need_rb = rc;
            s_ls.rc = rc;
        }
        __syncthreads();
    } else {
        if (s_ls.state == 1) {
            if (s_ls.need_rb || 2.0f * s_ls.disp > skin_eff) {
                const int rc = run_rebuild(d, a);
                if (rc == 2) return false;
                if (threadIdx.x == 0) {
                    s_ls.need_rb = rc;
                    s_ls.rc = rc;
                }
                __syncthreads();
            }
            if (s_ls.rc == 0) {
                run_s_pass<Real, UNI>(d, a, true);
                if (!grid_barrier(ctl, a.timeout_ns, 10)) return false;
                if (threadIdx.x == 0) s_ls.own_ok = single_chunk(d);
                run_f_pass<Real, UNI, BONDS, true>(d, a, F_STORE, s_ls.step);
                if (threadIdx.x == 0) s_ls.state = 0;  // read again only after the barrier
                thermo_partials(d, false, true, (double*)nullptr);
                if (!grid_barrier(ctl, a.timeout_ns, 11)) return false;
            }
        }
        if (s_ls.rc == 0 && s_ls.remaining > 0 && s_ls.state == 0) {
            const long long stp = s_ls.step;
            if (threadIdx.x == 0 && g_rank() == 0) ctl->dmax2[stp & 1] = 0u;
            if (!grid_barrier(ctl, a.timeout_ns, 12)) return false;
            run_open_pass(d, a, stp);
            __syncthreads();
            if (threadIdx.x == 0) {
                s_ls.pc ^= 1;
                s_ls.state = 2;
                s_ls.own_ok = 0;  // new positions in global memory only
            }
            if (!grid_barrier(ctl, a.timeout_ns, 13, &ctl->dmax2[stp & 1])) return false;
            add_disp(ctl, stp);
        }
        while (s_ls.rc == 0 && s_ls.state == 2) {
            const long long stp = s_ls.step;
            if (s_ls.need_rb || 2.0f * s_ls.disp > skin_eff) {
#if SWP_HAS_RESIDENT
                if constexpr (kRes)
                    if (s_ls.r_valid) {
                        // every block has read its halo; then the global state is
                        // brought up to date for the build to reorder
                        if (!grid_barrier(ctl, a.timeout_ns, 24)) return false;
                        r_flush(d, s_ls.pc, s_ls.ac);
                    }
#endif
                const int rc = run_rebuild(d, a);
                if (rc == 2) return false;
                if (threadIdx.x == 0) {
                    s_ls.need_rb = rc;
                    s_ls.rc = rc;
                    s_ls.r_valid = 0;
                    s_ls.r_try = (kRes && a.resident && single_chunk(d)) ? 1 : 0;
                }
                __syncthreads();
                if (rc) break;
            }
#if SWP_HAS_RESIDENT
            if constexpr (kRes) {
                if (s_ls.r_try)
                    if (!r_enter(d, a)) return false;
                if (s_ls.r_valid) {
                    int rc = 0;
                    expo_switch<UNI>(a, [&](auto x) { rc = r_run<UNI, decltype(x)::value>(d, a); });
                    if (rc == 0) return false;
                    if (rc == 1) {  // the last step is done: its partials are complete after the barrier
                        if (!grid_barrier(ctl, a.timeout_ns, 21)) return false;
                        if (threadIdx.x == 0) s_ls.state = 0;
                        __syncthreads();
                    }
                    continue;
                }
            }
#endif
            const bool more = s_ls.remaining > 1;
            // the thermo terms are summed on the launch's last step (the one a
            // launch reports) and on the logged steps only
            const bool logged = s_ls.tlog_left == 1;
            const bool th = !more || logged;
            const int flags = F_CLOSING | (more ? F_OPENING : F_STORE);
            if (threadIdx.x == 0 && g_rank() == 0) ctl->dmax2[(stp + 1) & 1] = 0u;
            run_s_pass<Real, UNI>(d, a, th);
            if (!grid_barrier(ctl, a.timeout_ns, 20)) return false;
            if (threadIdx.x == 0) s_ls.own_ok = single_chunk(d);
            if (th)
                run_f_pass<Real, UNI, BONDS, true>(d, a, flags, stp + 1);
            else
                run_f_pass<Real, UNI, BONDS, false>(d, a, flags, stp + 1);
            if (threadIdx.x == 0) {  // every thread read these before the passes' barrier
                s_ls.step = stp + 1;
                s_ls.remaining--;
                s_ls.done++;
                if (s_ls.tlog_left > 0) s_ls.tlog_left = logged ? a.tlog_every : s_ls.tlog_left - 1;
            }
            double* lg = logged ? d.tlog + ((size_t)s_ls.tlog_slot * a.max_blocks + g_rank()) * kNQ : nullptr;
            if (logged && threadIdx.x == 0 && g_rank() == 0) {
                d.tlog_step[2 * s_ls.tlog_slot] = stp + 1;
                d.tlog_step[2 * s_ls.tlog_slot + 1] = g_size();
            }
            // a logged step that is not the launch's last adds its terms up while
            // it waits (the record is read after the launch); the last step writes
            // the partials that the launch reduces before its arrival
            const bool late = th && more;
            if (th && !late) thermo_partials(d, false, true, lg);
            BarState bs;
            bs.target = s_ls.bar_target;
            bar_arrive(ctl, bs, more ? &ctl->dmax2[(stp + 1) & 1] : nullptr, &s_ls.dmax_bits);
            if (late) thermo_partials(d, false, false, lg);
            if (threadIdx.x == 0) s_ls.bar_target = bs.target;
            if (!bar_wait(ctl, bs, a.timeout_ns, 21, &s_ls.ok)) return false;
            if (logged && threadIdx.x == 0) {  // every thread used the slot before the barrier
                s_ls.tlog_k++;
                s_ls.tlog_slot = s_ls.tlog_slot + 1 == d.tlog_cap ? 0 : s_ls.tlog_slot + 1;
            }
            if (more) {
                if (threadIdx.x == 0) s_ls.pc ^= 1;
                add_disp(ctl, stp + 1);
            } else {
                if (threadIdx.x == 0) s_ls.state = 0;
                __syncthreads();
            }
        }
    }
    cp_async_wait_all();  // copies issued for a step that did not come
#if SWP_HAS_RESIDENT
    if constexpr (kRes)
        if (s_ls.r_valid) r_flush(d, s_ls.pc, s_ls.ac);
#endif
    if (s_ls.have_thermo) {
        // the partials were written before the arrival at the barrier that
        // followed their pass, which every block has passed
        if (kBatched && g_size() < kNQA)
            reduce_small(d);
        else
            run_reduce_thermo(d);
    }
    if (g_rank() == 0 && threadIdx.x == 0) {
        ctl->state = s_ls.state;
        ctl->pos_cur = s_ls.pc;
        ctl->arr_cur = s_ls.ac;
        ctl->step = s_ls.step;
        ctl->disp = s_ls.disp;
        ctl->n_rebuilds += s_ls.rebuilds;
        ctl->steps_done = s_ls.done;
        ctl->need_rebuild = s_ls.need_rb;
        ctl->resident_steps = s_ls.r_steps;
        ctl->tlog_n += s_ls.tlog_k;
        if (s_ls.rebuilds > 0) {
            ctl->list_grid = s_ls.rc == 0 ? g_size() : -1;
            ctl->list_chunk = blockDim.x;
        }
    }
    return true;
}

#if !SWP_BATCHED
template <typename Real, bool UNI, bool BONDS>
__global__ void __launch_bounds__(kThreads, 1) k_run(Dev<Real> d, RunArgs a)
{
    run_system<Real, UNI, BONDS>(d, a);
}
#else

// Batched launch: many independent systems in one cooperative launch.  Block
// b works through items[item_ofs[b] .. item_ofs[b + 1]), each (system, rank in
// the system's group, group size): a system either has a group of blocks to
// itself or runs on one block, which then advances its systems one after the
// other.  A block that belongs to a group of more than one block has no other
// item, so the group barriers only ever wait for blocks working on the same
// system.
template <typename Real, bool UNI, bool BONDS>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_batch(const Dev<Real>* devs, const RunArgs* args,
                                                     const int* item_ofs, const int4* items)
{
    __shared__ Dev<Real> s_dev;
    __shared__ RunArgs s_args;
    const int i0 = item_ofs[blockIdx.x], i1 = item_ofs[blockIdx.x + 1];
    for (int it = i0; it < i1; it++) {
        const int4 w = items[it];
        __syncthreads();  // the previous system is done with the shared copies
        const int* sd = (const int*)&devs[w.x];
        const int* sa = (const int*)&args[w.x];
        for (int k = threadIdx.x; k < (int)(sizeof(Dev<Real>) / 4); k += blockDim.x) ((int*)&s_dev)[k] = sd[k];
        for (int k = threadIdx.x; k < (int)(sizeof(RunArgs) / 4); k += blockDim.x) ((int*)&s_args)[k] = sa[k];
        if (threadIdx.x == 0) {
            s_grp[0] = w.y;
            s_grp[1] = w.z;
        }
        __syncthreads();
        if (!run_system<Real, UNI, BONDS>(s_dev, s_args)) {
            // a wait of this system ran out (latched in its status word): its
            // copies in flight land before the next system reuses the shared
            // buffers, and the block goes on with its other systems
            cp_async_wait_all();
            __syncthreads();
        }
    }
}
#endif  // SWP_BATCHED

#if SWP_HAS_RESIDENT
// ---------------------------------------------------------------------------
// Host-exchange kernels (user order <-> slot order).

// A new state from user-order arrays in device memory (v, type, mass, img null:
// zero, 0, one, zero), read where they are; also zeroes the counts of the list build and marks
// the control block (cleared before) for forces to be computed on a new list.
template <typename Real>
__global__ void k_set_state(Dev<Real> d, const double* x_in, const double* v_in, const int* type, const double* mass,
                            const int* img)
{
    typedef typename Dev<Real>::R4 R4;
    typedef typename Dev<Real>::P4 P4;
    const int n = d.n, t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    if (t == 0) {
        d.ctl->state = 1;
        d.ctl->need_rebuild = 1;
    }
    for (int c = t; c < d.ncell; c += nt) d.cell_cnt[c] = 0;
    for (int b = t; b < d.nbsum; b += nt) d.bsum[b] = 0;
    for (int i = t; i < n; i += nt) {
        long long qs[3];
        for (int c = 0; c < 3; c++) {
            // wrap into [0, L) and round to the fixed-point grid: one rounding per
            // operation (no contraction), so the conversion is reproducible
            const double L = (double)d.Lq[c] * kInvFix, x = x_in[3 * i + c];
            double xw = x;
            int im = 0;
            // inside the box already (the bits of non-negative doubles order like
            // their values): the quotient below is less than 1 and its floor 0, so
            // nothing changes, and the division, most of this kernel's FP64 work
            // (7 of the 200 us of a force call on 100,000 particles), is left out
            if (!((unsigned long long)__double_as_longlong(x) < (unsigned long long)__double_as_longlong(L))) {
                const double fl = floor(__ddiv_rn(x, L));
                im = (int)fl;
                xw = __dsub_rn(x, __dmul_rn(fl, L));
            }
            long long q = __double2ll_rn(__dmul_rn(xw, kFix));
            if (q >= d.Lq[c]) {
                q -= d.Lq[c];
                im++;
            }
            if (q < 0) {
                q += d.Lq[c];
                im--;
            }
            d.xq[0][c * n + i] = q;
            d.img[0][c * n + i] = im + (img ? img[3 * i + c] : 0);
            qs[c] = q;
        }
        int ty = type ? type[i] : 0;
        if ((unsigned)ty >= (unsigned)d.ntypes) {  // (device input is not checked on the host)
            atomicOr(&d.ctl->status, kStatusBadType);
            ty = 0;
        }
        P4 p;
        p.x = snap_coord(qs[0], 0, d);
        p.y = snap_coord(qs[1], 1, d);
        p.z = snap_coord(qs[2], 2, d);
        p.w = snap_bits((i << kTypeBits) | ty, d);
        d.pos[0][i] = p;
        R4 v;
        v.x = v_in ? (Real)v_in[3 * i + 0] : Real(0);
        v.y = v_in ? (Real)v_in[3 * i + 1] : Real(0);
        v.z = v_in ? (Real)v_in[3 * i + 2] : Real(0);
        v.w = mass ? (Real)(1.0 / mass[i]) : Real(1);
        d.vel[0][i] = v;
    }
}

// The state in user order into x, v, img (each may be null), device memory.
template <typename Real>
__global__ void k_get_state(Dev<Real> d, int pc, int ac, double* x, double* v_out, int* img)
{
    typedef typename Dev<Real>::R4 R4;
    const int n = d.n;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const size_t tag = pos_bits(d.pos[pc][q]) >> kTypeBits;
        const R4 v = d.vel[ac][q];
        for (int c = 0; c < 3; c++) {
            if (x) x[3 * tag + c] = (double)d.xq[ac][c * n + q] * kInvFix;
            if (img) img[3 * tag + c] = d.img[ac][c * n + q];
        }
        if (v_out) {
            v_out[3 * tag + 0] = (double)v.x;
            v_out[3 * tag + 1] = (double)v.y;
            v_out[3 * tag + 2] = (double)v.z;
        }
    }
}

// Forces in user order into f (device memory).  pc < 0: the current snapshot set
// as the control block records it.  U (may be null): the potential energy of the
// thermo record.
template <typename Real>
__global__ void k_get_forces(Dev<Real> d, int pc, double* f_out, double* U)
{
    typedef typename Dev<Real>::R4 R4;
    const int n = d.n;
    if (pc < 0) pc = d.ctl->pos_cur;
    if (U && blockIdx.x == 0 && threadIdx.x == 0) U[0] = d.ctl->thermo[Q_U2] + d.ctl->thermo[Q_U3];
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const size_t tag = pos_bits(d.pos[pc][q]) >> kTypeBits;
        const R4 f = d.force[q];
        f_out[3 * tag + 0] = (double)f.x;
        f_out[3 * tag + 1] = (double)f.y;
        f_out[3 * tag + 2] = (double)f.z;
    }
}

template <typename Real>
__global__ void k_get_nlist(Dev<Real> d, int pc, int* rows, int* counts, int width)
{
    const int n = d.n;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const int tag = pos_bits(d.pos[pc][q]) >> kTypeBits;
        const int4 inf = d.pinfo[q];
        counts[2 * tag] = inf.y;
        counts[2 * tag + 1] = inf.y + inf.w;
        int* out = rows + (size_t)tag * width;
        int k = 0;
        for (int m = 0; m < inf.y && k < width; m++, k++)
            out[k] = pos_bits(d.pos[pc][d.ent_j[(unsigned)inf.x + m]]) >> kTypeBits;
        for (int m = 0; m < inf.w && k < width; m++, k++)
            out[k] = pos_bits(d.pos[pc][d.ent_j[(unsigned)inf.z + m]]) >> kTypeBits;
    }
}

// ---------------------------------------------------------------------------
// Derivatives with respect to the reactive pair's coefficients (lambda, eps,
// sigma), at the current positions and list, for one reactive type pair
// (a^2 = lambda eps) and the unshifted form.  With x = (sigma/r)^n:
//   v = 4 eps (x^2 - x),  vh = 4 (x - x^2) beyond r_min (1 inside),
//   Q = 4 n (2x^2 - x) (= -r v'/eps), q = Q beyond r_min (0 inside) (= r vh'),
//   S_i = sum_k vh_ik, D_i = sum_k q_ik (over i's reactive partners inside r_cut),
//   T = sum_i sum_{j<k} vh_ij vh_ik = 1/2 sum_i (S_i^2 - sum_j vh_ij^2),
//   U = sum_pairs v + lambda eps T (+ the pairs that do not depend on theta).
// Then dU/dlambda = eps T, dU/deps = sum_pairs v/eps + lambda T,
//   dU/dsigma = (eps sum_pairs Q + lambda eps sum_i (sum_j vh_ij q_ij - S_i D_i)) / sigma,
// and, with the pair force F_i = -ft (x_j - x_i), ft = eps (Q - lambda g q) / r^2,
// g = S_i + S_j - 2 vh:
//   dft/dlambda = -eps g q / r^2,   dft/deps = (Q - lambda g q) / r^2,
//   dft/dsigma = (eps Q_s - lambda eps ((2q - D_i - D_j) q + g q_s)) / (sigma r^2),
//   Q_s = 4 n^2 x (4x - 1) (= sigma dQ/dsigma), q_s = Q_s beyond r_min (0 inside).
// Decisions (inside r_cut, beyond r_min) are the force kernels' own.

//
// Both passes are bound by the FP64 pipe (19 cycles per warp instruction on an
// SM, however many lanes are on).  A lane takes one particle (FP32: in the
// threads' order of the list, alike rows in a warp), first lines up the partners
// inside the cut-off (they are half of the listed ones) and then works through
// them, so that a warp's FP64 work is that of its fullest particle; sums are kept
// of the bare products (x, x^2, ...), the factors follow once per particle.
// Blocks of two warps spread 20,000 particles over every SM.  (Four lanes per
// particle, every listed partner, a division for each derivative: a
// gradient over 16 snapshots of 20,000 took 2.62 ms, now 1.93.)

constexpr int kPgThreads = 64;

// A particle's reactive partners inside the cut-off, a few at a time.
template <typename Real>
struct PgLine {
    static constexpr int kCap = 12;
    struct Item {
        Real r2, dx, dy, dz;
        int j;
    };
    Item item[kCap][kPgThreads];
};

// Particle of index q in the order the two passes take them, and its list ranges.
__device__ __forceinline__ int pg_particle(const Dev<float>& d, int q, int4& inf)
{
    inf = d.tinfo[q];
    return d.perm[q];
}
__device__ __forceinline__ int pg_particle(const Dev<double>& d, int q, int4& inf)
{
    inf = d.pinfo[q];
    return q;
}

// f(item) for every reactive partner of the lane's particle inside the cut-off,
// in list order; the warp's lanes go through their lines together.
template <typename Real, typename F>
__device__ __forceinline__ void pg_partners(const Dev<Real>& d, const typename Dev<Real>::P4* pos, Real rc2,
                                            const typename Dev<Real>::P4& pi, const int4& inf, PgLine<Real>& line, F&& f)
{
    typedef typename Dev<Real>::P4 P4;
    const int t = threadIdx.x;
    int k = 0;
    while (__any_sync(0xffffffffu, k < inf.y)) {
        int m = 0;
        for (; k < inf.y && m + 4 <= PgLine<Real>::kCap; k += 4) {
            int j[4];
            P4 pj[4];
#pragma unroll
            for (int u = 0; u < 4; u++) j[u] = k + u < inf.y ? d.ent_j[(unsigned)inf.x + k + u] : -1;
#pragma unroll
            for (int u = 0; u < 4; u++) pj[u] = pos[max(j[u], 0)];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                Real dx, dy, dz;
                const Real r2 = dist2_listed(pi, pj[u], d, dx, dy, dz);
                if (j[u] >= 0 && r2 < rc2) {
                    line.item[m][t] = {r2, dx, dy, dz, j[u]};
                    m++;
                }
            }
        }
        __syncwarp();
        for (int e = 0; __any_sync(0xffffffffu, e < m); e++)
            if (e < m) f(line.item[e][t]);
        __syncwarp();
    }
}

// Pass 1: S_i and D_i per slot into sd[2i], sd[2i+1]; per-block sums of
// (T, sum_i (sum_j vh q - S D), sum_pairs v/eps, sum_pairs Q) into part[4b..].
// pair: the reactive pair's place in the table.
template <typename Real>
__global__ void __launch_bounds__(kPgThreads) k_pgrad_sums(Dev<Real> d, int pc, int pair, double* sd, double* part)
{
    __shared__ PgLine<Real> line;
    __shared__ double red[4][kPgThreads / 32];
    const int n = d.n;
    if (pc < 0) pc = d.ctl->pos_cur;
    const PairP<Real> p = d.table[pair];
    const double nn = (double)p.n_real;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int q0 = blockIdx.x * kPgThreads; q0 < n; q0 += gridDim.x * kPgThreads) {
        const int q = q0 + threadIdx.x;
        int4 inf = make_int4(0, 0, 0, 0);
        const int i = q < n ? pg_particle(d, q, inf) : 0;
        const typename Dev<Real>::P4 pi = d.pos[pc][i];
        // with w = x - x^2 and u = 2x^2 - x: v/eps = -4 w, vh = 4 w and q = Q = 4 n u beyond r_min
        double w1 = 0.0, x2 = 0.0, wb = 0.0, ub = 0.0, ww = 0.0, wu = 0.0;
        int inside = 0;  // partners inside r_min (vh = 1, q = 0)
        pg_partners(d, d.pos[pc], p.rc2, pi, inf, line, [&](const typename PgLine<Real>::Item& it) {
            const double x = (double)pair_power<kExpoAny, true>(p, p.sig2 * recip(it.r2));
            const double xx = x * x, w = x - xx, u = xx - w;
            const bool beyond = it.r2 > p.rmin2;
            w1 += w;
            x2 += xx;
            const double wo = beyond ? w : 0.0, uo = beyond ? u : 0.0;
            inside += !beyond;
            wb += wo;
            ub += uo;
            ww += wo * wo;
            wu += wo * uo;
        });
        if (q < n) {
            const double S = 4.0 * wb + (double)inside, Dn = 4.0 * nn * ub;
            sd[2 * i] = S;
            sd[2 * i + 1] = Dn;
            acc[0] += 0.5 * (S * S - (16.0 * ww + (double)inside));
            acc[1] += 16.0 * nn * wu - S * Dn;
            acc[2] -= 2.0 * w1;  // each pair is listed from both ends
            acc[3] += 2.0 * nn * (x2 - w1);
        }
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) red[k][wp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int k = 0; k < kPgThreads / 32; k++) t += red[threadIdx.x][k];
        part[4 * blockIdx.x + threadIdx.x] = t;
    }
}

// Pass 2: dF/dtheta per particle, in user order: out[(k n + tag) 3 + c];
// theta = (lambda, eps, sigma) in device memory.
template <typename Real>
__global__ void __launch_bounds__(kPgThreads) k_pgrad_forces(Dev<Real> d, int pc, int pair, const double* sd,
                                                             const double* theta, double* out)
{
    __shared__ PgLine<Real> line;
    const int n = d.n;
    if (pc < 0) pc = d.ctl->pos_cur;
    const PairP<Real> p = d.table[pair];
    const double lam = theta[0], eps = theta[1], sig = theta[2], nn = (double)p.n_real, n4 = 4.0 * nn;
    for (int q0 = blockIdx.x * kPgThreads; q0 < n; q0 += gridDim.x * kPgThreads) {
        const int q = q0 + threadIdx.x;
        int4 inf = make_int4(0, 0, 0, 0);
        const int i = q < n ? pg_particle(d, q, inf) : 0;
        const typename Dev<Real>::P4 pi = d.pos[pc][i];
        const double Si = sd[2 * i], Di = sd[2 * i + 1];
        double g[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
        pg_partners(d, d.pos[pc], p.rc2, pi, inf, line, [&](const typename PgLine<Real>::Item& it) {
            const double Sj = sd[2 * it.j], Dj = sd[2 * it.j + 1];
            const double x = (double)pair_power<kExpoAny, true>(p, p.sig2 * recip(it.r2));
            const bool beyond = it.r2 > p.rmin2;
            const double c = n4 * (1.0 / (double)it.r2);  // 4 n / r^2
            const double xx = x * x, w = x - xx, u = xx - w, z = 4.0 * xx - x;
            const double vh = beyond ? 4.0 * w : 1.0;
            const double gg = (Si + Sj) - 2.0 * vh;
            const double Q = c * u, Qs = c * nn * z;  // Q / r^2, Q_s / r^2
            const double qb = beyond ? Q : 0.0, qs = beyond ? Qs : 0.0;
            const double h = gg * qb;
            // dft/dlambda = -eps h, dft/deps = Q/r^2 - lambda h,
            // dft/dsigma = eps/sigma (Q_s/r^2 - lambda ((2q - D_i - D_j) q/r^2 + g q_s/r^2))
            const double a = (2.0 * (n4 * u) - (Di + Dj)) * qb + gg * qs;
            const double f[3] = {h, Q - lam * h, Qs - lam * a};
            const double dv[3] = {(double)it.dx, (double)it.dy, (double)it.dz};
#pragma unroll
            for (int k = 0; k < 3; k++)
#pragma unroll
                for (int e = 0; e < 3; e++) g[k][e] += f[k] * dv[e];
        });
        if (q < n) {
            const size_t tag = pos_bits(pi) >> kTypeBits;
            const double scale[3] = {eps, -1.0, -eps / sig};  // F_i = -ft (x_j - x_i)
#pragma unroll
            for (int k = 0; k < 3; k++)
#pragma unroll
                for (int e = 0; e < 3; e++) out[((size_t)k * n + tag) * 3 + e] = scale[k] * g[k][e];
        }
    }
}

// Pass 3: one block of four warps adds the per-block sums into total[4] --
// warp k sums quantity k, lane l the blocks l, l + 32, ... in order, then a
// fixed shuffle tree -- and forms dU/dtheta from them into dU[3] (when given).
static __global__ void k_pgrad_total(const double* part, int nblocks, double* total, const double* theta,
                                     double* dU)
{
    __shared__ double t[4];
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k < 4) {
        double v = 0.0;
        for (int b = lane; b < nblocks; b += 32) v += part[4 * b + k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            total[k] = v;
            t[k] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && dU) {
        // t = (T, sum_i (sum_j vh q - S D), sum_pairs v/eps, sum_pairs Q)
        const double lam = theta[0], eps = theta[1], sig = theta[2];
        dU[0] = eps * t[0];
        dU[1] = t[2] + lam * t[0];
        dU[2] = (eps * t[3] + lam * eps * t[1]) / sig;
    }
}

// Start of one device-driven evaluation (swp_eval_grad), one warp: clears the
// control block (k_set_state follows) and writes the reactive pair's coefficients
// from theta = (lambda, eps, sigma) in device memory into both (ti, tj) entries
// of the device pair table (the theta-dependent ones; the same arithmetic as the
// host table).  c_rmin = 2^(1/n), c_rb = ((1 - sqrt(1/2)) / 2)^(-1/n) (host
// constants), rbond > 0: the bond radius as given.
template <typename Real>
__global__ void k_eval_prep(Dev<Real> d, int ti, int tj, const double* theta, double c_rmin, double c_rb, double rbond)
{
    int* w = (int*)d.ctl;
    for (int k = threadIdx.x; k < (int)(sizeof(Ctl) / sizeof(int)); k += 32) w[k] = 0;
    if (threadIdx.x == 0) {
        const double lam = theta[0], eps = theta[1], sig = theta[2];
        PairP<Real>* tab = (PairP<Real>*)d.table;
        PairP<Real> e = tab[ti * d.ntypes + tj];
        e.four_eps = (Real)(4.0 * eps);
        e.sig2 = (Real)(sig * sig);
        const double rmin = sig * c_rmin;
        e.rmin2 = (Real)(rmin * rmin);
        e.a = (Real)sqrt(lam * eps);
        e.inv_epshat = (Real)(1.0 / eps);
        const double rb = rbond > 0.0 ? rbond : sig * c_rb;
        e.rbond2 = (Real)(rb * rb);
        tab[ti * d.ntypes + tj] = e;
        tab[tj * d.ntypes + ti] = e;
    }
}

// Before a batched launch: every system's barrier counter starts at zero.
template <typename Real>
__global__ void k_batch_begin(const Dev<Real>* devs, int m)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < m) devs[r].ctl->barrier = 0;
}

// After it: the control blocks of the systems that hold a place in pinned memory,
// one warp per system, the ticket last.
template <typename Real>
__global__ void k_batch_end(const Dev<Real>* devs, int m)
{
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (r >= m || !devs[r].slot) return;
    const int* src = (const int*)devs[r].ctl;
    int* dst = (int*)&devs[r].slot->ctl;
    for (int k = lane; k < (int)(sizeof(Ctl) / sizeof(int)); k += 32) dst[k] = src[k];
    __syncwarp();
    __threadfence_system();
    if (lane == 0) *(volatile unsigned long long*)&devs[r].slot->ticket = devs[r].ticket;
}

#endif  // SWP_HAS_RESIDENT

}  // namespace single / wide / SWP_BATCH_NS
}  // namespace swp
