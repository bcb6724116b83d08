// resident.cuh -- p(l)-CG of small and mid-sized stencil systems with every
// row's state in its thread (l <= 3, R = 1, 2 or 4 rows per thread).
//
// An iteration of a small system is a chain of latencies, not a stream of
// bytes.  Here a thread keeps its rows for the whole solve -- z^(l)_i and
// z^(l)_{i-1}, the current and previous vector of every other basis, phat and
// x in registers -- and only z^(l)_{i+1} goes to global memory, for the
// neighbours.  (At 512 threads a block there are 128 registers: the compiler keeps
// part of a thread's state in local memory, in the L1 -- 290 bytes of spill stores
// in the code for FP32, l = 1, R = 1 up to 1600 for FP64, l = 3, R = 4.)
// What bounds an iteration on GB300 then: an FP64 warp instruction
// takes 64 cycles on its SM sub-partition whether one lane or all are active,
// so the scalar chain and the reductions cost as much as the sweep, and an L2
// round trip costs about ten of them.  Hence
//  * warp 0 forms the coefficients, warp 1 the other scalars, the rest sweep
//    (the first sweeping warps sit on the two sub-partitions these leave free);
//  * no fences and no grid barrier in an iteration: every 64-bit word another
//    CTA reads carries its own tag (see ResExch), rows wait for their
//    neighbours' z, and only the scalars wait for all CTAs' dots (with a
//    barrier, fences and partials read after it, 100^2 p(1)-CG took 4.9 us);
//  * the scalar step in three: what needs no new dot product (pre), what the
//    sweep waits for (crit: one reciprocal square root, gamma, K4's
//    coefficients one lane each) and what only the next step needs (post); pre
//    and post run during the sweep, with l >= 2 crit does, too (Algorithm 2's
//    overlap of the reduction), and with l = 1 the sweep's loads overlap it.
// Measured on GB300 against the grid and cluster paths (us per iteration): 2D
// 32^2 FP64 p(1) 5.13 -> 2.98, p(2) 5.14 -> 2.77; 2D 100^2 FP64 p(1) 6.51 ->
// 3.27, p(2) 6.03 -> 2.90, FP32 p(1) 7.54 -> 3.10; 3D 50^3 FP32 p(1) 13.7 ->
// 4.7; 3D 75 x 61 x 57 FP64 (4 rows per thread, bound by FP64 instructions and
// the neighbour loads) p(1) 15.96 -> 10.4, p(3) 17.6 -> 14.7.  At 272k rows, the
// most four rows per thread hold, it still leads (2D 512^2: FP64 1.16-1.5x,
// FP32 2.0-2.4x).
// The arithmetic on a row is that of solver.cuh's sweep, operation for
// operation (FP32 solutions are bit-identical in practice); dots are summed in
// another fixed order.
#pragma once

#include "fastroot.h"
#include "solver.cuh"

namespace plcg {

// FP32 dots (sum and error) widened and added: with widen_f32 where all are zero
// or normal; subnormals, infinities and NaN take the conversions (out of line:
// inlined, they were issued ahead of the test, and a conversion costs as much as
// any FP64 instruction -- 3D 50^3 p(1)-CG 4.7 -> 5.0 us per iteration).
static __device__ __noinline__ double widened_sum_any(float s, float t) { return (double)s + (double)t; }

template <int N, class Acc>
__device__ __forceinline__ void widened_sums(const Acc (&d)[N], double (&v)[N])
{
    uint32_t lo = 0xffffffffu, hi = 0u;   // of |x| - 1 (zero: the largest) and |x|, as integers
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const uint32_t a = __float_as_uint(d[q].s) & 0x7fffffffu, b = __float_as_uint(d[q].t) & 0x7fffffffu;
        lo = min(lo, min(a - 1u, b - 1u));
        hi = max(hi, max(a, b));
        v[q] = widen_f32(d[q].s) + widen_f32(d[q].t);
    }
    if (__builtin_expect(lo < 0x007fffffu || hi >= 0x7f800000u, 0)) {
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = widened_sum_any(d[q].s, d[q].t);
    }
}

template <typename T, int L>
struct ResCoef {
    int rec;                  // recurrences (i >= l), else the fill phase
    int first;                // m = 0: phat_0 = v_0
    int end;                  // -1: continue, else SegEnd
    int fmode;                // as Coef::fmode
    int kseg;                 // k of the iterate the segment returns (when end >= 0)
    T sig;                    // fill: sigma_i
    T co[4 + L];              // K4: 0 1/delta, 1 of z^(l)_i, 2 of z_{i-1}, 3 of the neighbour sum, 4 + k of z^(k)
    T zx, pp;
    T f1, f2, fpv, fpp;       // final update
};

template <typename T, int L>
struct ResSmem {
    double red[2][kResBlock / 32][L + 1];   // dots of the sweeping warps, iterations i & 1
    double raw[L + 1];
    double norms[2];
    double G[L + 1][2 * L + 1];      // finalised columns c-l .. c (column c at c mod (l+1))
    double Ginv[L + 1];
    double gam[L + 1], del[L + 1], idel[L + 1];
    double zeta[2], ieta[2];
    double sig[L];
    double A, D, igmm, B, C;         // pre: gamma = (A + D g_{m,c}) igmm, 1/delta = B / g_cc, delta = C g_cc
    double dm1, lam, zm;
    double arg, rg, gm, invd;        // crit -> post
    double X[32];                    // l = 1: res_coef_x by lane
    ResCoef<T, L> cf[2];
    // a bounded wait of this CTA ran out, or another CTA gave up: by the parity of
    // the iteration (2: exchange2), written before and read after that
    // iteration's CTA barrier.  A warp that is an iteration ahead writes the other
    // one, so all warps of the CTA leave after the same barrier.
    int fail[3];
};

__device__ __forceinline__ bool finite_bits(double v)
{
    return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

// ------------------------------------------------------------------------
// Exchanges between the CTAs without fences: every 64-bit word that another
// CTA reads carries a number (its exchange's or its iteration's), so a reader
// spins on the data itself and a writer need not order anything before a
// flag.  A double takes the two words {high half, tag} and {low half, tag},
// a float one.
//  * z^(l)_i of every row, in buffer i & 1.  A row's z_{i+2} is written after
//    its neighbours' z_{i+1} were read, and those were formed from the row's
//    z_i (the stencil is symmetric), so two buffers suffice.
//  * the dots of exchange e, in slot e mod kResSlots.  A CTA publishes
//    exchange e when every CTA has published e - l, and reads reach back l
//    exchanges, so fewer than kResSlots are ever in use.
// Tags grow through a launch; the kernel clears the z tags of its rows before
// the first exchange, the launch the packets.
// ------------------------------------------------------------------------
__device__ __forceinline__ void st_tagged(unsigned long long *p, double v, unsigned e)
{
    const unsigned long long h = ((unsigned long long)(unsigned)__double2hiint(v) << 32) | e;
    const unsigned long long l = ((unsigned long long)(unsigned)__double2loint(v) << 32) | e;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(h), "l"(l) : "memory");
}

__device__ __forceinline__ void st_tagged(unsigned long long *p, float v, unsigned e)
{
    const unsigned long long w = ((unsigned long long)__float_as_uint(v) << 32) | e;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

// The words at p (a batch of loads is issued before the first is looked at,
// without branches between them), their value, and whether they carry tag e.
template <typename T>
struct Tagged;
template <>
struct Tagged<double> {
    unsigned long long h, l;
    __device__ __forceinline__ void load(const unsigned long long *p)
    {
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(h), "=l"(l) : "l"(p) : "memory");
    }
    __device__ __forceinline__ double value() const { return __hiloint2double((int)(h >> 32), (int)(l >> 32)); }
    __device__ __forceinline__ bool is(unsigned e) const { return (((unsigned)h ^ e) | ((unsigned)l ^ e)) == 0u; }
};
template <>
struct Tagged<float> {
    unsigned long long w;
    __device__ __forceinline__ void load(const unsigned long long *p)
    {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    }
    __device__ __forceinline__ float value() const { return __uint_as_float((unsigned)(w >> 32)); }
    __device__ __forceinline__ bool is(unsigned e) const { return (unsigned)w == e; }
};

struct ResExch {
    unsigned long long *pkt;
    int P, rank, nd;            // CTAs, this CTA, doubles per packet
    unsigned long long limit;   // a poll is an L2 round trip of several loads: an eighth of the grid barrier's
    unsigned force;             // test hook: waits of exchanges from this number on run out
    int *abort_flag;
    __device__ __forceinline__ unsigned long long *at(unsigned e, int cta, int q) const
    {
        return pkt + (((size_t)(e % kResSlots) * P + cta) * nd + q) * 2;
    }
    // After the poll number `polls`: true to give up (the bound ran out or
    // another CTA gave up).
    __device__ __forceinline__ bool give_up(unsigned long long polls) const
    {
        if ((polls & 63) != 0) return false;
        if (polls > limit) atomicExch(abort_flag, 1);
        return ld_volatile(abort_flag) != 0;
    }
    // One warp: wait for dots q0 .. q0 + NA - 1 of exchange e from every CTA;
    // v[k][q] = dot q0 + q of CTA lane + 32 k (0 past the last CTA).  False:
    // gave up.
    template <int NA>
    __device__ __forceinline__ bool wait(unsigned e, int q0, double (&v)[kResChunks][NA]) const
    {
        const int lane = threadIdx.x & 31;
        const unsigned want = e + (e >= force ? 1u : 0u);   // (no tag of this slot: those differ by kResSlots)
        const unsigned long long *p[kResChunks];
#pragma unroll
        for (int k = 0; k < kResChunks; ++k) p[k] = at(e, min(lane + 32 * k, P - 1), q0);
        for (unsigned long long polls = 1;; ++polls) {
            Tagged<double> t[kResChunks][NA];
#pragma unroll
            for (int k = 0; k < kResChunks; ++k) {
                if (32 * k >= P) continue;   // uniform
#pragma unroll
                for (int q = 0; q < NA; ++q) t[k][q].load(p[k] + 2 * q);
            }
            bool ready = true;
#pragma unroll
            for (int k = 0; k < kResChunks; ++k) {
#pragma unroll
                for (int q = 0; q < NA; ++q) {
                    v[k][q] = 0.0;
                    if (32 * k >= P) continue;
                    ready &= t[k][q].is(want);
                    if (lane + 32 * k < P) v[k][q] = t[k][q].value();
                }
            }
            if (__all_sync(0xffffffffu, ready)) return true;
            if (__any_sync(0xffffffffu, give_up(polls))) return false;
        }
    }
};

// The sums over the CTAs of wait()'s values (a fixed order, so every CTA gets
// the same bits), written to dst[0 .. NA-1].
template <int NA>
__device__ __forceinline__ void res_sum(const double (&v)[kResChunks][NA], int P, double *dst)
{
    const int lane = threadIdx.x & 31;
    double t[NA];
#pragma unroll
    for (int q = 0; q < NA; ++q) {
        t[q] = v[0][q];
        // a chunk without CTAs adds nothing: its instructions are skipped
        if (P > 64) t[q] = (t[q] + v[1][q]) + (P > 96 ? v[2][q] + v[3][q] : v[2][q]);
        else if (P > 32) t[q] += v[1][q];
        if (P > 128) t[q] += v[4][q];
    }
    constexpr int S = NA <= 1 ? 0 : NA <= 2 ? 1 : 2;
    const double r = warp_reduce_scatter<NA>(t, lane);
    if ((lane & ((32 >> S) - 1)) == 0) {
        const int q = lane >> (5 - S);
        if (q < NA) dst[q] = r;
    }
    __syncwarp();
}
static_assert(kResChunks == 5, "res_sum adds five chunks of 32 CTAs");

// Sum of column q of red over the nw sweeping warps, two lanes' worth at a
// time: lanes 0 .. 15 hold column q0, lanes 16 .. 31 column q0 + 1; the sums
// end in lanes 0 and 16.
template <int NA>
__device__ __forceinline__ double res_warps_sum(const double (*red)[NA], int q0, int nw)
{
    const int lane = threadIdx.x & 31, q = q0 + (lane >> 4), w = lane & 15;
    double t = (w < nw && q < NA) ? red[w][q] : 0.0;
    if (nw > 8) t += __shfl_xor_sync(0xffffffffu, t, 8);
    if (nw > 4) t += __shfl_xor_sync(0xffffffffu, t, 4);
    if (nw > 2) t += __shfl_xor_sync(0xffffffffu, t, 2);
    if (nw > 1) t += __shfl_xor_sync(0xffffffffu, t, 1);
    return t;
}

// One warp: the CTA's totals of red's columns, published as exchange e.
template <int NA>
__device__ __forceinline__ void res_publish(const ResExch &x, unsigned e, const double (*red)[NA], int nw)
{
    const int lane = threadIdx.x & 31;
    double t[(NA + 1) / 2];
#pragma unroll
    for (int h = 0; h < (NA + 1) / 2; ++h) t[h] = res_warps_sum<NA>(red, 2 * h, nw);
#pragma unroll
    for (int h = 0; h < (NA + 1) / 2; ++h) {
        const int q = 2 * h + (lane >> 4);
        if ((lane & 15) == 0 && q < NA) st_tagged(x.at(e, x.rank, q), t[h], e);
    }
}

// ------------------------------------------------------------------------
// The scalar step of iteration i in three parts (m = i - l, c = m + 1).
// ------------------------------------------------------------------------
// One lane; after crit(i) has published its coefficients.
template <typename T, int L>
__device__ __forceinline__ void res_post(ResSmem<T, L> &s, int i)
{
    const int m = i - L, c = m + 1;
    if (m < 0) return;
    const double gcc = s.arg * s.rg, dm = gcc * s.C;
    s.G[c % (L + 1)][2 * L] = gcc;
    s.del[m % (L + 1)] = dm;
    s.idel[m % (L + 1)] = s.invd;
    s.gam[m % (L + 1)] = s.gm;
    const double em = m >= 1 ? s.gm - s.lam * s.dm1 : s.gm;
    s.ieta[m & 1] = fast_rcp(em);
}

// One lane; needs post(i - 1).
template <typename T, int L>
__device__ __forceinline__ void res_pre(ResSmem<T, L> &s, int i, double rn, double tau, long long budget)
{
    ResCoef<T, L> &cf = s.cf[i & 1];
    const int m = i - L;
    cf.end = -1;
    cf.fmode = 0;
    cf.f1 = T(0);
    cf.rec = m >= 0;
    if (m < 0) {
        cf.sig = (T)s.sig[i];
        return;
    }
    cf.first = m == 0;
    cf.kseg = m;
    const double *col = s.G[m % (L + 1)];
    const double gmm = col[2 * L], igmm = s.Ginv[m % (L + 1)];
    double dm1 = 0.0, lam = 0.0, zm = rn;
    if (m >= 1) {
        dm1 = s.del[(m - 1) % (L + 1)];
        const double iep = s.ieta[(m - 1) & 1], ze = s.zeta[(m - 1) & 1];
        lam = dm1 * iep;
        zm = -lam * ze;
        cf.zx = (T)(ze * iep);
        cf.pp = (T)(-lam);
        if (!finite_bits(zm)) {
            cf.end = kSegNonfinite;
        } else if (fabs(zm) < tau || m >= budget) {
            cf.end = fabs(zm) < tau ? kSegConverged : kSegMaxit;
            cf.f1 = cf.zx;
        }
    }
    s.zeta[m & 1] = zm;
    s.dm1 = dm1;
    s.lam = lam;
    s.zm = zm;
    const double gd = m >= 1 ? col[2 * L - 1] * dm1 : 0.0;
    s.igmm = igmm;
    if (m < L) {
        s.A = s.sig[m] * gmm - gd;
        s.D = 1.0;
        s.B = gmm;
        s.C = igmm;
    } else {
        const double d = s.del[(m - L) % (L + 1)];
        s.A = gmm * s.gam[(m - L) % (L + 1)] - gd;
        s.D = d;
        s.B = gmm * s.idel[(m - L) % (L + 1)];
        s.C = d * igmm;
    }
}

// K4's coefficients are all X / delta_m; X by lane: 0 1, 1 kc - gamma (FP32:
// -gamma, the sweep's coefficient being rounded as in solver.cuh), 2
// -delta_{m-1}, 3 kn, 4 + k sigma_k - gamma.
template <typename T, int L>
__device__ __forceinline__ double res_coef_x(const ResSmem<T, L> &s, int m, double gm, T kc, T kn)
{
    const int lane = threadIdx.x & 31;
    const double c0 = lane == 0 ? 1.0 : lane == 1 ? (sizeof(T) == 8 ? (double)kc : 0.0)
                    : lane == 2 ? (m >= 1 ? -s.dm1 : 0.0) : lane == 3 ? (double)kn : s.sig[lane - 4 < L ? lane - 4 : 0];
    return (lane == 0 || lane == 2 || lane == 3) ? c0 : c0 - gm;
}

// ... written from 1 / delta_m, one lane per coefficient.
template <typename T, int L>
__device__ __forceinline__ void res_coefs(ResCoef<T, L> &cf, double X, double invd, T kc, T kn)
{
    const int lane = threadIdx.x & 31;
    T v = (T)(X * invd);
    if constexpr (sizeof(T) == 4) {
        const T inv = __shfl_sync(0xffffffffu, v, 0);
        v = lane == 1 ? fma(kc, inv, v) : lane == 3 ? kn * inv : v;
    }
    if (lane < 4 + L) cf.co[lane] = v;
}

// The breakdown test of iteration i (arg <= thr = 64 eps |graw|) in full, out
// of line.
template <typename T, int L>
__device__ __noinline__ void res_breakdown(ResSmem<T, L> &s, ResCoef<T, L> &cf, int m, double graw, double arg, double gm)
{
    if (threadIdx.x & 31) return;
    const double thr = 64.0 * Eps<T>::v * fabs(graw);
    const double zep = m >= 1 ? s.zeta[(m - 1) & 1] : 0.0, iep = m >= 1 ? s.ieta[(m - 1) & 1] : 0.0;
    if (!finite_bits(arg) || !finite_bits(gm)) {
        cf.end = kSegNonfinite;
        cf.f1 = T(0);
    } else if (arg <= thr) {
        if (arg >= -thr) {   // lucky breakdown: x_{m+1} is exact in this Krylov space
            if (m == 0) {
                cf.fmode = 2;
                cf.fpv = (T)(1.0 / gm);
                cf.f2 = (T)s.zm;
            } else {
                const double iem = 1.0 / (gm - s.lam * s.dm1);
                cf.fmode = 1;
                cf.f1 = (T)(zep * iep);
                cf.fpv = (T)iem;
                cf.fpp = (T)(-s.dm1 * iem * iep);
                cf.f2 = (T)s.zm;
            }
            cf.end = kSegLucky;
            cf.kseg = m + 1;
        } else {             // breakdown: keep x_m and restart
            cf.fmode = 0;
            cf.f1 = (T)(m >= 1 ? zep * iep : 0.0);
            cf.end = kSegBreakdown;
        }
    }
}

// ... the exponents decide it in all but the close cases (an FP64 comparison
// costs as much as any FP64 instruction).  Whole warp, uniform; pre has
// written the end that the other stop tests ask for.
template <typename T, int L>
__device__ __forceinline__ void res_end(ResSmem<T, L> &s, ResCoef<T, L> &cf, int m, double graw, double arg, double gm)
{
    constexpr int kThr = 6 - (sizeof(T) == 8 ? 52 : 23);
    const int ea = (__double2hiint(arg) >> 20), eg = (__double2hiint(graw) >> 20) & 0x7ff;   // ea < 0: arg < 0; 0: zero or subnormal
    if (__builtin_expect(!finite_bits(arg) || !finite_bits(gm) || ea <= max(eg + kThr + 1, 0), 0))
        res_breakdown<T, L>(s, cf, m, graw, arg, gm);
}

__device__ __forceinline__ void res_bar_all() { asm volatile("bar.sync 0;" ::: "memory"); }
__device__ __forceinline__ void res_bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void res_bar_arrive(int id, int n)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// crit for l >= 2: a whole warp, every lane on the same values; raw = the
// dots of iteration i - l, positions l .. 2l; join(): until pre(i) is done
// (its results are used from there on).
template <typename T, int L, class Join>
__device__ __forceinline__ void res_crit(ResSmem<T, L> &s, int i, T kc, T kn, const Join &join)
{
    ResCoef<T, L> &cf = s.cf[i & 1];
    const int m = i - L, c = m + 1;
    double col[2 * L];
    // rows c-2l .. c-l-1 by the symmetry of G (Sec. 2.2), c-l as computed, the
    // others less their projections; rows before 0 are zero
#pragma unroll
    for (int q = 0; q < L; ++q) col[q] = (c - 2 * L + q >= 0) ? s.G[(c - L + q) % (L + 1)][2 * L - q] : 0.0;
#pragma unroll
    for (int q = L; q < 2 * L; ++q) {
        const int j = c - 2 * L + q;
        col[q] = 0.0;
        if (j < 0) continue;
        double t = s.raw[q - L];
        if (q > L) {
            const double *gj = s.G[j % (L + 1)];
#pragma unroll
            for (int k = 0; k < q; ++k) t -= gj[2 * L - q + k] * col[k];
            t *= s.Ginv[j % (L + 1)];
        }
        col[q] = t;
    }
    const double graw = s.raw[L];
    double arg = graw;
#pragma unroll
    for (int q = 0; q < 2 * L; ++q) arg -= col[q] * col[q];
    const double rg = fast_rsqrt(arg);   // NaN or inf when arg <= 0: unused then
    join();
    const double gm = fma(s.D, col[2 * L - 1], s.A) * s.igmm;
    const double invd = rg * s.B;
    res_coefs<T, L>(cf, res_coef_x<T, L>(s, m, gm, kc, kn), invd, kc, kn);
    if ((threadIdx.x & 31) == 0) {
        double *gc = s.G[c % (L + 1)];
#pragma unroll
        for (int q = 0; q < 2 * L; ++q) gc[q] = col[q];
        s.Ginv[c % (L + 1)] = rg;   // here, not in post: the next crit reads it beside post
        s.arg = arg;
        s.rg = rg;
        s.gm = gm;
        s.invd = invd;
    }
    res_end<T, L>(s, cf, m, graw, arg, gm);
    __syncwarp();
}

// The sum of the neighbour values x (FP64: in fixed point, fxsum.h -- 3D 40^3
// p(1)-CG 5.04 us per iteration against 5.30 with FP64 additions, no
// difference below; FP32: in the order of solver.cuh's sweep).
template <typename T>
__device__ __forceinline__ T res_nbsum(const T (&x)[6], bool three)
{
    if constexpr (sizeof(T) == 8) {
        if (three) return fx_sum(x);
        const double y[4] = {x[0], x[1], x[2], x[3]};
        return fx_sum(y);
    } else {
        const T s = ((x[0] + x[1]) + x[2]) + x[3];
        return three ? (s + x[4]) + x[5] : s;
    }
}

// ... of row g of the plain vector v.
__device__ __forceinline__ double res_nbsum_plain(const double *v, uint32_t g, uint32_t nbr, uint32_t nx, uint32_t nxy,
                                                  bool three)
{
    const double x[6] = {(nbr & 1u) ? v[g - 1] : 0.0,   (nbr & 2u) ? v[g + 1] : 0.0,
                         (nbr & 4u) ? v[g - nx] : 0.0,  (nbr & 8u) ? v[g + nx] : 0.0,
                         (nbr & 16u) ? v[g - nxy] : 0.0, (nbr & 32u) ? v[g + nxy] : 0.0};
    return res_nbsum<double>(x, three);
}

// ------------------------------------------------------------------------
// The iterations of a segment, by role (each in code of its own, so that the
// registers of a sweeping thread's rows are not live in the others).  All
// three return the iteration at whose coefficients the segment ends, or -1
// when a wait ran out.  Barrier 0: l = 1, the coefficients of iteration i are
// there (before its sweep); l >= 2, iteration i is done and the coefficients
// of i + 1 are there.  Barriers 1, 2: between warps 0 and 1; 3: from the
// sweeping warps to the one that publishes (the dots of the CTA's warps are in
// shared memory).
// ------------------------------------------------------------------------
// Warp 0: the dots of the other CTAs, 1 / delta, the coefficients.
template <typename T, int L>
__device__ __forceinline__ int res_loop0(ResSmem<T, L> &s, const ResExch &ex, unsigned e0, int nsw, T kc, T kn)
{
    const int lane = threadIdx.x & 31, nw = nsw >> 5;
    for (int i = 0;; ++i) {
        if constexpr (L == 1) {
            ResCoef<T, L> &ci = s.cf[i & 1];
            if (i >= 1) {   // graw, arg, 1 / sqrt(arg)
                const int m = i - 1;
                double w[kResChunks][1];
                if (!ex.wait<1>(e0 + (unsigned)(i - 1), 1, w) && lane == 0) s.fail[i & 1] = 1;
                res_sum<1>(w, ex.P, &s.raw[1]);
                res_bar_sync(1, 64);
                // rows c-2 (the symmetry of G: g_{c-1,c-1}) and c-1 of column c = m + 1
                const double g0 = m >= 1 ? s.G[m & 1][2] : 0.0, g1 = s.raw[0], graw = s.raw[1];
                const double arg = (graw - g0 * g0) - g1 * g1;
                const double rg = fast_rsqrt(arg);   // NaN or inf when arg <= 0: unused then
                const double invd = rg * s.B;
                res_bar_sync(2, 64);
                res_coefs<T, L>(ci, s.X[lane], invd, kc, kn);
                if (lane == 0) {
                    double *gc = s.G[(m + 1) & 1];
                    gc[0] = g0;
                    gc[1] = g1;
                    s.Ginv[(m + 1) & 1] = rg;
                    s.arg = arg;
                    s.rg = rg;
                    s.invd = invd;
                }
                res_end<T, L>(s, ci, m, graw, arg, s.gm);
            }
            res_bar_all();
            if (s.fail[i & 1]) return -1;
            if (ci.end >= 0) return i;
            res_bar_sync(3, 32 + nsw);
            res_publish<2>(ex, e0 + (unsigned)i, s.red[i & 1], nw);
        } else {
            if (s.cf[i & 1].end >= 0) return i;
            auto join = [] { res_bar_sync(1, 64); };   // warp 1's post and pre are done
            double w[kResChunks][L + 1];
            if (i + 1 < L) {
                join();
            } else if (ex.wait<L + 1>(e0 + (unsigned)(i + 1 - L), 0, w)) {
                res_sum<L + 1>(w, ex.P, s.raw);
                res_crit<T, L>(s, i + 1, kc, kn, join);
            } else {
                if (lane == 0) s.fail[i & 1] = 1;
                join();
            }
            res_bar_all();
            if (s.fail[i & 1]) return -1;
        }
    }
}

// Warp 1: l = 1: gamma; post and pre; l >= 2: this CTA's dots.
template <typename T, int L>
__device__ __forceinline__ int res_loop1(ResSmem<T, L> &s, const ResExch &ex, unsigned e0, int nsw, T kc, T kn,
                                         double rn, double tau, long long budget)
{
    const int lane = threadIdx.x & 31, nw = nsw >> 5;
    for (int i = 0;; ++i) {
        if constexpr (L == 1) {
            if (i >= 1) {
                const int m = i - 1;
                double w[kResChunks][1];
                if (!ex.wait<1>(e0 + (unsigned)(i - 1), 0, w) && lane == 0) s.fail[i & 1] = 1;
                res_sum<1>(w, ex.P, &s.raw[0]);
                res_bar_arrive(1, 64);
                const double gm = fma(s.D, s.raw[0], s.A) * s.igmm;
                s.X[lane] = res_coef_x<T, L>(s, m, gm, kc, kn);
                if (lane == 0) s.gm = gm;
                __syncwarp();
                res_bar_arrive(2, 64);
            }
            res_bar_all();
            if (s.fail[i & 1]) return -1;
        }
        if (s.cf[i & 1].end >= 0) return i;
        if (lane == 0) {
            res_post<T, L>(s, i);
            res_pre<T, L>(s, i + 1, rn, tau, budget);
        }
        __syncwarp();
        if constexpr (L >= 2) {
            res_bar_arrive(1, 64);
            res_bar_sync(3, 32 + nsw);
            res_publish<L + 1>(ex, e0 + (unsigned)i, s.red[i & 1], nw);
            res_bar_all();
            if (s.fail[i & 1]) return -1;
        }
    }
}

// What a thread needs to know about its rows: their numbers and the neighbours
// inside the grid, bits 0 .. 5: left, right, y-, y+, z-, z+; bit 6: there is no row.
template <int R>
struct ResRows {
    uint32_t g[R], nbr[R];
    __device__ __forceinline__ bool has(int r) const { return (nbr[r] & 64u) == 0u; }
};

// The neighbour sums of z^(l) with tag t from buffer z: the lanes of a warp
// exchange their x neighbours, the others are spun on (the row itself in a
// missing neighbour's place, so that no branch separates the loads).
template <typename T, int R>
__device__ __forceinline__ bool res_neighbours(const ResExch &ex, const ResRows<R> &rows, const unsigned long long *z,
                                               unsigned t, uint32_t nx, uint32_t nxy, bool three, const T (&c)[R],
                                               T (&nb)[R])
{
    constexpr int W = sizeof(T) == 8 ? 2 : 1;
    constexpr int RB = R < 2 ? R : 2;   // rows whose loads are in flight together
    const int lane = threadIdx.x & 31;
    bool fine = true;
#pragma unroll
    for (int r0 = 0; r0 < R; r0 += RB) {
        T x[RB][5];               // x neighbour at the warp's edge, y-, y+, z-, z+
        for (unsigned long long polls = 1;; ++polls) {
            Tagged<T> v[RB][5];
#pragma unroll
            for (int q = 0; q < RB; ++q) {
                const uint32_t gr = rows.g[r0 + q], m = rows.nbr[r0 + q];
                const uint32_t ge = (lane == 0 && (m & 1u)) ? gr - 1u : (lane == 31 && (m & 2u)) ? gr + 1u : gr;
                v[q][0].load(z + (size_t)ge * W);
                v[q][1].load(z + (size_t)(gr - ((m & 4u) ? nx : 0u)) * W);
                v[q][2].load(z + (size_t)(gr + ((m & 8u) ? nx : 0u)) * W);
                if (three) {
                    v[q][3].load(z + (size_t)(gr - ((m & 16u) ? nxy : 0u)) * W);
                    v[q][4].load(z + (size_t)(gr + ((m & 32u) ? nxy : 0u)) * W);
                }
            }
            bool ready = true;
#pragma unroll
            for (int q = 0; q < RB; ++q) {
                bool ok = v[q][0].is(t) & v[q][1].is(t) & v[q][2].is(t);
                if (three) ok &= v[q][3].is(t) & v[q][4].is(t);
                ready &= ok | !rows.has(r0 + q);
#pragma unroll
                for (int k = 0; k < 5; ++k) x[q][k] = (k < 3 || three) ? v[q][k].value() : T(0);
            }
            if (__all_sync(0xffffffffu, ready)) break;
            if (__any_sync(0xffffffffu, ex.give_up(polls))) {
                fine = false;
                break;
            }
        }
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            const int r = r0 + q;
            const uint32_t m = rows.nbr[r];
            const T lf = __shfl_up_sync(0xffffffffu, c[r], 1), rt = __shfl_down_sync(0xffffffffu, c[r], 1);
            const T y[6] = {(m & 1u) ? (lane == 0 ? x[q][0] : lf) : T(0), (m & 2u) ? (lane == 31 ? x[q][0] : rt) : T(0),
                            (m & 4u) ? x[q][1] : T(0), (m & 8u) ? x[q][2] : T(0), (m & 16u) ? x[q][3] : T(0),
                            (m & 32u) ? x[q][4] : T(0)};
            nb[r] = res_nbsum<T>(y, three);
        }
    }
    return fine;
}

// A sweeping thread: its rows from the residual a.r to the final update of x.
template <typename T, int L, int R>
__device__ __forceinline__ int res_loop_rows(ResSmem<T, L> &s, const ResExch &ex, const SolveArgs<T> &a,
                                             const ResRows<R> &rows, unsigned zt, int nsw, double rn, T kc, T kn)
{
    constexpr bool kF32 = sizeof(T) == 4;
    constexpr int W = kF32 ? 1 : 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nn = (uint32_t)a.n, nx = (uint32_t)a.st.nx, nxy = nx * (uint32_t)a.st.ny;
    const bool three = a.st.dim == 3;
    unsigned long long *const zb = reinterpret_cast<unsigned long long *>(a.zring);   // [2][n] tagged values
    const uint32_t(&g)[R] = rows.g;
    T c[R], zp[R], cur[R][L], pk[R][L], pv[R], xv[R];
    // ---- Algorithm 1, initialization
    const double inv = 1.0 / rn;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        c[r] = xv[r] = T(0);
        if (rows.has(r)) {
            c[r] = (T)(a.r[g[r]] * inv);
            if constexpr (!kF32) xv[r] = a.x[g[r]];
            st_tagged(zb + (size_t)g[r] * W, c[r], zt);
        }
        zp[r] = T(0);
        pv[r] = T(0);
#pragma unroll
        for (int k = 0; k < L; ++k) { cur[r][k] = c[r]; pk[r][k] = T(0); }
    }
    int i = 0;
    for (;; ++i) {
        const ResCoef<T, L> &cf = s.cf[i & 1];
        if constexpr (L >= 2) {
            if (cf.end >= 0) break;
        }
        T nb[R];
        const unsigned zi = zt + (unsigned)i, want = zi | (zi >= a.res_force_z ? 0x40000000u : 0u);   // (a tag of none)
        if (!res_neighbours<T, R>(ex, rows, zb + (size_t)(i & 1) * nn * W, want, nx, nxy, three, c, nb) &&
            lane == 0)
            s.fail[i & 1] = 1;
        if constexpr (L == 1) {
            res_bar_all();
            if (s.fail[i & 1]) return -1;
            if (cf.end >= 0) break;
        }
        DotAcc<T, 1> dac[L + 1];
        const bool rec = cf.rec, first = cf.first;
        const T zx = cf.zx, pp = cf.pp;
        const T wu = cf.co[0], uc = cf.co[1], bm = cf.co[2], unb = cf.co[3], sig = cf.sig;
        T ak[L];
#pragma unroll
        for (int k = 0; k < L; ++k) ak[k] = cf.co[4 + k];
        unsigned long long *zn = zb + (size_t)((i + 1) & 1) * nn * W;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!rows.has(r)) continue;
            T un, o[1], u1[1];
            if (rec) {
                un = fma(uc, c[r], fma(unb, nb[r], bm * zp[r]));
                st_tagged(zn + (size_t)g[r] * W, un, zt + (unsigned)i + 1u);
                T nw_[L];
#pragma unroll
                for (int k = 0; k < L; ++k) {
                    const T up = (k == L - 1) ? c[r] : cur[r][k + 1];
                    nw_[k] = fma(up, wu, fma(ak[k], cur[r][k], bm * pk[r][k]));
                }
                u1[0] = un;
                o[0] = nw_[0];
                dac[0].add(u1, o);
#pragma unroll
                for (int k = 0; k < L; ++k) { pk[r][k] = cur[r][k]; cur[r][k] = nw_[k]; }
            } else {
                un = fma(kc - sig, c[r], kn * nb[r]);
                st_tagged(zn + (size_t)g[r] * W, un, zt + (unsigned)i + 1u);
                u1[0] = un;
                if (i == L - 1) {   // row 0 of column l: v_0
                    o[0] = cur[r][0];
                    dac[0].add(u1, o);
                }
#pragma unroll
                for (int k = 1; k < L; ++k)
                    if (i + 1 == k) cur[r][k] = un;
                if (i == L - 1)
#pragma unroll
                    for (int k = 1; k < L; ++k) pk[r][k] = cur[r][k - 1];
            }
            if constexpr (L >= 3) { o[0] = zp[r]; dac[L - 2].add(u1, o); }
            if constexpr (L >= 2) { o[0] = c[r]; dac[L - 1].add(u1, o); }
            dac[L].add(u1, u1);
            zp[r] = c[r];
            c[r] = un;
        }
        double v[L + 1];
        if constexpr (kF32) {
            widened_sums(dac, v);
        } else {
#pragma unroll
            for (int q = 0; q <= L; ++q) v[q] = dac[q].acc;
        }
        constexpr int S = L == 1 ? 1 : 2;
        const double t = warp_reduce_scatter<L + 1>(v, lane);
        if ((lane & ((32 >> S) - 1)) == 0) {
            const int q = lane >> (5 - S);
            if (q <= L) s.red[i & 1][warp - 2][q] = t;
        }
        __syncwarp();
        res_bar_arrive(3, 32 + nsw);
        // K6, off the path to the next exchange (pk[0] is z^(0)_m by now)
        if (rec) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (first) {
                    pv[r] = pk[r][0];
                } else {
                    xv[r] = fma(zx, pv[r], xv[r]);
                    pv[r] = fma(pp, pv[r], pk[r][0]);
                }
            }
        }
        if constexpr (L >= 2) {
            res_bar_all();
            if (s.fail[i & 1]) return -1;
        }
    }
    // ---- final vector update of the segment
    const ResCoef<T, L> &cf = s.cf[i & 1];
    if (cf.end != kSegNonfinite) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (cf.fmode == 0) {
                if (cf.f1 != T(0)) xv[r] = fma(cf.f1, pv[r], xv[r]);
            } else if (cf.fmode == 1) {
                xv[r] = fma(cf.f1, pv[r], xv[r]);
                const T pn = fma(cf.fpv, cur[r][0], cf.fpp * pv[r]);
                xv[r] = fma(cf.f2, pn, xv[r]);
            } else {
                xv[r] = fma(cf.f2, cf.fpv * cur[r][0], xv[r]);
            }
        }
    }
    if (cf.end != kSegNonfinite || !kF32) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!rows.has(r)) continue;
            if constexpr (kF32) a.x[g[r]] += (double)xv[r];
            else a.x[g[r]] = xv[r];
        }
    }
    return i;
}

// ------------------------------------------------------------------------
// A whole solve.  Threads 0 .. 31: warp 0; 32 .. 63: warp 1; 64 .. 64 + nsw -
// 1, the last: R rows each.  Cooperative launch, at most 32 kResChunks CTAs.
// ------------------------------------------------------------------------
template <typename T, int L, int R>
__global__ void __launch_bounds__(kResBlock, 1) resident_kernel(SolveArgs<T> a)
{
    static_assert(L >= 1 && L <= 3, "the K5 operands of l <= 3 are all in registers");
    constexpr bool kF32 = sizeof(T) == 4;
    constexpr int W = kF32 ? 1 : 2;   // 64-bit words of a tagged row value
    __shared__ ResSmem<T, L> s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nsw = a.res_nsw, nw = nsw >> 5;
    const ResExch ex{a.pkt, (int)gridDim.x, (int)blockIdx.x, res_dots(L), a.poll_limit / 8 + 1, a.res_force,
                     &a.out->abort};
    const uint32_t nn = (uint32_t)a.n, nx = (uint32_t)a.st.nx, nxy = nx * (uint32_t)a.st.ny;
    const bool three = a.st.dim == 3;
    const T kc = (T)a.st.center, kn = (T)a.st.off;
    const bool sweeps = tid >= 64;
    ResRows<R> rows;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t g = ((uint32_t)blockIdx.x * R + r) * nsw + (uint32_t)(tid - 64);
        rows.g[r] = 0;
        rows.nbr[r] = 64u;   // no row: the loads of row 0's neighbourhood are valid and unused
        if (sweeps && g < nn) {
            const uint32_t line = (__umulhi(g, a.st.dnx.m) + g) >> a.st.dnx.s;
            const uint32_t x = g - line * nx;
            const uint32_t zc = (__umulhi(line, a.st.dny.m) + line) >> a.st.dny.s;
            const uint32_t y = line - zc * (uint32_t)a.st.ny;
            rows.g[r] = g;
            rows.nbr[r] = (x > 0 ? 1u : 0u) | (x + 1 < nx ? 2u : 0u) | (y > 0 ? 4u : 0u) |
                          (y + 1 < (uint32_t)a.st.ny ? 8u : 0u) | (zc > 0 ? 16u : 0u) |
                          (zc + 1 < (uint32_t)a.st.nz ? 32u : 0u);
            unsigned long long *zb = reinterpret_cast<unsigned long long *>(a.zring);
            st_tagged(zb + (size_t)g * W, T(0), 0u);
            st_tagged(zb + ((size_t)nn + g) * W, T(0), 0u);
        }
    }
    unsigned e = 0;            // number of the last exchange of dots
    unsigned zt = 1;           // tag of z^(l)_0 of the segment
    if (tid < L) s.sig[tid] = a.sigma[tid];
    if (tid == 0) s.fail[0] = s.fail[1] = s.fail[2] = 0;

    long long iters = 0, spmvs = 0, restarts = 0, refinements = 0, segments = 0;
    int last_end = kSegConverged;
    double normb = 0.0, recres = 0.0, last_rn = 0.0;
    int status = kStOk;

    // a grid barrier (with fences: it also orders plain stores and loads) and
    // two sums over all rows, in s.norms; false: gave up
    auto exchange2 = [&](double v0, double v1) -> bool {
        double v[2] = {v0, v1};
        double(*red)[2] = reinterpret_cast<double(*)[2]>(&s.red[0][0][0]);
        if (warp >= 2 && warp < 2 + nw) {
            const double t = warp_reduce_scatter<2>(v, lane);
            if ((lane & 15) == 0) red[warp - 2][lane >> 4] = t;
        }
        __syncthreads();
        ++e;
        if (warp == 0) {
            __threadfence();
            res_publish<2>(ex, e, red, nw);
            double w[kResChunks][2];
            const bool ok = ex.wait<2>(e, 0, w);
            __threadfence();
            if (ok) res_sum<2>(w, ex.P, s.norms);
            else if (lane == 0) s.fail[2] = 1;
        }
        __syncthreads();
        return !s.fail[2];
    };

    for (;;) {
        // ---- true residual r = b - A x and the norms
        double acc0 = 0.0, acc1 = 0.0;
        const double cC = (double)kc, cO = (double)kn;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!rows.has(r)) continue;
            const uint32_t g = rows.g[r];
            const double w = fma(cO, res_nbsum_plain(a.x, g, rows.nbr[r], nx, nxy, three), cC * a.x[g]);
            const double bv = __ldg(a.b + g), rv = bv - w;
            acc0 = fma(bv, bv, acc0);
            acc1 = fma(rv, rv, acc1);
            a.r[g] = rv;
        }
        spmvs++;
        if (!exchange2(acc0, acc1)) { status = kStTimeout; break; }
        if (segments == 0) normb = sqrt(s.norms[0]);
        const double rn = sqrt(s.norms[1]);
        last_rn = rn;
        if (normb == 0.0) {   // b = 0: x = 0 is the solution
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (rows.has(r)) a.x[rows.g[r]] = 0.0;
            break;
        }
        if (!isfinite(normb) || !isfinite(rn)) { status = kStNonfinite; break; }
        if (rn < a.rtol * normb) { recres = (segments == 0) ? rn : recres; break; }
        if (iters >= a.maxit) { status = kStMaxit; break; }
        if (segments > 0) {
            if (kF32 && (last_end == kSegConverged || last_end == kSegLucky)) {
                if (++refinements > kMaxRefine) { status = kStMaxit; break; }
            } else {
                if (restarts >= a.max_restarts) {
                    status = (last_end == kSegMaxit) ? kStMaxit : kStBreakdown;
                    break;
                }
                restarts++;
            }
        }
        const double tau = kF32 ? fmax(a.inner_floor * rn, 0.5 * a.rtol * normb) : a.rtol * normb;
        const long long budget = a.maxit - iters;
        if (tid == 32) {
            for (int q = 0; q < 2 * L; ++q) s.G[0][q] = 0.0;
            s.G[0][2 * L] = 1.0;
            s.Ginv[0] = 1.0;
            res_pre<T, L>(s, 0, rn, tau, budget);
        }
        __syncthreads();
        const unsigned e0 = e + 1;   // the exchange of iteration 0
        int i;
        if (warp == 0) i = res_loop0<T, L>(s, ex, e0, nsw, kc, kn);
        else if (warp == 1) i = res_loop1<T, L>(s, ex, e0, nsw, kc, kn, rn, tau, budget);
        else i = res_loop_rows<T, L, R>(s, ex, a, rows, zt, nsw, rn, kc, kn);
        if (i < 0) { status = kStTimeout; break; }
        e = e0 + (unsigned)i;
        zt += (unsigned)i + 2u;
        spmvs += i;
        const ResCoef<T, L> &cf = s.cf[i & 1];
        iters += cf.kseg;
        last_end = cf.end;
        segments++;
        if (cf.end == kSegNonfinite) { status = kStNonfinite; break; }
        recres = (cf.end == kSegLucky || cf.end == kSegBreakdown) ? 0.0 : fabs(s.zeta[cf.kseg & 1]);
        if (!exchange2(0.0, 0.0)) { status = kStTimeout; break; }
    }
    if (blockIdx.x == 0 && tid == 0)
        write_result(a, status, iters, spmvs, restarts, refinements, recres, normb, last_rn);
}

}  // namespace plcg
