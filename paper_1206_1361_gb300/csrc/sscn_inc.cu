// sscn_inc.cu -- Crank-Nicolson sweeps (calclux, calcluy, calcluz, calcnu
// fused) of a complex128 psi whose increment is computed on the FP32 pipe; the
// same for the radial lines of the axially symmetric form, and for a float-float
// psi on grids whose lines are too few or too long for the TMA pipeline.
//
// What bounds the FP64 sweeps.  GB300 issues a warp-wide FP64 instruction every
// 64 clocks per quarter-SM against 2 for a packed FP32 one; a sweep's 12 (real
// time) or 6 - 8 (imaginary time) FP64 instructions a point, 28 with calcnu,
// hold it at a seventh of the HBM bandwidth.
//
// Here psi stays FP64, but the sweep computes the increment 2 Delta of
//     (I - kappa L) Delta = kappa L psi,   u = psi + 2 Delta,
// in float-float arithmetic (sscn_ff.cuh, ~48 significant bits) and adds it to
// the FP64 psi: 4 FP64 instructions a point (2 with drop's MERGE).  |2 Delta| is
// at most 8 kappa max|psi| and about kappa (k h)^2 |psi| on a smooth state, so with kappa up to
// kIncKappaReal / kIncKappaImag the rounding of the increment stays at or below
// that of the FP64 form u = 2 v - psi, which rounds at full size several times.
// calcnu likewise: the nonlinear factor's distance from 1 is computed in
// float-float, the potential factor multiplies in FP64.
//
// Measured (GB300, 256^3 real time, kappa = 0.0125): y and z sweeps 392 -> 226
// us, x with calcnu 889 -> 433 us (8 FP64 instructions a point there: 230 us of
// the FP64 pipe); the y sweep issues about 330 instructions a point, half of
// them integer conversions and addresses, 63 % of the issue slots, with the FP64
// pipe 57 % busy (x: 555, 55 % and 53 %).  Relative L2
// error against FP64 truth, start and here: 64^3 imaginary, 100 steps, 5.3e-15
// and 2.1e-15; 256^3 real, 10 steps, 6.8e-15 and 4.4e-15; 128 x 96 x 80 real at
// kappa = 0.05, 20 steps, 1.5e-14 and 6.6e-15.  In imaginary time the state
// hardly changes from step to step and the rounding repeats:
// at kappa = 0.05 (500 x 384, 40 steps) 2.4e-15 against 1.6e-15, hence the
// smaller kIncKappaImag.  In real time the error moves with kappa through the
// rounding of the coefficients, the same at every step, in both forms; 20 steps,
// mean and largest (e-15), FP64 sweeps and here: kappa 0.004 .. 0.05, 80 x 64 x 50
// 8.7, 12.9 and 5.7, 7.5; 500 x 384 5.6, 10.0 and 4.8, 8.0; kappa 0.05 .. 0.06 8.1,
// 18.4 and 7.3, 9.4; 8.1, 16.5 and 5.0, 6.8.  Imaginary time, kappa 0.004 .. 0.025:
// 2.3, 3.1 and 1.4, 2.0; 1.6, 2.1 and 1.4, 2.0.  (The FP64 truth, dense matrices,
// has an error of 1.4 to 3e-15 itself: see axial_inc.)
//
// The lines are cut and solved as in sscn_split.cu (half sub-lines of at most P
// rows, whole lines in shared memory).  Per row, r_j = kappa mult_j:
//     s_j = psi_{j-1} - 2 psi_j + psi_{j+1}
//     e_j = s_j + r_{j-1} e_{j-1}              forward, from either end
//     g_k = kappa mid_k (s_k + r e_{k-1} + r e_{k+1}),  2 Delta_k = 2 g_k
//     g_j = r_j (e_j + g_{j+1}),               2 Delta_j = 2 g_j
// (Delta = kappa D with (I - kappa L) D = s): the product that carries the back
// substitution to the next row is the increment itself.  A window's rows
// further than `near` rows from the lane's own, whose carry is damped below
// 2^-26 on the way, run in plain FP32.
//
// Conversions go through the bits of the double with integer instructions (the
// FP64 <-> FP32 conversion instructions run on the FP64 pipe).  Values enter
// multiplied by 2^kLift, which puts the full float-float precision at 2^-165
// .. 2^33 (|psi| of 10^9, a cloud of a micrometre in metres, lies below).  A
// block whose largest value lies below 2^-135 (psi is small everywhere, or its
// lines run far outside the cloud) or above 2^33 lifts it to 2^20 instead
// (below 2^-855 as far as the exponents go); outside 2^-940 .. 2^1000, and with
// anything not finite, it sweeps in FP64.  So
// an increment that comes with fewer bits (values below 2^-165) or none (below
// 2^-216) belongs to a value 2^30 or 2^81 times smaller than the largest of the
// block.  (Rows of the x sweep that lie in one warp: of the warp.)  On the ground
// state of the 256^3 quench, whose lines end at 2^-118 and far below, 41 % of
// the rows choose: y 242 us against 228 where psi is nowhere small, x 441
// against 436, a step 910 against 876 (with a constant lift 868 on both, and the
// rows' increments lost).  A usual lift of 2^30, with which more choose, took 257
// and 473 under the profiler; FP64 from 2^-800 down, which the state of a
// float-float run reaches outside its support, 995 against 927 a step.

#include "sscn_ff.cuh"
#include "sscn_rho.cuh"
#include "sscn_split.cuh"

namespace gp {

using namespace gp::sp;
using gp::ff::f2;
using FC = gp::ff::C;

namespace {

constexpr int kIncP = 8;                 // rows a lane
constexpr double kIncKappaReal = 0.06, kIncKappaImag = 0.025;
constexpr int kLift = 90;
constexpr int kIncEnds = 2 * kSplitEnds + 1;

struct IncArgs {
    SplitArgs<double> s;
    int near;                            // window rows in float-float
    FfCoef rinf;                         // r past conv
    FfCoef kmid[kIncEnds];               // kappa mid_k
};

// ------------------------------------------------------------- conversions

// FP64 - FP32 exponent in the high word, of values multiplied by 2^e on the way.
__host__ __device__ constexpr unsigned offset_of(int e) { return (unsigned)(1023 - 127 - e) << 20; }
constexpr unsigned kOff = offset_of(kLift);

// High word from which on a value is too large for a float lifted with off, or not
// finite (with 2^margin to spare).
__host__ __device__ constexpr unsigned most_of(unsigned off, unsigned margin = 0) { return off + ((250u - margin) << 20); }

__device__ __forceinline__ bool too_large(double x, unsigned off)
{
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) >= most_of(off);
}

// 2^e x (off: offset_of(e)) as a float-float pair: hi the nearest float (ties away from zero),
// lo the float nearest the rest.  With x = s m 2^(e-52), m the 53-bit
// significand: hi = s r 2^(e-23), r = (m + 2^28) >> 29, and x - hi = s d
// 2^(e-52), d = m - 2^29 r = ((m + 2^28) mod 2^29) - 2^28.
__device__ __forceinline__ float2 lift(double x, unsigned off)
{
    const unsigned L = (unsigned)__double2loint(x), H = (unsigned)__double2hiint(x);
    const unsigned sign = H & 0x80000000u, L2 = L + 0x10000000u;
    const int E = (int)((H & 0x7fffffffu) - off), E2 = E + (L2 < L ? 1 : 0);
    float hi = __uint_as_float(__funnelshift_l(L2, (unsigned)E2, 3) | sign);
    const int d = (int)(L2 & 0x1fffffffu) - 0x10000000;
    const float ulp = __uint_as_float((((unsigned)(E - (52 << 20)) << 3) & 0x7f800000u) | sign);   // s 2^(e-52)
    float lo = __int2float_rn(d) * ulp;
    if (E < (53 << 20)) lo = 0.f;
    if (E < (1 << 20)) hi = 0.f;
    return f2(hi, lo);
}

// 2^-e x (off: offset_of(e)) as FP64: exact, zero for zero and FP32 denormals.
__device__ __forceinline__ double widen(float x, unsigned off)
{
    const unsigned f = __float_as_uint(x), mag = f & 0x7fffffffu;
    const unsigned H = mag < 0x800000u ? 0u : (mag >> 3) + off;
    return __hiloint2double((int)(H | (f & 0x80000000u)), (int)(f << 29));
}

// 2^-e (hi + lo) as FP64 with one FP64 addition; or (MERGE) with
// none: hi's bits as FP64 bits plus lo, renormalised to at most half an ulp of
// hi, in units of FP64's last place (carries and borrows run through the
// exponent field as they should; below a power of two the place is half as
// large).  MERGE takes about 12 more instructions: for the x sweep, which the
// FP64 pipe bounds.
template <bool MERGE> __device__ __forceinline__ double drop(float h, float l, unsigned off)
{
    if (!MERGE) return widen(h, off) + widen(l, off);
    const float2 z = ff::s_two_sum(h, l);
    const unsigned f = __float_as_uint(z.x), ef = f & 0x7f800000u;
    const float units = __uint_as_float(ef >= (53u << 23) ? (306u << 23) - ef : 0u);      // 2^(52 - e)
    int li = __float2int_rn(z.y * units);
    const int neg = (int)f >> 31;
    li = (li ^ neg) - neg;
    if ((f & 0x7fffffu) == 0u && li < 0) li *= 2;
    const long long b = __double_as_longlong(widen(z.x, off)) + (long long)li;
    return ef == 0u ? 0.0 : __longlong_as_double(b);
}

__device__ __forceinline__ FC lift(double2 p, unsigned off = kOff)
{
    const float2 x = lift(p.x, off), y = lift(p.y, off);
    return FC{f2(x.x, y.x), f2(x.y, y.y)};
}

// p + 2^TIMES z, z lifted
template <int TIMES, bool MERGE> __device__ __forceinline__ double2 plus(double2 p, FC z, unsigned off = kOff)
{
    off += (unsigned)TIMES << 20;
    return make_double2(p.x + drop<MERGE>(z.hi.x, z.lo.x, off), p.y + drop<MERGE>(z.hi.y, z.lo.y, off));
}

__device__ __forceinline__ float4 pack(FC z) { return make_float4(z.hi.x, z.hi.y, z.lo.x, z.lo.y); }
__device__ __forceinline__ FC unpack(float4 v) { return FC{f2(v.x, v.y), f2(v.z, v.w)}; }

// The largest magnitude a lane has seen, as a high word; 1 for an FP64 denormal
// whose high word is zero.
struct Seen {
    unsigned top = 0, low = 0;

    __device__ __forceinline__ void add(double2 p)
    {
        top = max(top, max((unsigned)__double2hiint(p.x) & 0x7fffffffu, (unsigned)__double2hiint(p.y) & 0x7fffffffu));
        low |= (unsigned)__double2loint(p.x) | (unsigned)__double2loint(p.y);
    }
    __device__ __forceinline__ unsigned value() const { return top == 0u && low != 0u ? 1u : top; }
};

// High words between which some lift reaches full precision.
constexpr unsigned kLeast = (1023u - 940u) << 20, kHuge = (1023u + 1000u) << 20;

// The offset that lifts values up to `top` (a high word; 0: all zero), or 0 where
// they go to FP64.  ANY: the largest lift there is below kLeast.
template <int MARGIN, bool ANY = false> __device__ __forceinline__ unsigned offset_for(unsigned top)
{
    constexpr unsigned most = most_of(kOff, MARGIN), tiny = (1023u - 45u - kLift) << 20;
    if (top == 0u || (top >= tiny && top < most)) return kOff;
    if ((!ANY && top < kLeast) || top >= kHuge) return 0u;
    return max((int)(top >> 20) - 127 - 20, 1) << 20;
}

// The offset of the block's lift, from what its lanes have seen; 0: the block
// sweeps in FP64.  One barrier where some lane has seen an ordinary value and
// none a larger one, whatever the others have (a line that ends far outside the
// cloud); another one otherwise.  block_top: zero before.
template <int MARGIN = 0> __device__ __forceinline__ unsigned block_offset(const Seen &seen, unsigned *block_top)
{
    constexpr unsigned most = most_of(kOff, MARGIN), tiny = (1023u - 45u - kLift) << 20;
    unsigned top = seen.value();
    // the barrier counts 1 for a warp with an ordinary value, 31 for one with a larger
    const bool usual = __any_sync(0xffffffffu, top >= tiny && top < most), large = __any_sync(0xffffffffu, top >= most);
    const int votes = __syncthreads_count((threadIdx.x & 31) == 0 ? usual : large);
    static_assert(kSplitThreads / 32 < 31, "the two counts stay apart");
    if (votes > 0 && votes < 31) return kOff;
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(block_top, top);
    __syncthreads();
    return offset_for<MARGIN>(*block_top);
}

// ------------------------------------------------------------------ calcnu

// G of the step, and G 2^(-2 k) as a pair with the offset of values times 2^k: a =
// G |p|^2 is formed as (G 2^(-2 k)) |2^k p|^2 with k from G's exponent, so that
// where the series below serves (|a| < 2^-8) |2^k p| is below 2^-3 whatever the
// units of psi and G, and what underflows belongs to an a below 2^-90.  (With
// psi's own lift, G of a |psi| beyond 10^6 fell among the denormals.)
struct NlScale {
    double G;
    float2 g;
    unsigned off;
};

__device__ __forceinline__ NlScale nl_scale(double G)
{
    const int e = (__double2hiint(G) >> 20) & 0x7ff;
    // 2^(-2 k) G in [1/2, 2); zero and what is not finite as they are
    const int k = e == 0 ? (G == 0.0 ? 0 : -512) : e == 0x7ff ? 0 : (e - 1022) >> 1;
    const double s = __hiloint2double((1023 - k) << 20, 0), g = G * s * s;
    const float h = (float)g;
    return NlScale{G, f2(h, (float)(g - (double)h)), offset_of(k)};
}

// Real time: exp(-i a) p, a = G |p|^2, as p + (exp(-i a) - 1) p with the factor
// from its Taylor series in float-float for |a| < 2^-8 (first dropped terms
// a^6 / 720 and a^7 / 5040 below 2^-57), in FP64 beyond.
__device__ __forceinline__ double2 nonlinear_real(double2 p, const NlScale &s)
{
    const FC z = lift(p, s.off);
    const float2 a = ff::s_mul(s.g, ff::abs2(z));
    if (fabsf(a.x) < 0x1p-8f && !too_large(p.x, s.off) && !too_large(p.y, s.off)) {
        const float q = __fmul_rn(a.x, a.x);
        float qe = fmaf(a.x, a.x, -q);
        qe = fmaf(2.f * a.x, a.y, qe);
        const float2 dr = f2(-0.5f * q, fmaf(q * q, 1.f / 24, -0.5f * qe));
        const float2 di = f2(-a.x, fmaf(a.x * q, fmaf(q, -1.f / 120, 1.f / 6), -a.y));
        const FfCoef D{f2(dr.x, dr.x), f2(dr.y, dr.y), f2(-di.x, di.x), f2(-di.y, di.y)};
        return plus<0, true>(p, ff::cmul(z, D), s.off);
    }
    double cs, sn;
    expmi_small(s.G * fma(p.x, p.x, p.y * p.y), cs, sn);
    return make_double2(fma(cs, p.x, sn * p.y), fma(cs, p.y, -sn * p.x));
}

// Imaginary time: f exp(-a), a = G |p|^2, as f + f (exp(-a) - 1) likewise.
__device__ __forceinline__ double factor_imag(double2 p, double f, const NlScale &s)
{
    const float2 a = ff::s_mul(s.g, ff::abs2(lift(p, s.off)));
    if (fabsf(a.x) < 0x1p-8f && !too_large(p.x, s.off) && !too_large(p.y, s.off)) {
        const float q = __fmul_rn(a.x, a.x);
        float qe = fmaf(a.x, a.x, -q);
        qe = fmaf(2.f * a.x, a.y, qe);
        const float2 d = ff::s_two_sum(-a.x, 0.5f * q);
        const float tail = fmaf(q, fmaf(a.x, -1.f / 120, 1.f / 24) * q, -a.x * q * (1.f / 6));
        const float2 eps = ff::s_norm(f2(d.x, d.y + ((0.5f * qe - a.y) + tail)));
        return fma(f, drop<true>(eps.x, eps.y, offset_of(0)), f);
    }
    return f * expm_small(s.G * fma(p.x, p.x, p.y * p.y));
}

// calcnu at stored point i (MODE 0: c.pyz carries the pending scale).
template <int MODE, bool P3>
__device__ __forceinline__ double2 calcnu_at(double2 p, const Calcnu<double, MODE> &c, int i, double2 p3,
                                             const NlScale &s)
{
    if (MODE == 0) {
        const double f = factor_imag(p, c.pyz.x * c.px[i].x, s);
        return make_double2(p.x * f, p.y * f);
    }
    const double2 w = nonlinear_real(p, s);
    return P3 ? cmulc(w, p3) : cmulc(cmulc(w, c.pyz), c.px[i]);
}

// ------------------------------------------------------------------- solve

// r_t for t = -1 .. conv and the middle rows' kappa mid_k in shared memory.
__host__ __device__ __forceinline__ size_t inc_coef_bytes(int conv) { return (size_t)(conv + 2 + kIncEnds) * sizeof(FfCoef); }

template <int MODE> __device__ __forceinline__ void stage_inc(const IncArgs &A, void *to)
{
    FfCoef *tab = static_cast<FfCoef *>(to);
    const int len = A.s.conv + 2;
    for (int q = threadIdx.x; q < len; q += blockDim.x) {
        FfCoef r = A.rinf;
        if (q == 0) r = ff::expand(0.0, 0.0);
        else if (q <= A.s.conv) {
            const double2 v = ktimes<double, MODE>(A.s.k, A.s.mult[q - 1]);
            r = ff::expand(v.x, v.y);
        }
        tab[q] = r;
    }
    for (int q = threadIdx.x; q < kIncEnds; q += blockDim.x) tab[len + q] = A.kmid[q];
}

// z r: kappa-scaled coefficients are real in imaginary time
template <int MODE> __device__ __forceinline__ FC rtimes(FC z, const FfCoef &r)
{
    return MODE == 0 ? ff::rmul(z, r) : ff::cmul(z, r);
}

template <int MODE> struct IncLane : HalfLine {
    const IncArgs &A;
    const FfCoef *tab;       // stage_inc

    __device__ __forceinline__ IncLane(const IncArgs &args, const void *tables, int seg)
        : HalfLine(args.s.n, args.s.S, args.s.W, seg), A(args), tab(static_cast<const FfCoef *>(tables))
    {
    }
    __device__ __forceinline__ const FfCoef &r(int t) const { return tab[min(t, A.s.conv) + 1]; }

    // Solve.  ld(i): lifted psi at row i (0 at rows 0 and n); out(q, i, g): the
    // row's g (lifted), q its place among the lane's rows (0 .. P -
    // 1 from `first`).  SYNC: a block barrier between the last ld and the first
    // out.  Every thread of the block calls this; `active` marks lanes with a
    // line, pair is the lane distance of a sub-line's halves.
    template <bool SYNC, typename Ld, typename Out>
    __device__ __forceinline__ void solve(bool active, int pair, Ld ld, Out out) const
    {
        FC e = ff::cz(), ev[kIncP], cur = ff::cz(), d0 = ff::cz();
        if (active) {
            int t = ts;
            const int t1 = max(ts, to - A.near);
            if (t < t1) {
                // far rows of the window in FP32
                float2 ee = f2(0.f, 0.f);
                const FC a0 = ld(row(t - 1));
                FC a1 = ld(row(t));
                float2 dd = ff::add(ff::sub(a1.hi, a0.hi), ff::sub(a1.lo, a0.lo));
                for (; t < t1; ++t) {
                    const FC a2 = ld(row(t + 1));
                    const float2 dn = ff::add(ff::sub(a2.hi, a1.hi), ff::sub(a2.lo, a1.lo));
                    const FfCoef &k = r(t - 1);
                    float2 s = ff::sub(dn, dd);
                    s = ff::fma2(ee, k.rh, s);
                    if (MODE != 0) s = ff::fma2(ff::swap(ee), k.ih, s);
                    ee = s;
                    dd = dn;
                    a1 = a2;
                }
                e.hi = ee;
            }
            cur = ld(row(t));
            d0 = ff::sub(cur, ld(row(t - 1)));
            auto rhs = [&](int at) {
                const FC next = ld(row(at + 1)), d1 = ff::sub(next, cur), s = ff::sub(d1, d0);
                cur = next;
                d0 = d1;
                return s;
            };
            for (; t < to; ++t) e = ff::add(rhs(t), rtimes<MODE>(e, r(t - 1)));
            // (coefficients from shared memory for every lane: a separate path
            // with the constants in registers made the warps that hold a line's
            // end run both)
#pragma unroll
            for (int q = 0; q < kIncP; ++q)
                if (to + q <= te) ev[q] = e = ff::add(rhs(to + q), rtimes<MODE>(e, r(to + q - 1)));
        }
        // the carries of both halves meet in the middle row
        const FC c = rtimes<MODE>(e, r(te));
        FC o;
        o.hi.x = __shfl_xor_sync(0xffffffffu, c.hi.x, pair);
        o.hi.y = __shfl_xor_sync(0xffffffffu, c.hi.y, pair);
        o.lo.x = __shfl_xor_sync(0xffffffffu, c.lo.x, pair);
        o.lo.y = __shfl_xor_sync(0xffffffffu, c.lo.y, pair);
        FC g = ff::cz();
        if (active && top) {
            const FC next = ld(row(kt + 1)), s = ff::sub(ff::sub(next, cur), d0);
            g = rtimes<MODE>(ff::add(ff::add(s, c), o), tab[A.s.conv + 2 + mid_at(A.s.S)]);
        }
        if (SYNC) __syncthreads();
        if (active && top) out(kt - to, row(kt), g);
        FC w;
        w.hi.x = __shfl_xor_sync(0xffffffffu, g.hi.x, pair);
        w.hi.y = __shfl_xor_sync(0xffffffffu, g.hi.y, pair);
        w.lo.x = __shfl_xor_sync(0xffffffffu, g.lo.x, pair);
        w.lo.y = __shfl_xor_sync(0xffffffffu, g.lo.y, pair);
        if (!top) g = w;
        if (active) {
#pragma unroll
            for (int q = kIncP - 1; q >= 0; --q)
                if (to + q <= te) {
                    g = rtimes<MODE>(ff::add(ev[q], g), r(to + q));
                    out(q, row(to + q), g);
                }
        }
    }
};

// ------------------------------------------------------------------ radial
//
// The radial operator of the axially symmetric form, rows i = 0 .. m - 1, times
// rho_i / h = i + 1/2, is the difference of the fluxes i (psi_i - psi_{i-1})
// through the faces either side: symmetric, its couplings whole numbers that
// float-float products take exactly.  As above with (face f between a row and
// the one its half came from, f' the face ahead, p the row's coefficient in
// radial_inc_tables):
//     S = f' (psi_{t+1} - psi_t) - f (psi_t - psi_{t-1})
//     e_t = S + f p_{t-1} e_{t-1},   g_k = p_k (S_k + both carries)
//     g_t = p_t (e_t + f' g_{t+1}),  2 Delta_t = 2 g_t
struct RadArgs {
    SplitArgs<double> s;
    int near;
    const float4 *mid;
    double2 *work;
    RadialTables rt;
};

constexpr int kRadialBits = 15;          // S and e are at most 2^15 times psi

__device__ __forceinline__ FC ntimes(FC z, float n) { return ff::lmul(z, f2(n, n), f2(0.f, 0.f)); }
__device__ __forceinline__ FfCoef expand(float4 v) { return FfCoef{f2(v.x, v.x), f2(v.z, v.z), f2(-v.y, v.y), f2(-v.w, v.w)}; }

// both coefficient tables of m rows in shared memory
__host__ __device__ __forceinline__ size_t rad_table_bytes(int m) { return (size_t)2 * (slot_of(m) + 1) * sizeof(float4); }

template <int MODE> struct RadLane : HalfLine {
    const RadArgs &A;
    const float4 *tab;

    __device__ __forceinline__ RadLane(const RadArgs &args, const float4 *tables, int seg)
        : HalfLine(args.s.n, args.s.S, args.s.W, seg), A(args), tab(tables + (top ? 0 : slot_of(m) + 1))
    {
    }
    __device__ __forceinline__ float face(int t) const { return (float)(top ? t : m - t); }
    __device__ __forceinline__ FfCoef p(int t) const
    {
        t = max(t, 0);                   // (before the first row: its carry is zero)
        return expand(tab[slot_of(top ? t : m - 1 - t)]);
    }

    // As IncLane::solve<true>.
    template <typename Ld, typename Out> __device__ __forceinline__ void solve(bool active, Ld ld, Out out) const
    {
        FC e = ff::cz(), ev[kIncP], cur = ff::cz(), d0 = ff::cz();
        const float f0 = face(to), ahead = top ? 1.f : -1.f;       // the faces in the direction of t
        if (active) {
            int t = ts;
            const int t1 = max(ts, to - A.near);
            if (t < t1) {
                float2 ee = f2(0.f, 0.f);
                const FC a0 = ld(row(t - 1));
                FC a1 = ld(row(t));
                float f = face(t);
                float2 dd = ff::mul(f2(f, f), ff::add(ff::sub(a1.hi, a0.hi), ff::sub(a1.lo, a0.lo)));
                for (; t < t1; ++t) {
                    const FC a2 = ld(row(t + 1));
                    const float fn = face(t + 1);
                    const float2 dn = ff::mul(f2(fn, fn), ff::add(ff::sub(a2.hi, a1.hi), ff::sub(a2.lo, a1.lo)));
                    const FfCoef k = p(t - 1);
                    const float2 q = ff::mul(f2(f, f), ee);
                    float2 s = ff::sub(dn, dd);
                    s = ff::fma2(q, k.rh, s);
                    if (MODE != 0) s = ff::fma2(ff::swap(q), k.ih, s);
                    ee = s;
                    dd = dn;
                    a1 = a2;
                    f = fn;
                }
                e.hi = ee;
            }
            cur = ld(row(t));
            d0 = ntimes(ff::sub(cur, ld(row(t - 1))), face(t));
            auto rhs = [&](int at, float f) {
                const FC next = ld(row(at + 1)), d1 = ntimes(ff::sub(next, cur), f), s = ff::sub(d1, d0);
                cur = next;
                d0 = d1;
                return s;
            };
            for (float f = face(t); t < to; ++t, f += ahead)
                e = ff::add(rhs(t, f + ahead), ntimes(rtimes<MODE>(e, p(t - 1)), f));
#pragma unroll
            for (int q = 0; q < kIncP; ++q)
                if (to + q <= te)
                    ev[q] = e = ff::add(rhs(to + q, fmaf(q + 1, ahead, f0)),
                                        ntimes(rtimes<MODE>(e, p(to + q - 1)), fmaf(q, ahead, f0)));
        }
        const FC c = ntimes(rtimes<MODE>(e, p(te)), face(kt));
        FC o;
        o.hi.x = __shfl_xor_sync(0xffffffffu, c.hi.x, 1);
        o.hi.y = __shfl_xor_sync(0xffffffffu, c.hi.y, 1);
        o.lo.x = __shfl_xor_sync(0xffffffffu, c.lo.x, 1);
        o.lo.y = __shfl_xor_sync(0xffffffffu, c.lo.y, 1);
        FC g = ff::cz();
        if (active && top) {
            const FC next = ld(row(kt + 1)), s = ff::sub(ntimes(ff::sub(next, cur), face(kt + 1)), d0);
            g = rtimes<MODE>(ff::add(ff::add(s, c), o), expand(__ldg(A.mid + kt)));
        }
        __syncthreads();
        if (active && top) out(row(kt), g);
        FC w;
        w.hi.x = __shfl_xor_sync(0xffffffffu, g.hi.x, 1);
        w.hi.y = __shfl_xor_sync(0xffffffffu, g.hi.y, 1);
        w.lo.x = __shfl_xor_sync(0xffffffffu, g.lo.x, 1);
        w.lo.y = __shfl_xor_sync(0xffffffffu, g.lo.y, 1);
        if (!top) g = w;
        if (active) {
#pragma unroll
            for (int q = kIncP - 1; q >= 0; --q)
                if (to + q <= te) {
                    g = rtimes<MODE>(ff::add(ev[q], ntimes(g, fmaf(q + 1, ahead, f0))), p(to + q));
                    out(row(to + q), g);
                }
        }
    }
};

// ----------------------------------------------------------------- kernels

// A lane's points once more, with another lift: i = first, first + step, ... < end of
// a contiguous row, to row i + shift of the tile; all loads in flight.  (Functions of
// their own: inlined, they took registers from the kernels, which rarely come here.)
__noinline__ __device__ void lift_again(const double2 *row, float4 *tile, int first, int step, int end, int shift, unsigned off)
{
    double2 v[kIncP];
#pragma unroll
    for (int b = 0; b < kIncP; ++b)
        if (first + b * step < end) v[b] = row[first + b * step];
#pragma unroll
    for (int b = 0; b < kIncP; ++b)
        if (first + b * step < end) tile[slot_of(first + b * step + shift)] = pack(lift(v[b], off));
}

// The same for the rows row, row + dir, ... row + dir last of a strided line.
__noinline__ __device__ void lift_again(const double2 *line, long long stride, float4 *tile, int XL, int row, int dir, int last,
                                        unsigned off)
{
    double2 p[kIncP];
#pragma unroll
    for (int q = 0; q < kIncP; ++q)
        if (q <= last) p[q] = line[(row + q * dir) * stride];
#pragma unroll
    for (int q = 0; q < kIncP; ++q)
        if (q <= last) tile[slot_of(row + q * dir) * XL] = pack(lift(p[q], off));
}

// Resident blocks the kernels are compiled for: 3 of 256 threads (80 registers
// a thread), or 2 of 512 (64; lines of more than 1024 rows: the z sweep of an
// axial 1024 x 2048 took 62 us with one, 52 with two).
template <int THREADS> constexpr int kMinBlocks = THREADS == 256 ? 3 : 2;

// x sweep: as k_split_x, thread (row, seg) moving the row's points seg, seg + 2 S,
// ...  A point's calcnu goes back to memory and is read again (from L1 or L2)
// when its increment is there: kept in registers, it cost a third of the
// resident warps.
template <int MODE, bool NL, bool P3, int THREADS>
__global__ void __launch_bounds__(THREADS, kMinBlocks<THREADS>) k_inc_x(const __grid_constant__ IncArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ NlScale nl_of_step;
    __shared__ unsigned block_top;
    if (threadIdx.x == 0) block_top = 0u;
    const SplitArgs<double> &a = A.s;
    const int n = a.n, pitch = slot_of(n) + 1;
    unsigned char *coef = smem_raw, *coef64 = coef + inc_coef_bytes(a.conv);
    Calcnu<double, MODE> *row_nl = reinterpret_cast<Calcnu<double, MODE> *>(coef64 + coef_bytes<double>(a.conv));
    float4 *tile = reinterpret_cast<float4 *>(row_nl + a.per);
    const int line0 = blockIdx.x * a.per;
    const int rows = min(a.per, a.lines_a * a.lines_b - line0);
    const int lanes = 2 * a.S;
    const int q = threadIdx.x / lanes, seg = threadIdx.x - q * lanes;
    const bool active = q < rows;
    const int at = (active ? q : 0) * pitch;
    double2 *row = a.psi + (long long)(line0 + (active ? q : 0)) * n;
    // (tables and set-up before the wait for the kernel before this one)
    stage_inc<MODE>(A, coef);
    for (int r = threadIdx.x; r < a.per; r += blockDim.x)
        tile[r * pitch] = tile[r * pitch + slot_of(n)] = make_float4(0.f, 0.f, 0.f, 0.f);
    pdl_wait();
    double2 v[kIncP], f3[NL && P3 ? kIncP : 1];
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = 1 + seg + b * lanes;
            if (i < n) {
                v[b] = row[i];
                if constexpr (NL && P3) f3[b] = a.p3[(long long)(line0 + q) * n + i];
            }
        }
    }
    if (NL && threadIdx.x == 0) {
        const double G = a.sg.value(), sc = MODE == 0 && a.scale ? *a.scale : 1.0;
        nl_of_step = nl_scale(G * sc * sc);
    }
    if (NL && !P3)
        for (int r = threadIdx.x; r < rows; r += blockDim.x) {
            const int L = line0 + r;
            row_nl[r].setup(a.px, a.py, a.pz, nullptr, nullptr, nullptr, L % a.lines_a, L / a.lines_a, 0.0, a.scale);
        }
    if (NL) __syncthreads();                 // row_nl, G
    Seen seen;
    if (active) {
        const NlScale ns = NL ? nl_of_step : NlScale{};
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = 1 + seg + b * lanes;
            if (i < n) {
                if constexpr (NL) {
                    v[b] = calcnu_at<MODE, P3>(v[b], row_nl[P3 ? 0 : q], i, f3[P3 ? b : 0], ns);
                    row[i] = v[b];
                }
                seen.add(v[b]);
            }
        }
    }
    const int own = active ? seg : (threadIdx.x & 1);
    // rows that lie in one warp each take its lift, without a vote of the block,
    // which still sweeps in FP64 where all of it is below kLeast
    const bool in_warp = 32 % lanes == 0;
    const unsigned top = in_warp ? __reduce_max_sync(0xffffffffu, seen.value()) : 0u;
    unsigned off = offset_for<0, true>(top);
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b)
            if (1 + seg + b * lanes < n) tile[at + slot_of(1 + seg + b * lanes)] = pack(lift(v[b], off ? off : kOff));
    }
    bool fp64;
    if (in_warp) {
        // the barrier counts 1 for a warp that a lift serves, 31 for one it does not
        const int votes = __syncthreads_count((threadIdx.x & 31) == 0 ? top >= kLeast && top < kHuge : top >= kHuge);
        fp64 = votes >= 31 || (votes == 0 && __syncthreads_or(top != 0u));
    } else {
        off = block_offset(seen, &block_top);
        fp64 = off == 0u;
    }
    if (fp64) {
        double2 *t64 = reinterpret_cast<double2 *>(tile);
        stage_coefs<MODE>(a, coef64);
        if (active)
            for (int i = 1 + seg; i < n; i += lanes) t64[at + slot_of(i)] = row[i];
        __syncthreads();
        const Share<kFp64, MODE> lane(a, coef64, own);
        lane.template solve<kIncP, true>(
            active, 1, [&](int i) { return t64[at + slot_of(i)]; }, 0, 0,
            [&](int i, double2 u) { t64[at + slot_of(i)] = u; });
        __syncthreads();
        if (active)
            for (int i = 1 + seg; i < n; i += lanes) row[i] = t64[at + slot_of(i)];
        return;
    }
    if (!in_warp && off != kOff) {
        if (active) lift_again(row, tile + at, 1 + seg, lanes, n, 0, off);
        __syncthreads();
    }
    const IncLane<MODE> lane(A, coef, own);
    lane.template solve<true>(
        active, 1, [&](int i) { return unpack(tile[at + slot_of(i)]); },
        [&](int, int i, FC g) { tile[at + slot_of(i)] = pack(g); });
    __syncthreads();
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = 1 + seg + b * lanes;
            if (i < n) row[i] = plus<1, true>(row[i], unpack(tile[at + slot_of(i)]), off);
        }
    }
}

// y / z sweep: as k_split_yz; a lane reads the FP64 values of its rows again
// (from L1 or L2) when it adds the increments.  Without calcnu the lift's offset
// waits in shared memory: a register for it spilled (256^3 real time 880 us a
// step with it, 876 so, 872 with a constant lift).
template <int MODE, bool NORM, bool NLOUT, bool P3, int THREADS>
__global__ void __launch_bounds__(THREADS, kMinBlocks<THREADS>) k_inc_yz(const __grid_constant__ IncArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[32];
    __shared__ NlScale nl_of_step;
    __shared__ volatile unsigned lift_off;
    __shared__ unsigned block_top;
    if (threadIdx.x == 0) {
        lift_off = kOff;
        block_top = 0u;
    }
    const SplitArgs<double> &a = A.s;
    unsigned char *coef = smem_raw, *coef64 = coef + inc_coef_bytes(a.conv);
    float4 *tile = reinterpret_cast<float4 *>(coef64 + coef_bytes<double>(a.conv));
    const int n = a.n, XL = a.per;
    const int xl = threadIdx.x & (XL - 1), seg = threadIdx.x / XL;
    const int la = blockIdx.x * XL + xl, lb = blockIdx.y;
    const bool active = la < a.lines_a && seg < 2 * a.S;
    const IncLane<MODE> lane(A, coef, seg < 2 * a.S ? seg : (seg & 1));
    const long long base = active ? (long long)la * a.stride_a + (long long)lb * a.stride_b : 0;
    double2 *line = a.psi + base;
    stage_inc<MODE>(A, coef);
    pdl_wait();
    if (NLOUT && threadIdx.x == 0) nl_of_step = nl_scale(a.sg.value());
    auto at_of = [&](int i) { return slot_of(i) * XL + xl; };
    Seen seen;
    if (active) {
        double2 p[kIncP];
#pragma unroll
        for (int q = 0; q < kIncP; ++q)
            if (lane.first + q <= lane.last) p[q] = line[(long long)lane.row(lane.first + q) * a.pstride];
#pragma unroll
        for (int q = 0; q < kIncP; ++q)
            if (lane.first + q <= lane.last) {
                seen.add(p[q]);
                tile[at_of(lane.row(lane.first + q))] = pack(lift(p[q]));
            }
        if (seg == 0) tile[at_of(0)] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (seg == 1) tile[at_of(n)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const unsigned off = block_offset(seen, &block_top);
    Calcnu<double, MODE> nl{};
    const NlScale ns = NLOUT ? nl_of_step : NlScale{};
    if (NLOUT && !P3 && active) nl.setup(a.px, a.py, a.pz, nullptr, nullptr, nullptr, la, lb, 0.0, nullptr);
    double acc = 0.0;
    auto finish = [&](int i, double2 u) {
        const long long at = (long long)i * a.pstride;
        if constexpr (NLOUT) {
            double2 f = make_double2(0.0, 0.0);
            if constexpr (P3) f = a.p3[base + at];
            u = calcnu_at<MODE, P3>(u, nl, i, f, ns);
        }
        line[at] = u;
        if (NORM) acc = fma(u.x, u.x, fma(u.y, u.y, acc));
    };
    if (off == 0u) {
        double2 *t64 = reinterpret_cast<double2 *>(tile);
        stage_coefs<MODE>(a, coef64);
        if (active) {
#pragma unroll
            for (int q = 0; q < kIncP; ++q)
                if (lane.first + q <= lane.last) {
                    const int i = lane.row(lane.first + q);
                    t64[at_of(i)] = line[(long long)i * a.pstride];
                }
        }
        __syncthreads();
        const Share<kFp64, MODE> lane64(a, coef64, seg < 2 * a.S ? seg : (seg & 1));
        lane64.template solve<kIncP, false>(
            active, XL, [&](int i) { return t64[at_of(i)]; }, 0, 0, finish);
    } else {
        if (off != kOff) {
            if (threadIdx.x == 0) lift_off = off;
            if (active) lift_again(line, a.pstride, tile + xl, XL, lane.row(lane.first), lane.top ? 1 : -1, lane.last - lane.first, off);
            __syncthreads();
        }
        lane.template solve<false>(
            active, XL, [&](int i) { return unpack(tile[at_of(i)]); },
            [&](int, int i, FC g) { finish(i, plus<1, false>(line[(long long)i * a.pstride], g, NLOUT ? off : lift_off)); });
    }
    if (NORM) {
        if (a.lw && active) acc *= a.lw[la];
        block_partial(active ? acc : 0.0, red, &a.partials[(long long)blockIdx.y * gridDim.x + blockIdx.x]);
    }
}

// The float-float form (psi itself a pair): as k_inc_x and k_inc_yz, without the
// conversions.  Nothing here is too large for the lifted form's range that calcnu
// or the norm, which square psi in FP32, would not lose as well.
struct FfIncArgs {
    IncArgs i;
    const FfCoef *px;
};

__device__ __forceinline__ FC plus_twice(FC p, FC g)
{
    const float2 two = f2(2.f, 2.f);
    return ff::norm(ff::add(p, FC{ff::mul(two, g.hi), ff::mul(two, g.lo)}));
}

template <int MODE, bool NL, int THREADS>
__global__ void __launch_bounds__(THREADS, kMinBlocks<THREADS>) k_ffinc_x(const __grid_constant__ FfIncArgs F)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const IncArgs &A = F.i;
    const SplitArgs<double> &a = A.s;
    const int n = a.n, pitch = slot_of(n) + 1;
    ff::FfRow<MODE> *row_nl = reinterpret_cast<ff::FfRow<MODE> *>(smem_raw + inc_coef_bytes(a.conv));
    static_assert(sizeof(ff::FfRow<MODE>) <= sizeof(Calcnu<double, 0>), "the plan's bytes a row");
    float4 *tile = reinterpret_cast<float4 *>(row_nl + a.per);
    const int line0 = blockIdx.x * a.per;
    const int rows = min(a.per, a.lines_a * a.lines_b - line0);
    const int lanes = 2 * a.S;
    const int q = threadIdx.x / lanes, seg = threadIdx.x - q * lanes;
    const bool active = q < rows;
    const int at = (active ? q : 0) * pitch;
    float4 *row = reinterpret_cast<float4 *>(a.psi) + (long long)(line0 + (active ? q : 0)) * n;
    stage_inc<MODE>(A, smem_raw);
    for (int r = threadIdx.x; r < a.per; r += blockDim.x)
        tile[r * pitch] = tile[r * pitch + slot_of(n)] = make_float4(0.f, 0.f, 0.f, 0.f);
    pdl_wait();
    float4 v[kIncP];
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = 1 + seg + b * lanes;
            if (i < n) v[b] = row[i];
        }
    }
    if (NL) {
        for (int r = threadIdx.x; r < rows; r += blockDim.x) {
            const int L = line0 + r;
            row_nl[r].setup(a.py[L % a.lines_a], a.pz[L / a.lines_a], a.sg.value(),
                            MODE == 0 && a.scale ? *a.scale : 1.0);
        }
        __syncthreads();
    }
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = 1 + seg + b * lanes;
            if (i < n) {
                if constexpr (NL) {
                    v[b] = pack(row_nl[q].apply(unpack(v[b]), F.px[i]));
                    row[i] = v[b];
                }
                tile[at + slot_of(i)] = v[b];
            }
        }
    }
    __syncthreads();
    const IncLane<MODE> lane(A, smem_raw, active ? seg : (threadIdx.x & 1));
    lane.template solve<true>(
        active, 1, [&](int i) { return unpack(tile[at + slot_of(i)]); },
        [&](int, int i, FC g) { tile[at + slot_of(i)] = pack(g); });
    __syncthreads();
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = 1 + seg + b * lanes;
            if (i < n) row[i] = pack(plus_twice(unpack(row[i]), unpack(tile[at + slot_of(i)])));
        }
    }
}

template <int MODE, bool NORM, int THREADS>
__global__ void __launch_bounds__(THREADS, kMinBlocks<THREADS>) k_ffinc_yz(const __grid_constant__ FfIncArgs F)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[32];
    const IncArgs &A = F.i;
    const SplitArgs<double> &a = A.s;
    float4 *tile = reinterpret_cast<float4 *>(smem_raw + inc_coef_bytes(a.conv));
    const int n = a.n, XL = a.per;
    const int xl = threadIdx.x & (XL - 1), seg = threadIdx.x / XL;
    const int la = blockIdx.x * XL + xl, lb = blockIdx.y;
    const bool active = la < a.lines_a && seg < 2 * a.S;
    const IncLane<MODE> lane(A, smem_raw, seg < 2 * a.S ? seg : (seg & 1));
    float4 *line = reinterpret_cast<float4 *>(a.psi) + (active ? (long long)la * a.stride_a + (long long)lb * a.stride_b : 0);
    stage_inc<MODE>(A, smem_raw);
    pdl_wait();
    auto at_of = [&](int i) { return slot_of(i) * XL + xl; };
    if (active) {
        float4 p[kIncP];
#pragma unroll
        for (int q = 0; q < kIncP; ++q)
            if (lane.first + q <= lane.last) p[q] = line[(long long)lane.row(lane.first + q) * a.pstride];
#pragma unroll
        for (int q = 0; q < kIncP; ++q)
            if (lane.first + q <= lane.last) tile[at_of(lane.row(lane.first + q))] = p[q];
        if (seg == 0) tile[at_of(0)] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (seg == 1) tile[at_of(n)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    float2 acc = f2(0.f, 0.f);
    lane.template solve<false>(
        active, XL, [&](int i) { return unpack(tile[at_of(i)]); },
        [&](int, int i, FC g) {
            const FC u = plus_twice(unpack(tile[at_of(i)]), g);
            line[(long long)i * a.pstride] = pack(u);
            if (NORM) acc = ff::s_add(acc, ff::abs2(u));
        });
    if (NORM)
        block_partial(active ? ff::join(acc) : 0.0, red, &a.partials[(long long)blockIdx.y * gridDim.x + blockIdx.x]);
}

// Radial sweep: as k_inc_x (NL), stored point i of a line being row i + 1.
// Measured at 1024 x 2048, real time: 73 us (the segmented windows, with calcnu
// as a pass of its own: 175).  The potential's two complex products, 8 FP64
// instructions a point, hold the FP64 pipe 27 us of it; the rest is issue slots
// and the latency of blocks of two lines (three resident an SM, next to 36 KB of
// coefficients each).
template <int MODE, int THREADS>
__global__ void __launch_bounds__(THREADS, kMinBlocks<THREADS>) k_inc_rho(const __grid_constant__ RadArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ NlScale nl_of_step;
    __shared__ unsigned block_top;
    if (threadIdx.x == 0) block_top = 0u;
    const SplitArgs<double> &a = A.s;
    const int n = a.n, m = n - 1, pitch = slot_of(n) + 1;
    float4 *coef = reinterpret_cast<float4 *>(smem_raw);
    Calcnu<double, MODE> *row_nl = reinterpret_cast<Calcnu<double, MODE> *>(smem_raw + rad_table_bytes(m));
    float4 *tile = reinterpret_cast<float4 *>(row_nl + a.per);
    const int line0 = blockIdx.x * a.per;
    const int rows = min(a.per, a.lines_a - line0);
    const int lanes = 2 * a.S;
    const int q = threadIdx.x / lanes, seg = threadIdx.x - q * lanes;
    const bool active = q < rows;
    const int at = (active ? q : 0) * pitch;
    double2 *row = a.psi + (long long)(line0 + (active ? q : 0)) * m;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        coef[slot_of(i)] = A.rt.inc_top[i];
        coef[slot_of(m) + 1 + slot_of(i)] = A.rt.inc_bot[i];
    }
    for (int r = threadIdx.x; r < a.per; r += blockDim.x)
        tile[r * pitch] = tile[r * pitch + slot_of(n)] = make_float4(0.f, 0.f, 0.f, 0.f);
    pdl_wait();
    double2 v[kIncP];
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = seg + b * lanes;
            if (i < m) v[b] = row[i];
        }
    }
    if (threadIdx.x == 0) {
        const double G = a.sg.value(), sc = MODE == 0 && a.scale ? *a.scale : 1.0;
        nl_of_step = nl_scale(G * sc * sc);
    }
    for (int r = threadIdx.x; r < rows; r += blockDim.x)
        row_nl[r].setup(a.px, a.py, a.pz, nullptr, nullptr, nullptr, line0 + r, 0, 0.0, a.scale);
    __syncthreads();                         // row_nl, G
    Seen seen;
    if (active) {
        const NlScale ns = nl_of_step;
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = seg + b * lanes;
            if (i < m) {
                v[b] = calcnu_at<MODE, false>(v[b], row_nl[q], i, make_double2(0.0, 0.0), ns);
                row[i] = v[b];
                seen.add(v[b]);
                tile[at + slot_of(i + 1)] = pack(lift(v[b]));
            }
        }
    }
    const unsigned off = block_offset<kRadialBits>(seen, &block_top);
    if (off == 0u) {
        const long long base = (long long)(line0 + (active ? q : 0)) * m;
        solve_rho<MODE>(a.psi + base, A.work + base, A.rt, m, active && seg < 2, seg == 0, 1,
                        [](double2 p, int) { return p; });
        return;
    }
    if (off != kOff) {
        if (active) lift_again(row, tile + at, seg, lanes, m, 1, off);
        __syncthreads();
    }
    const RadLane<MODE> lane(A, coef, active ? seg : (threadIdx.x & 1));
    lane.solve(active, [&](int i) { return unpack(tile[at + slot_of(i)]); },
               [&](int i, FC g) { tile[at + slot_of(i)] = pack(g); });
    __syncthreads();
    if (active) {
#pragma unroll
        for (int b = 0; b < kIncP; ++b) {
            const int i = seg + b * lanes;
            if (i < m) row[i] = plus<1, true>(row[i], unpack(tile[at + slot_of(i + 1)]), off);
        }
    }
}

IncArgs inc_args(const SplitPlan &p, int mode, void *psi, const AxisTables &ax, const SweepGeom &g,
                 const NonlinArgs *nl, const Partials *norm_out)
{
    IncArgs a{};
    a.s = split_args<kFp64>(p, mode, psi, ax, g, nl, norm_out);
    a.rinf = ff_expand(a.s.rinf);
    for (int q = 0; q < kIncEnds; ++q) {
        const double2 f = a.s.mid[q];
        a.kmid[q] = ff_expand(mode == 0 ? make_double2(a.s.k * f.x, 0.0) : make_double2(-a.s.k * f.y, a.s.k * f.x));
    }
    // rows nearer than this reach the lane's own damped by less than 2^-26
    const double r = std::hypot(a.s.rinf.x, a.s.rinf.y);
    a.near = 1;
    for (double q = r; q >= 0x1p-26; q *= r) ++a.near;
    return a;
}

template <int MODE, bool NL, bool P3> cudaError_t go_x(const SplitPlan &p, const IncArgs &a, cudaStream_t st)
{
    auto kern = p.threads <= 256 ? k_inc_x<MODE, NL, P3, 256> : k_inc_x<MODE, NL, P3, kSplitThreads>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(p.after, kern, p.grid_x, p.threads, p.smem, st, a);
}

template <int MODE, bool NORM, bool NLOUT, bool P3>
cudaError_t go_yz(const SplitPlan &p, const IncArgs &a, cudaStream_t st)
{
    auto kern = p.threads <= 256 ? k_inc_yz<MODE, NORM, NLOUT, P3, 256> : k_inc_yz<MODE, NORM, NLOUT, P3, kSplitThreads>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(p.after, kern, dim3(p.grid_x, p.grid_y), p.threads, p.smem, st, a);
}

}  // namespace

cudaError_t launch_sweep_ffinc(const SplitPlan &p, int mode, void *psi, const AxisTables &ax, const SweepGeom &g,
                               const FfNonlin *nl, const Partials *norm_out, cudaStream_t st)
{
    if (p.x ? norm_out != nullptr : nl != nullptr) return cudaErrorInvalidValue;
    FfIncArgs a{};
    a.i = inc_args(p, mode, psi, ax, g, nullptr, norm_out);
    if (nl) {
        a.px = nl->px;
        a.i.s.py = nl->py;
        a.i.s.pz = nl->pz;
        a.i.s.sg = nl->g;
        a.i.s.scale = nl->scale;
    }
    const bool small = p.threads <= 256;
    void (*kern)(const FfIncArgs);
#define GP_PICK(K, M, B) (small ? K<M, B, 256> : K<M, B, kSplitThreads>)
    if (p.x && mode == 0) kern = nl ? GP_PICK(k_ffinc_x, 0, true) : GP_PICK(k_ffinc_x, 0, false);
    else if (p.x) kern = nl ? GP_PICK(k_ffinc_x, 1, true) : GP_PICK(k_ffinc_x, 1, false);
    else if (mode == 0) kern = norm_out ? GP_PICK(k_ffinc_yz, 0, true) : GP_PICK(k_ffinc_yz, 0, false);
    else kern = norm_out ? GP_PICK(k_ffinc_yz, 1, true) : GP_PICK(k_ffinc_yz, 1, false);
#undef GP_PICK
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(p.after, kern, dim3(p.grid_x, p.grid_y), p.threads, p.smem, st, a);
}

bool rho_inc_plan(const RadialTables &rt, int nr, int nz, SplitPlan &p)
{
    p = SplitPlan{};
    if (rt.win < 1 || rt.near < 1 || rt.kre > kIncKappaImag || rt.kim > kIncKappaReal) return false;
    const size_t tables = rad_table_bytes(nr);
    const size_t row = (size_t)(slot_of(nr + 1) + 1) * sizeof(float4) + sizeof(Calcnu<double, 0>);
    p.P = kIncP;
    p.S = (nr + 2 * kIncP - 1) / (2 * kIncP);
    p.W = rt.win + 1;
    p.x = p.increment = p.after = true;
    const int lanes = 2 * p.S;
    if (lanes > kSplitThreads || tables + row > kSplitSmem) return false;
    // as the x sweep: about 256 lanes and at most 64 KB of rows
    int per = lanes >= 256 ? 1 : 256 / lanes;
    while (per > 1 && per * row > 64 * 1024) --per;
    if (nz < kSms * per) per = (nz + kSms - 1) / kSms;
    p.per = per;
    p.smem = tables + per * row;
    p.grid_x = (unsigned)((nz + per - 1) / per);
    p.grid_y = 1;
    p.threads = (per * lanes + 31) / 32 * 32;
    return true;
}

cudaError_t launch_sweep_rho_inc(const SplitPlan &p, int mode, void *psi, void *work, const RadialTables &rt,
                                 int nr, int nz, const NonlinArgs &nl, cudaStream_t st)
{
    RadArgs a{};
    a.s.psi = static_cast<double2 *>(psi);
    a.s.n = nr + 1;
    a.s.S = p.S;
    a.s.W = p.W;
    a.s.per = p.per;
    a.s.lines_a = nz;
    a.s.px = nl.px;
    a.s.py = nl.py;
    a.s.pz = nl.pz;
    a.s.sg = nl.g;
    a.s.scale = nl.scale;
    a.near = rt.near + 1;
    a.mid = rt.inc_mid;
    a.work = static_cast<double2 *>(work);
    a.rt = rt;
    auto kern = p.threads <= 256 ? (mode == 0 ? k_inc_rho<0, 256> : k_inc_rho<1, 256>)
                                 : (mode == 0 ? k_inc_rho<0, kSplitThreads> : k_inc_rho<1, kSplitThreads>);
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(p.after, kern, p.grid_x, p.threads, p.smem, st, a);
}

bool inc_applies(const AxisTables &ax) { return ax.kre <= kIncKappaImag && ax.kim <= kIncKappaReal; }

size_t inc_extra_smem(int conv) { return inc_coef_bytes(conv); }

cudaError_t launch_sweep_inc(const SplitPlan &p, int mode, void *psi, const AxisTables &ax, const SweepGeom &g,
                             const NonlinArgs *nl, bool nlout, const Partials *norm_out, cudaStream_t st)
{
    const IncArgs a = inc_args(p, mode, psi, ax, g, nl, norm_out);
    const bool p3 = a.s.p3 != nullptr, norm = norm_out != nullptr;
    if (p.x) {
        if (nlout || norm || (p3 && mode == 0)) return cudaErrorInvalidValue;
        if (!nl) return mode == 0 ? go_x<0, false, false>(p, a, st) : go_x<1, false, false>(p, a, st);
        if (mode == 0) return go_x<0, true, false>(p, a, st);
        return p3 ? go_x<1, true, true>(p, a, st) : go_x<1, true, false>(p, a, st);
    }
    if ((nl && !nlout) || (norm && (mode == 1 || nlout)) || (nlout && mode == 0)) return cudaErrorInvalidValue;
    if (mode == 0) return norm ? go_yz<0, true, false, false>(p, a, st) : go_yz<0, false, false, false>(p, a, st);
    if (!nlout) return go_yz<1, false, false, false>(p, a, st);
    return p3 ? go_yz<1, false, true, true>(p, a, st) : go_yz<1, false, true, false>(p, a, st);
}

}  // namespace gp
