// sscn_split.cuh -- what the sub-line sweeps share (sscn_split.cu: FP64 and
// complex64 arithmetic; sscn_inc.cu: FP64 psi, float-float increments): the cut
// of a line into half sub-lines, the kernel arguments and their coefficients,
// and the FP64 solve of half a sub-line.  The method is described in
// sscn_split.cu.
#pragma once

#include <algorithm>
#include <cmath>
#include <complex>

#include <cuda_runtime.h>

#include "sscn_accum.cuh"
#include "sscn_internal.h"
#include "sscn_line.cuh"
#include "sscn_pdl.cuh"

namespace gp {
namespace sp {

constexpr int kSplitThreads = 512;       // most threads of a block
constexpr size_t kSplitSmem = 200 * 1024;
constexpr int kSplitConv = 256;          // most rows before the elimination coefficients are constant
constexpr int kSms = 152;
constexpr int kSplitEnds = 4;            // sub-lines at either end with a middle-row multiplier of their own

// Shared-memory index of row i of a line: one element of padding every 8 rows,
// so lanes whose rows lie 2 P apart fall on different banks.
__host__ __device__ __forceinline__ int slot_of(int i) { return i + (i >> 3); }

template <typename T> struct SplitArgs {
    using C = typename Cx<T>::t;
    using F = typename Coef<T>::t;
    C *psi;
    int n, S, W, conv;
    int per;                 // lines per block (x: rows R; y / z: neighbouring lines XL, a power of two)
    int lines_a, lines_b;
    long long stride_a, stride_b, pstride;
    unsigned magic;          // ceil(2^32 / (n - 1)) (x)
    T k;                     // kappa or kappa / i
    C rinf, tinf;            // constants past conv
    C mid[2 * kSplitEnds + 1];   // middle-row multipliers of the first and last sub-lines, and of the others
    C mlo[2 * kSplitEnds + 1];   // FP64: what 2 mid lacks (see split_args)
    const F *mult, *cp;      // m entries
    F minf, cinf, mid1;      // complex64: their constants past conv, the one middle row's multiplier
    const F *px, *py, *pz;
    const float *tx, *ty, *tz;
    StepG sg;
    const double *scale;
    double *partials;
    const double *lw;
    const double2 *p3;
};


// p + f e
template <int MODE, typename C> __device__ __forceinline__ C cfma(C f, C e, C p)
{
    C r;
    if (MODE == 0) {
        r.x = fma(f.x, e.x, p.x);
        r.y = fma(f.x, e.y, p.y);
    } else {
        r.x = fma(-f.y, e.y, fma(f.x, e.x, p.x));
        r.y = fma(f.y, e.x, fma(f.x, e.y, p.y));
    }
    return r;
}

// kappa z
template <typename T, int MODE> __device__ __forceinline__ typename Cx<T>::t ktimes(T k, typename Cx<T>::t z)
{
    return MODE == 0 ? cx<T>(k * z.x, k * z.y) : cx<T>(-k * z.y, k * z.x);
}

// A sweep's coefficients in shared memory.  A lane near a line's end would
// otherwise wait on a table load from memory in every step of its chain, and a
// division for its middle row would cost about as much FP64-pipe time as all
// its rows.  FP64: r_t for t = -1 .. conv (entry t + 1; no row before the
// first: r = 0), t_t likewise, the middle-row multipliers and their rests.  complex64: mult and
// c' (hi + lo pairs) for t = 0 .. conv.
template <typename T> __host__ __device__ __forceinline__ size_t coef_bytes(int conv)
{
    return sizeof(T) == 8 ? (size_t)(2 * (conv + 2) + 2 * (2 * kSplitEnds + 1)) * 16 : (size_t)2 * (conv + 1) * 16;
}

template <int MODE> __device__ __forceinline__ void stage_coefs(const SplitArgs<double> &a, void *to)
{
    double2 *tab = static_cast<double2 *>(to);
    const int len = a.conv + 2;
    for (int q = threadIdx.x; q < len; q += blockDim.x) {
        double2 r = a.rinf, t = a.tinf;
        if (q == 0) r = make_double2(0.0, 0.0);
        else if (q <= a.conv) {
            const double2 f = a.mult[q - 1];
            r = ktimes<double, MODE>(a.k, f);
            t = make_double2(2.0 * f.x, 2.0 * f.y);
        }
        tab[q] = r;
        tab[len + q] = t;
    }
    for (int q = threadIdx.x; q <= 2 * kSplitEnds; q += blockDim.x) {
        tab[2 * len + q] = a.mid[q];
        tab[2 * len + 2 * kSplitEnds + 1 + q] = a.mlo[q];
    }
}

template <int MODE> __device__ __forceinline__ void stage_coefs(const SplitArgs<float> &a, void *to)
{
    float4 *tab = static_cast<float4 *>(to);
    for (int q = threadIdx.x; q <= a.conv; q += blockDim.x) {
        tab[q] = q < a.conv ? a.mult[q] : a.minf;
        tab[a.conv + 1 + q] = q < a.conv ? a.cp[q] : a.cinf;
    }
}

enum { kFp64 = 0, kTwoEnded = 1, kIncrement = 2 };       // FORM
template <int FORM> struct Num { using T = float; };
template <> struct Num<kFp64> { using T = double; };

// One lane's share of a line.
template <int FORM, int MODE> struct Share;

// Half a sub-line (segment 2 s: top, 2 s + 1: bottom of sub-line s).  Rows are
// addressed by their distance t from the end of the line the lane's elimination
// comes from: row 1 + t (top) or m - t; its own rows are t = to .. te (te < to:
// none), the window starts at ts; it moves rows first .. last (the top half's
// with the middle row, at distance kt).
struct HalfLine {
    bool top;
    int m, s, to, te, ts, kt, first, last;

    __device__ __forceinline__ HalfLine(int n, int S, int W, int seg)
    {
        m = n - 1;
        s = seg >> 1;
        const int lo = 1 + s * m / S, hi = (s + 1) * m / S;
        const int k = lo + ((hi - lo) >> 1);
        top = (seg & 1) == 0;
        to = top ? lo - 1 : m - hi;
        te = top ? k - 2 : m - k - 1;
        kt = top ? k - 1 : m - k;
        ts = max(0, to - W);
        first = to;
        last = top ? kt : te;
    }
    __device__ __forceinline__ int row(int t) const { return top ? 1 + t : m - t; }
    // where the sub-line's middle-row multiplier lies among the 2 kSplitEnds + 1
    __device__ __forceinline__ int mid_at(int S) const
    {
        return s < kSplitEnds ? s : (S - s <= kSplitEnds ? 2 * kSplitEnds - (S - s) : 2 * kSplitEnds);
    }
};

// FP64 arithmetic on half a sub-line.
template <int MODE> struct Share<kFp64, MODE> : HalfLine {
    using C = double2;
    const SplitArgs<double> &a;
    const C *tab;            // stage_coefs

    __device__ __forceinline__ Share(const SplitArgs<double> &args, const void *tables, int seg)
        : HalfLine(args.n, args.S, args.W, seg), a(args), tab(static_cast<const C *>(tables))
    {
    }
    // r_t and t_t of the row at distance t
    __device__ __forceinline__ C r(int t) const { return tab[min(t, a.conv) + 1]; }
    __device__ __forceinline__ C out_mul(int t) const { return tab[a.conv + 3 + min(t, a.conv)]; }
    __device__ __forceinline__ const C *mid_mul() const { return tab + 2 * (a.conv + 2) + mid_at(a.S); }

    // Solve; ld(i): psi at row i, out(i, u) stores.  pair: lane distance of the
    // two halves.  barrier() separates the forward pass (which reads other
    // lanes' rows) from the stores.  Every thread of the block calls this;
    // `active` marks lanes with a line.
    template <int P, bool SYNC, typename Ld, typename LdD, typename PutD, typename Out>
    __device__ __forceinline__ void solve(bool active, int pair, Ld ld, LdD, PutD, Out out) const
    {
        const C zero = make_double2(0.0, 0.0);
        C e = zero, ev[P];
        if (active) {
            int t = ts;
            for (; t < to && t - 1 < a.conv; ++t) e = cfma<MODE>(r(t - 1), e, ld(row(t)));
#pragma unroll 4
            for (; t < to; ++t) e = cfma<MODE>(a.rinf, e, ld(row(t)));
            if (to > a.conv) {
#pragma unroll
                for (int q = 0; q < P; ++q)
                    if (to + q <= te) ev[q] = e = cfma<MODE>(a.rinf, e, ld(row(to + q)));
            } else {
#pragma unroll
                for (int q = 0; q < P; ++q)
                    if (to + q <= te) ev[q] = e = cfma<MODE>(r(to + q - 1), e, ld(row(to + q)));
            }
        }
        // the carries of both halves meet in the middle row
        const C c = cfma<MODE>(r(te), e, zero);
        C o;
        o.x = __shfl_xor_sync(0xffffffffu, c.x, pair);
        o.y = __shfl_xor_sync(0xffffffffu, c.y, pair);
        C v = zero, pk = zero, x = zero;
        const C *mm = mid_mul();
        if (active && top) {
            pk = ld(row(kt));
            x = make_double2(pk.x + c.x + o.x, pk.y + c.y + o.y);
            v = cfma<MODE>(*mm, x, zero);
        }
        if (SYNC) __syncthreads();
        C w;
        w.x = __shfl_xor_sync(0xffffffffu, v.x, pair);
        w.y = __shfl_xor_sync(0xffffffffu, v.y, pair);
        if (top) w = v;
        // (off the chain: the lanes of the other half have v by now)
        if (active && top)
            out(row(kt), cfma<MODE>(mm[2 * kSplitEnds + 1], x, make_double2(fma(2.0, v.x, -pk.x), fma(2.0, v.y, -pk.y))));
        C f = MODE == 0 ? make_double2(a.k, 0.0) : make_double2(0.0, a.k);   // kappa v_k enters first
        if (active) {
            auto step = [&](int q, C rf, C tf) {
                w = cfma<MODE>(f, w, ev[q]);
                f = rf;
                const int i = row(to + q);
                const C p = ld(i);
                out(i, cfma<MODE>(tf, w, make_double2(-p.x, -p.y)));
            };
            if (to >= a.conv) {
#pragma unroll
                for (int q = P - 1; q >= 0; --q)
                    if (to + q <= te) step(q, a.rinf, a.tinf);
            } else {
#pragma unroll
                for (int q = P - 1; q >= 0; --q)
                    if (to + q <= te) step(q, r(to + q), out_mul(to + q));
            }
        }
    }
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Fixed-order sum over the block into *out (thread 0); red: 32 doubles.
__device__ __forceinline__ void block_partial(double part, double *red, double *out)
{
    part = warp_sum(part);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x < 32) {
        const double v = warp_sum(threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0);
        if (threadIdx.x == 0) *out = v;
    }
}

// All of an SM's shared memory for resident blocks, and as much as any block of
// these kernels needs: without this a block's static and dynamic shared memory
// together may not pass 48 KB, so the dynamic part alone does not say whether
// it is needed.
template <typename K> cudaError_t allow_smem(K kern)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSplitSmem);
}

// Host: a sum of numbers and products to about twice FP64's bits.
struct LongSum {
    double h = 0.0, l = 0.0;

    void add(double x)
    {
        const double s = h + x, b = s - h;
        l += (h - (s - b)) + (x - b);
        h = s;
    }
    void add(double x, double y)
    {
        const double p = x * y;
        add(p);
        l += std::fma(x, y, -p);
    }
};

// Host: what f lacks of 1 / (1 + 2 kappa - kappa (ra + rb)), kappa = k or i k.
inline double2 inverse_rest(int mode, double k, double2 ra, double2 rb, double2 f)
{
    LongSum dx, dy;                      // the denominator
    dx.add(1.0);
    (mode == 0 ? dx : dy).add(2.0 * k);
    for (const double2 r : {ra, rb}) {
        if (mode == 0) dx.add(-k, r.x);
        else {
            dx.add(k, r.y);
            dy.add(-k, r.x);
        }
    }
    LongSum ex, ey;                      // 1 - denominator f
    ex.add(1.0);
    ex.add(-dx.h, f.x);
    ex.add(dy.h, f.y);
    ey.add(-dx.h, f.y);
    ey.add(-dy.h, f.x);
    const double x = ex.h + (ex.l - dx.l * f.x + dy.l * f.y), y = ey.h + (ey.l - dx.l * f.y - dy.l * f.x);
    return make_double2(x * f.x - y * f.y, x * f.y + y * f.x);
}

// Host: the kernel arguments of a sweep.
template <int FORM>
SplitArgs<typename Num<FORM>::T> split_args(const SplitPlan &p, int mode, void *psi, const AxisTables &ax,
                                            const SweepGeom &g, const NonlinArgs *nl, const Partials *norm_out)
{
    using T = typename Num<FORM>::T;
    using C = typename Cx<T>::t;
    constexpr bool D = FORM == kFp64;
    SplitArgs<T> a{};
    a.psi = static_cast<C *>(psi);
    a.n = g.n;
    a.S = p.S;
    a.W = p.W;
    a.per = p.per;
    a.lines_a = g.lines_a;
    a.lines_b = g.lines_b;
    a.stride_a = g.stride_a;
    a.stride_b = g.stride_b;
    a.pstride = g.pstride;
    a.magic = (unsigned)((0x100000000ull + (g.n - 2)) / (unsigned)(g.n - 1));
    a.conv = D ? ax.conv64 : ax.conv32;
    const double k = mode == 0 ? ax.kre : ax.kim;
    a.k = (T)k;
    if constexpr (D) {
        // constants past conv: r = kappa mult and the output multiplier
        const double2 mu = ax.minf64;
        a.rinf = mode == 0 ? make_double2(k * mu.x, 0.0) : make_double2(-k * mu.y, k * mu.x);
        a.tinf = make_double2(2.0 * mu.x, 2.0 * mu.y);
        a.mult = ax.mult64;
        // middle rows: 1 / (1 + 2 kappa - kappa (r above + r below)), r from the
        // recurrence the tables hold.  The roundings of mu and of these factors
        // repeat at every step.  One that all rows share only scales the state;
        // rows of their own rounding every 2 P rows leave a pattern that grows, so
        // mlo carries them to 2 mid exact (1 + delta), delta the relative rounding
        // of mu.  500 x 384 imaginary time, kappa 0.026 .. 0.05, 30 steps, error
        // against 64 bits on average: lane pairs per line 1.76e-15, without mlo
        // 1.91e-15, with it 1.67e-15; 300 x 260 1.61, 1.66 and 1.50e-15.
        const int m = g.n - 1, nrt = std::min(a.conv, m);
        double2 rt[kSplitConv], mult, cp = make_double2(0.0, 0.0);
        for (int t = 0; t < nrt; ++t) {
            thomas_step(ax.kre, ax.kim, cp.x, cp.y, mult, cp);
            rt[t] = make_double2(-cp.x, -cp.y);
        }
        auto r_at = [&](int t) { return t < 0 ? make_double2(0.0, 0.0) : t < nrt ? rt[t] : a.rinf; };
        const double2 rest = inverse_rest(mode, k, r_at(m - 2), make_double2(0.0, 0.0), mu);
        const std::complex<double> delta = -std::complex<double>(rest.x, rest.y) / std::complex<double>(mu.x, mu.y);
        auto mid_of = [&](int q, double2 ra, double2 rb) {
            const std::complex<double> kc(ax.kre, ax.kim);
            const std::complex<double> f = 1.0 / (1.0 + 2.0 * kc - kc * std::complex<double>(ra.x + rb.x, ra.y + rb.y));
            a.mid[q] = make_double2(f.real(), f.imag());
            const double2 lo = inverse_rest(mode, k, ra, rb, a.mid[q]);
            const std::complex<double> ml = 2.0 * (std::complex<double>(lo.x, lo.y) + delta * f);
            a.mlo[q] = make_double2(ml.real(), ml.imag());
        };
        for (int q = 0; q < 2 * kSplitEnds; ++q) {
            const int s = q < kSplitEnds ? q : p.S - 2 * kSplitEnds + q;
            if (s < 0 || s >= p.S) continue;
            const int lo = 1 + s * m / p.S, hi = (s + 1) * m / p.S, row = lo + ((hi - lo) >> 1);
            mid_of(q, r_at(row - 2), r_at(m - row - 1));
        }
        mid_of(2 * kSplitEnds, a.rinf, a.rinf);
    } else {
        a.mult = ax.mult32;
        a.cp = ax.cp32;
        a.minf = ax.minf32;
        a.cinf = ax.cinf32;
        a.mid1 = ax.mid32;
    }
    if (nl) {
        if constexpr (D) {
            a.px = nl->px;
            a.py = nl->py;
            a.pz = nl->pz;
            a.p3 = nl->p3;
        } else {
            a.px = nl->px32;
            a.py = nl->py32;
            a.pz = nl->pz32;
        }
        a.tx = nl->tx32;
        a.ty = nl->ty32;
        a.tz = nl->tz32;
        a.sg = nl->g;
        a.scale = nl->scale;
    }
    a.partials = norm_out ? norm_out->buf : nullptr;
    a.lw = norm_out ? norm_out->line_weight : nullptr;
    return a;
}

}  // namespace sp
}  // namespace gp
