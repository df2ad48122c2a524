// sscn_split.cu -- Crank-Nicolson sweeps (calclux, calcluy, calcluz, calcnu
// fused) with every grid line cut into sub-lines that many lanes solve at
// once: the sweeps of grids with too few lines to fill the GPU one lane pair
// per line (2D grids, small 3D grids).
//
// What bounds them.  k_sweep (sscn_kernels.cu) gives a line two lanes, so a
// 500 x 384 plane runs on 64 warps, each a serial chain of n / 2 dependent
// steps out and back: latency, at 2 % of the FP64 rate.  Here a line of m
// unknowns becomes S sub-lines of at most 2 P rows, each eliminated from both
// ends by a lane pair that meets in its middle row, so a lane's chain is W + P
// steps forward and P back, and the lanes are n / P per line.  The whole line
// sits in one block's shared memory: psi crosses global memory once each way
// (k_sweep: two reads, the elimination scratch written and read, one write).
//
// Windows.  An elimination that starts inside the line has no carry from the
// rows before it.  Each lane starts W rows outside its own rows from zero:
// the dropped carry reaches its first own row damped by the product of |c'|
// over the window, below 2^-55 (FP64) / 2^-40 (complex64) of the neighbouring
// values; a window that reaches the end of the line starts exactly there.
// The elimination coefficients are the line's own (they depend on the row's
// distance from the end the elimination comes from), so nothing else changes.
//
// FP64 arithmetic per row (kappa = k or i k, r_j = kappa mult_j, t_j = 2 mult_j):
//     e_j = p_j + r_{j-1} e_{j-1}            (from the top; mirrored from the bottom)
//     v_k = mid_k (p_k + r e_{k-1} + r e_{k+1})          (middle row)
//     w_j = e_j + r_{j+1} w_{j+1},  u_j = t_j w_j - p_j   (v_j = mult_j w_j)
// which is Thomas' recurrence with the multiplier moved out of the forward
// pass: 6 FP64 instructions a row in imaginary time (k_sweep: 8), 12 in real
// time.
//
// complex64 keeps the arithmetic and the direction of the kernels it stands in
// for (a state's observables are reported in FP64, where another order of FP32
// roundings shows): each half of a line (k_sweep, one middle row), or the whole
// line (k_sweep_tma: increment form, one direction), is cut into runs of at
// most P rows, and a lane runs the elimination over W rows before its run and
// the back substitution over W rows after it as well.  Once the dropped carry
// is below the last bit, the recurrences produce those kernels' bits.

#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include <cuda_runtime.h>

#include "sscn_accum.cuh"
#include "sscn_internal.h"
#include "sscn_line.cuh"

namespace gp {
namespace {

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
// first: r = 0), t_t likewise, the middle-row multipliers.  complex64: mult and
// c' (hi + lo pairs) for t = 0 .. conv.
template <typename T> __host__ __device__ __forceinline__ size_t coef_bytes(int conv)
{
    return sizeof(T) == 8 ? (size_t)(2 * (conv + 2) + 2 * kSplitEnds + 1) * 16 : (size_t)2 * (conv + 1) * 16;
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
    for (int q = threadIdx.x; q <= 2 * kSplitEnds; q += blockDim.x) tab[2 * len + q] = a.mid[q];
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

// One lane's share of a line.  Rows are addressed by their distance t from the
// end of the line the lane's elimination comes from: row 1 + t (top) or m - t;
// its own rows are t = to .. te (te < to: none), first .. last those it moves.
template <int FORM, int MODE> struct Share;

// FP64: half a sub-line (segment 2 s: top, 2 s + 1: bottom of sub-line s).
template <int MODE> struct Share<kFp64, MODE> {
    using C = double2;
    const SplitArgs<double> &a;
    const C *tab;            // stage_coefs
    bool top;
    int m, seg, to, te, ts;  // window from ts
    int kt;                  // the middle row's distance from this lane's end
    int first, last;

    __device__ __forceinline__ Share(const SplitArgs<double> &args, const void *tables, int segment)
        : a(args), tab(static_cast<const C *>(tables)), seg(segment)
    {
        m = a.n - 1;
        const int s = seg >> 1;
        const int lo = 1 + s * m / a.S, hi = (s + 1) * m / a.S;
        const int k = lo + ((hi - lo) >> 1);
        top = (seg & 1) == 0;
        to = top ? lo - 1 : m - hi;
        te = top ? k - 2 : m - k - 1;
        kt = top ? k - 1 : m - k;
        ts = max(0, to - a.W);
        first = to;
        last = top ? kt : te;
    }
    __device__ __forceinline__ int row(int t) const { return top ? 1 + t : m - t; }
    // r_t and t_t of the row at distance t
    __device__ __forceinline__ C r(int t) const { return tab[min(t, a.conv) + 1]; }
    __device__ __forceinline__ C out_mul(int t) const { return tab[a.conv + 3 + min(t, a.conv)]; }
    // the sub-line's middle-row multiplier
    __device__ __forceinline__ C mid_mul() const
    {
        const int s = seg >> 1;
        const int at = s < kSplitEnds ? s : (a.S - s <= kSplitEnds ? 2 * kSplitEnds - (a.S - s) : 2 * kSplitEnds);
        return tab[2 * (a.conv + 2) + at];
    }

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
        C v = zero, pk = zero;
        if (active && top) {
            pk = ld(row(kt));
            v = cfma<MODE>(mid_mul(), make_double2(pk.x + c.x + o.x, pk.y + c.y + o.y), zero);
        }
        if (SYNC) __syncthreads();
        if (active && top) out(row(kt), make_double2(fma(2.0, v.x, -pk.x), fma(2.0, v.y, -pk.y)));
        C w;
        w.x = __shfl_xor_sync(0xffffffffu, v.x, pair);
        w.y = __shfl_xor_sync(0xffffffffu, v.y, pair);
        if (top) w = v;
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

// complex64: a run of at most P rows of the top (even segments) or bottom half
// of the line; runs are numbered from the line's end to its middle.
template <int MODE> struct Share<kTwoEnded, MODE> {
    using C = float2;
    using F = float4;
    const SplitArgs<float> &a;
    const F *tab;            // stage_coefs
    bool top;
    int m, to, te, len, kt, first, last;

    __device__ __forceinline__ Share(const SplitArgs<float> &args, const void *tables, int seg)
        : a(args), tab(static_cast<const F *>(tables))
    {
        m = a.n - 1;
        const int k = (m + 1) >> 1, j = seg >> 1;
        top = (seg & 1) == 0;
        len = top ? k - 1 : m - k;
        to = j * len / a.S;
        te = (j + 1) * len / a.S - 1;
        kt = len;
        first = to;
        last = top && j == a.S - 1 ? kt : te;
    }
    __device__ __forceinline__ int row(int t) const { return top ? 1 + t : m - t; }
    __device__ __forceinline__ F mult(int t) const { return tab[min(t, a.conv)]; }
    __device__ __forceinline__ F cp(int t) const { return tab[a.conv + 1 + min(t, a.conv)]; }

    // As the FP64 form's; ldd / putd: d' of a row, kept where the lanes of the
    // line see it.
    template <int P, bool SYNC, typename Ld, typename LdD, typename PutD, typename Out>
    __device__ __forceinline__ void solve(bool active, int, Ld ld, LdD ldd, PutD putd, Out out) const
    {
        const LineOps<float, MODE> cn{a.k};
        C d = make_float2(0.f, 0.f), pk = d, dv[P];
        if (active) {
            int t = max(0, to - a.W);
            for (; t < to && t < a.conv; ++t) d = cn.fwd(ld(row(t)), d, mult(t));
#pragma unroll 4
            for (; t < to; ++t) d = cn.fwd(ld(row(t)), d, a.minf);
#pragma unroll
            for (int q = 0; q < P; ++q)
                if (to + q <= te) {
                    dv[q] = d = cn.fwd(ld(row(to + q)), d, to >= a.conv ? a.minf : mult(to + q));
                    putd(row(to + q), d);
                }
            pk = ld(row(kt));
        }
        __syncthreads();
        if (active) {
            int t = te + a.W;                 // the window's last row
            C v = make_float2(0.f, 0.f);
            if (t >= len - 1) {
                // it reaches the middle row: v_k from both halves' last d'
                const C x = len > 0 ? ldd(row(kt - 1)) : v;
                const int other = top ? m - ((m + 1) >> 1) : ((m + 1) >> 1) - 1;   // rows of the other half
                const C y = other > 0 ? ldd(row(kt + 1)) : v;
                v = cn.fwd(pk, make_float2(x.x + y.x, x.y + y.y), a.mid1);
                if (last == kt) out(row(kt), LineOps<float, MODE>::out(v, pk));
                t = len - 1;
            }
            for (; t > te && t >= a.conv; --t) v = cn.back(ldd(row(t)), a.cinf, v);
            for (; t > te; --t) v = cn.back(ldd(row(t)), cp(t), v);
#pragma unroll
            for (int q = P - 1; q >= 0; --q)
                if (to + q <= te) {
                    v = cn.back(dv[q], to >= a.conv ? a.cinf : cp(to + q), v);
                    const int i = row(to + q);
                    out(i, LineOps<float, MODE>::out(v, ld(i)));
                }
        }
    }
};

// complex64, increment form: a run of at most P rows of the line, eliminated
// from the top: (I - kappa L) D = kappa L p, u = p + 2 D, with the hi parts of
// the coefficients (k_sweep_tma's arithmetic; see there for why).
template <int MODE> struct Share<kIncrement, MODE> {
    using C = float2;
    using F = float4;
    const SplitArgs<float> &a;
    const F *tab;            // stage_coefs
    int m, to, te, first, last;

    __device__ __forceinline__ Share(const SplitArgs<float> &args, const void *tables, int seg)
        : a(args), tab(static_cast<const F *>(tables))
    {
        m = a.n - 1;
        to = seg * m / (2 * a.S);
        te = (seg + 1) * m / (2 * a.S) - 1;
        first = to;
        last = te;
    }
    __device__ __forceinline__ int row(int t) const { return 1 + t; }
    __device__ __forceinline__ F mult(int t) const { return tab[min(t, a.conv)]; }
    __device__ __forceinline__ F cp(int t) const { return tab[a.conv + 1 + min(t, a.conv)]; }

    // ld also reads rows 0 and n, which hold zero
    template <int P, bool SYNC, typename Ld, typename LdD, typename PutD, typename Out>
    __device__ __forceinline__ void solve(bool active, int, Ld ld, LdD ldd, PutD putd, Out out) const
    {
        const LineOps<float, MODE, true> cn{a.k};
        C d = make_float2(0.f, 0.f), dv[P];
        if (active) {
            int t = max(0, to - a.W);
            C pa = ld(t), pb = ld(t + 1);
            auto rhs = [&](int at) {
                const C pj = ld(at + 2), s = cn.lap(pa, pb, pj);
                pa = pb;
                pb = pj;
                return s;
            };
            for (; t < to && t < a.conv; ++t) d = cn.fwd(rhs(t), d, mult(t));
#pragma unroll 4
            for (; t < to; ++t) d = cn.fwd(rhs(t), d, a.minf);
#pragma unroll
            for (int q = 0; q < P; ++q)
                if (to + q <= te) {
                    dv[q] = d = cn.fwd(rhs(to + q), d, to >= a.conv ? a.minf : mult(to + q));
                    putd(row(to + q), d);
                }
        }
        __syncthreads();
        if (active) {
            C v = make_float2(0.f, 0.f);      // v_m = d'_m: zero beyond the last row
            int t = min(te + a.W, m - 1);
            for (; t > te && t >= a.conv; --t) v = cn.back(ldd(row(t)), a.cinf, v);
            for (; t > te; --t) v = cn.back(ldd(row(t)), cp(t), v);
#pragma unroll
            for (int q = P - 1; q >= 0; --q)
                if (to + q <= te) {
                    v = cn.back(dv[q], to >= a.conv ? a.cinf : cp(to + q), v);
                    const int i = row(to + q);
                    out(i, LineOps<float, MODE, true>::out_inc(v, ld(i)));
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

// x sweep: a block owns `per` lines, lane pair (2 s, 2 s + 1) of a line its
// sub-line s.  The lines come in coalesced (any row length), pass through
// calcnu once per point on the way into shared memory, and leave coalesced.
template <int FORM, int MODE, bool NL, bool P3, int P>
__global__ void __launch_bounds__(kSplitThreads) k_split_x(const __grid_constant__ SplitArgs<typename Num<FORM>::T> a)
{
    using T = typename Num<FORM>::T;
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, m = n - 1, pitch = slot_of(n) + 1;
    using Lane = Share<FORM, MODE>;
    Calcnu<T, MODE> *row_nl = reinterpret_cast<Calcnu<T, MODE> *>(smem_raw + coef_bytes<T>(a.conv));
    C *tile = reinterpret_cast<C *>(row_nl + a.per), *dtile = tile + a.per * pitch;
    const int line0 = blockIdx.x * a.per;
    const int rows = min(a.per, a.lines_a * a.lines_b - line0);
    __shared__ double g_of_step;
    if (P3 && threadIdx.x == 0) g_of_step = a.sg.value();
    if (NL && !P3)
        for (int q = threadIdx.x; q < rows; q += blockDim.x) {
            const int L = line0 + q;
            row_nl[q].setup(a.px, a.py, a.pz, a.tx, a.ty, a.tz, L % a.lines_a, L / a.lines_a, a.sg.value(),
                            a.scale);
        }
    stage_coefs<MODE>(a, smem_raw);
    if (FORM == kIncrement)
        for (int q = threadIdx.x; q < a.per; q += blockDim.x)
            tile[q * pitch] = tile[q * pitch + slot_of(n)] = cx<T>((T)0, (T)0);
    // points 1 .. m of all rows as one range, kB loads of a thread in flight
    constexpr int kB = 4;
    const int count = rows * m;
    const C *src = a.psi + (long long)line0 * n;
    const double2 *src3 = P3 ? a.p3 + (long long)line0 * n : nullptr;
    C v[kB];
    double2 f3[P3 ? kB : 1];
    auto place = [&](int idx, int &q, int &i) {
        q = (int)__umulhi((unsigned)idx, a.magic);
        i = 1 + idx - q * m;
    };
    auto fetch = [&](int base) {
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const int idx = base + b * blockDim.x;
            if (idx < count) {
                int q, i;
                place(idx, q, i);
                v[b] = src[q * n + i];
                if constexpr (P3) f3[b] = src3[q * n + i];
            }
        }
    };
    fetch(threadIdx.x);
    if (NL) __syncthreads();                 // row_nl, g_of_step
    const double G3 = P3 ? g_of_step : 0.0;
    for (int base = threadIdx.x; base < count; base += kB * blockDim.x) {
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const int idx = base + b * blockDim.x;
            if (idx < count) {
                int q, i;
                place(idx, q, i);
                if constexpr (NL && P3) {
                    double cs, sn;
                    expmi_small(G3 * fma(v[b].x, v[b].x, v[b].y * v[b].y), cs, sn);
                    const double2 z = make_double2(fma(cs, v[b].x, sn * v[b].y), fma(cs, v[b].y, -sn * v[b].x));
                    v[b] = cmulc(z, f3[b]);
                } else if constexpr (NL) {
                    v[b] = row_nl[q].apply(v[b], i);
                }
                tile[q * pitch + slot_of(i)] = v[b];
            }
        }
        fetch(base + kB * blockDim.x);
    }
    const int lanes = 2 * a.S;
    const int q = threadIdx.x / lanes, seg = threadIdx.x - q * lanes;
    const bool active = q < rows;
    const Lane lane(a, smem_raw, active ? seg : (threadIdx.x & 1));
    C *line = tile + (active ? q : 0) * pitch, *dline = dtile + (active ? q : 0) * pitch;
    __syncthreads();
    lane.template solve<P, true>(
        active, 1, [&](int i) { return line[slot_of(i)]; }, [&](int i) { return dline[slot_of(i)]; },
        [&](int i, C d) { dline[slot_of(i)] = d; }, [&](int i, C u) { line[slot_of(i)] = u; });
    __syncthreads();
    C *dst = a.psi + (long long)line0 * n;
    for (int idx = threadIdx.x; idx < count; idx += blockDim.x) {
        int r, i;
        place(idx, r, i);
        dst[r * n + i] = tile[r * pitch + slot_of(i)];
    }
}

// y / z sweep: a block owns `per` neighbouring lines (power of two, at most
// 16), lane segments of one line `per` lanes apart, so every row of the block
// is one contiguous piece of memory.  Each lane loads its own rows into shared
// memory and stores its results straight from registers.
template <int FORM, int MODE, bool NORM, bool NLOUT, bool P3, int P>
__global__ void __launch_bounds__(kSplitThreads) k_split_yz(const __grid_constant__ SplitArgs<typename Num<FORM>::T> a)
{
    using T = typename Num<FORM>::T;
    using C = typename Cx<T>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[32], g_of_step;
    using Lane = Share<FORM, MODE>;
    C *tile = reinterpret_cast<C *>(smem_raw + coef_bytes<T>(a.conv)), *dtile = tile + a.per * (slot_of(a.n) + 1);
    if (NLOUT && threadIdx.x == 0) g_of_step = a.sg.value();
    const int n = a.n, XL = a.per;
    const int xl = threadIdx.x & (XL - 1), seg = threadIdx.x / XL;
    const int la = blockIdx.x * XL + xl, lb = blockIdx.y;
    const bool active = la < a.lines_a && seg < 2 * a.S;
    const Lane lane(a, smem_raw, seg < 2 * a.S ? seg : (seg & 1));
    const long long base = active ? (long long)la * a.stride_a + (long long)lb * a.stride_b : 0;
    C *line = a.psi + base;
    constexpr int kOwn = FORM == kTwoEnded ? P + 1 : P;  // with the middle row
    C p[kOwn];
    if (active) {
        // own rows, all loads in flight
#pragma unroll
        for (int q = 0; q < kOwn; ++q)
            if (lane.first + q <= lane.last) p[q] = line[(long long)lane.row(lane.first + q) * a.pstride];
    }
    stage_coefs<MODE>(a, smem_raw);
    if (active) {
#pragma unroll
        for (int q = 0; q < kOwn; ++q)
            if (lane.first + q <= lane.last) tile[slot_of(lane.row(lane.first + q)) * XL + xl] = p[q];
        if (FORM == kIncrement) {
            if (lane.first == 0) tile[xl] = cx<T>((T)0, (T)0);
            if (lane.last == n - 2) tile[slot_of(n) * XL + xl] = cx<T>((T)0, (T)0);
        }
    }
    Acc<T> acc;
    __syncthreads();
    Calcnu<T, MODE> nl{};
    const double G3 = NLOUT ? g_of_step : 0.0;
    if (NLOUT && !P3 && active) nl.setup(a.px, a.py, a.pz, a.tx, a.ty, a.tz, la, lb, G3, a.scale);
    auto at_of = [&](int i) { return slot_of(i) * XL + xl; };
    lane.template solve<P, false>(
        active, XL, [&](int i) { return tile[at_of(i)]; }, [&](int i) { return dtile[at_of(i)]; },
        [&](int i, C d) { dtile[at_of(i)] = d; },
        [&](int i, C u) {
            const long long at = (long long)i * a.pstride;
            if constexpr (NLOUT && P3) {
                double cs, sn;
                expmi_small(G3 * fma(u.x, u.x, u.y * u.y), cs, sn);
                u = cmulc(make_double2(fma(cs, u.x, sn * u.y), fma(cs, u.y, -sn * u.x)), a.p3[base + at]);
            } else if constexpr (NLOUT) {
                u = nl.apply(u, i);
            }
            line[at] = u;
            if (NORM) acc.add(fma(u.x, u.x, u.y * u.y));
        });
    if (NORM) {
        double part = acc.get();
        if (a.lw && active) part *= a.lw[la];
        part = warp_sum(active ? part : 0.0);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
        __syncthreads();
        if (threadIdx.x < 32) {
            double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
            v = warp_sum(v);
            if (threadIdx.x == 0) a.partials[(long long)blockIdx.y * gridDim.x + blockIdx.x] = v;
        }
    }
}

template <typename K> cudaError_t allow_smem(K kern, size_t bytes)
{
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSplitSmem);
}

template <int FORM, int MODE, bool NL, bool P3, int P, typename T>
cudaError_t go_x(const SplitPlan &p, const SplitArgs<T> &a, cudaStream_t st)
{
    auto kern = k_split_x<FORM, MODE, NL, P3, P>;
    cudaError_t e = allow_smem(kern, p.smem);
    if (e != cudaSuccess) return e;
    kern<<<p.grid_x, p.threads, p.smem, st>>>(a);
    return cudaGetLastError();
}

template <int FORM, int MODE, bool NORM, bool NLOUT, bool P3, int P, typename T>
cudaError_t go_yz(const SplitPlan &p, const SplitArgs<T> &a, cudaStream_t st)
{
    auto kern = k_split_yz<FORM, MODE, NORM, NLOUT, P3, P>;
    cudaError_t e = allow_smem(kern, p.smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(p.grid_x, p.grid_y), p.threads, p.smem, st>>>(a);
    return cudaGetLastError();
}

template <int FORM, int MODE, int P, typename T>
cudaError_t pick(const SplitPlan &p, const SplitArgs<T> &a, bool nl, bool nlout, bool norm, cudaStream_t st)
{
    constexpr bool D = FORM == kFp64 && MODE == 1;       // forms with the factor table
    const bool p3 = a.p3 != nullptr;
    if (p.x) {
        if (nlout || norm || (p3 && !D)) return cudaErrorInvalidValue;
        if (!nl) return go_x<FORM, MODE, false, false, P>(p, a, st);
        if (D && p3) return go_x<FORM, MODE, true, D, P>(p, a, st);
        return go_x<FORM, MODE, true, false, P>(p, a, st);
    }
    if (nl || (norm && (MODE == 1 || nlout)) || (nlout && MODE == 0) || (p3 && !(nlout && D)))
        return cudaErrorInvalidValue;
    if constexpr (MODE == 0) {
        if (norm) return go_yz<FORM, 0, true, false, false, P>(p, a, st);
    } else {
        if (nlout && p3) return go_yz<FORM, 1, false, true, D, P>(p, a, st);
        if (nlout) return go_yz<FORM, 1, false, true, false, P>(p, a, st);
    }
    return go_yz<FORM, MODE, false, false, false, P>(p, a, st);
}

template <int FORM>
cudaError_t launch(const SplitPlan &p, int mode, void *psi, const AxisTables &ax, const SweepGeom &g,
                   const NonlinArgs *nl, bool nlout, const Partials *norm_out, cudaStream_t st)
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
        // recurrence the tables hold
        const int m = g.n - 1;
        std::vector<double2> rt(std::min(a.conv, m));
        double2 mult, cp = make_double2(0.0, 0.0);
        for (auto &v : rt) {
            thomas_step(ax.kre, ax.kim, cp.x, cp.y, mult, cp);
            v = make_double2(-cp.x, -cp.y);
        }
        auto r_at = [&](int t) { return t < 0 ? make_double2(0.0, 0.0) : t < (int)rt.size() ? rt[t] : a.rinf; };
        auto mid_of = [&](double2 ra, double2 rb) {
            const std::complex<double> kc(ax.kre, ax.kim);
            const std::complex<double> f = 1.0 / (1.0 + 2.0 * kc - kc * std::complex<double>(ra.x + rb.x, ra.y + rb.y));
            return make_double2(f.real(), f.imag());
        };
        for (int q = 0; q < 2 * kSplitEnds; ++q) {
            const int s = q < kSplitEnds ? q : p.S - 2 * kSplitEnds + q;
            if (s < 0 || s >= p.S) continue;
            const int lo = 1 + s * m / p.S, hi = (s + 1) * m / p.S, row = lo + ((hi - lo) >> 1);
            a.mid[q] = mid_of(r_at(row - 2), r_at(m - row - 1));
        }
        a.mid[2 * kSplitEnds] = mid_of(a.rinf, a.rinf);
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
    const bool fused = nl != nullptr && !nlout, out = nl != nullptr && nlout, norm = norm_out != nullptr;
    if (p.P != 8 && p.P != 16) return cudaErrorInvalidValue;
    if (mode == 0) return p.P == 8 ? pick<FORM, 0, 8>(p, a, fused, out, norm, st) : pick<FORM, 0, 16>(p, a, fused, out, norm, st);
    return p.P == 8 ? pick<FORM, 1, 8>(p, a, fused, out, norm, st) : pick<FORM, 1, 16>(p, a, fused, out, norm, st);
}

}  // namespace

namespace {

// Launch shape for sub-lines of at most 2 P rows; false if a block cannot hold
// a line that way.
bool shape_plan(SplitPlan &p, int P, int conv, int m, bool d, const SweepGeom &g)
{
    const long long lines = (long long)g.lines_a * g.lines_b;
    const size_t tables = d ? coef_bytes<double>(conv) : coef_bytes<float>(conv);
    // FP64: psi of a line; complex64: psi and d'
    const size_t line = (size_t)(slot_of(g.n) + 1) * 16;
    p.P = P;
    p.S = (m + 2 * P - 1) / (2 * P);
    const int lanes = 2 * p.S, least = p.x ? 1 : 2;
    if (d && p.S > 2 * kSplitEnds && conv > kSplitEnds * P) return false;
    if (lanes * least > kSplitThreads || tables + 64 + line * least > kSplitSmem) return false;
    if (p.x) {
        // rows per block: about 256 lanes and at most 64 KB, fewer rows while
        // there would be fewer blocks than SMs
        const size_t row = line + sizeof(Calcnu<double, 0>);
        int per = lanes >= 256 ? 1 : 256 / lanes;
        while (per > 1 && per * row > 64 * 1024) --per;
        if (lines < (long long)kSms * per) per = (int)((lines + kSms - 1) / kSms);
        p.per = per;
        p.smem = tables + per * row;
        p.grid_x = (unsigned)((lines + per - 1) / per);
        p.grid_y = 1;
    } else {
        // 16 neighbouring lines (a row of the block is 256 or 128 contiguous
        // bytes), fewer while the block is too large or blocks are scarce
        int per = 16;
        while (per > 2 && (lanes * per > kSplitThreads || per * line > 64 * 1024)) per /= 2;
        while (per > 2 && (long long)((g.lines_a + per - 1) / per) * g.lines_b < kSms) per /= 2;
        p.per = per;
        p.smem = tables + per * line;
        p.grid_x = (unsigned)((g.lines_a + per - 1) / per);
        p.grid_y = (unsigned)g.lines_b;
    }
    p.threads = (p.per * lanes + 31) / 32 * 32;
    return true;
}

// Microseconds of the two FP64 sweeps, fitted to measurements (GB300, both
// modes, 32^2 to 256^3).  A warp-wide FP64 instruction holds a quarter-SM's
// FP64 pipe for 64 clocks (0.034 us), so both are counted in such
// instructions: the sub-line sweep's per lane, at 2/3 of the pipe's rate; the
// two-lane sweep's a row, with the latency of a row as its floor while there
// are fewer than about two warps per quarter-SM (608 of them).
double split_us(const SplitPlan &p, bool real, long long lines)
{
    const double window = p.W * (1.0 - 1.0 / p.S), rows = p.P;
    const double instr = (real ? 4.0 : 2.0) * (window + 3.0 * rows) + (p.x ? (real ? 15.0 : 12.0) * rows : 0.0);
    const double warps = (double)lines * 2 * p.S / 32 / (4 * kSms);
    return 6.0 + std::max(1.0, warps) * instr * 0.05;
}

double pair_us(bool x, bool real, int m, long long lines)
{
    const double warps = (double)lines / 16 / (4 * kSms) + 0.35;
    const double row = x ? (real ? std::max(1.4, 1.08 * warps) : std::max(1.1, 0.87 * warps))
                         : (real ? std::max(0.75, 0.46 * warps) : std::max(0.65, 0.32 * warps));
    return 4.0 + 0.5 * m * row;
}

}  // namespace

bool split_plan(int prec, const AxisTables &ax, const SweepGeom &g, SplitPlan &p, bool increment)
{
    p = SplitPlan{};
    p.increment = increment;
    const bool d = prec == kC128, real = ax.kim != 0.0;
    const int win = d ? ax.win64 : ax.win32, conv = d ? ax.conv64 : ax.conv32, m = g.n - 1;
    if (prec == kCFF || win < 1 || conv > kSplitConv) return false;
    const long long lines = (long long)g.lines_a * g.lines_b;
    p.W = win + 1;
    p.x = g.pstride == 1;
    SplitPlan p16 = p;
    const bool ok8 = shape_plan(p, 8, conv, m, d, g);
    const bool ok16 = shape_plan(p16, 16, conv, m, d, g);
    if (!ok8 && !ok16) return false;
    // complex64: 8 rows a lane while more lanes mean less latency (128^3 y
    // sweep: 16.4 against 17.1 us), 16 where the windows' extra work counts
    // (256^3: 91 against 82 us; 2000 x 1500: 29 against 25 us)
    if (!d) {
        if (!ok8 || (ok16 && lines * m > 2500000)) p = p16;
        return true;
    }
    if (!ok8 || (ok16 && split_us(p16, real, lines) < split_us(p, real, lines))) p = p16;
    return split_us(p, real, lines) < pair_us(p.x, real, m, lines);
}

int split_blocks(const SplitPlan &p) { return (int)(p.grid_x * p.grid_y); }

int split_most_blocks(const SweepGeom &g)
{
    return g.pstride == 1 ? 0 : ((g.lines_a + 1) / 2) * g.lines_b;
}

cudaError_t launch_sweep_split(const SplitPlan &p, int prec, int mode, void *psi, const AxisTables &ax,
                               const SweepGeom &g, const NonlinArgs *nl, bool nl_at_output,
                               const Partials *norm_out, cudaStream_t st)
{
    if (prec == kC128) return launch<kFp64>(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
    if (p.increment) return launch<kIncrement>(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
    return launch<kTwoEnded>(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
}

}  // namespace gp
