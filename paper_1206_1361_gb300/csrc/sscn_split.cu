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
// time.  (Where kappa is small enough, sscn_inc.cu computes the same sweep's
// increment on the FP32 pipe instead.)
//
// Measured (GB300, us a step): 500 x 384 FP64 imaginary 385 -> 31, 64^3 71 -> 43;
// complex64 193 x 130 x 97 139 -> 58, 64^3 46 (TMA 44) -> 17.
//
// complex64 keeps the arithmetic and the direction of the kernels it stands in
// for (a state's observables are reported in FP64, where another order of FP32
// roundings shows): each half of a line (k_sweep, one middle row), or the whole
// line (k_sweep_tma: increment form, one direction), is cut into runs of at
// most P rows, and a lane runs the elimination over W rows before its run and
// the back substitution over W rows after it as well.  Once the dropped carry
// is below the last bit, the recurrences produce those kernels' bits.

#include "sscn_split.cuh"

namespace gp {
namespace sp {

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

}  // namespace sp

using namespace gp::sp;

namespace {

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
    stage_coefs<MODE>(a, smem_raw);
    pdl_wait();
    if (P3 && threadIdx.x == 0) g_of_step = a.sg.value();
    if (NL && !P3)
        for (int q = threadIdx.x; q < rows; q += blockDim.x) {
            const int L = line0 + q;
            row_nl[q].setup(a.px, a.py, a.pz, a.tx, a.ty, a.tz, L % a.lines_a, L / a.lines_a, a.sg.value(),
                            a.scale);
        }
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
    stage_coefs<MODE>(a, smem_raw);
    pdl_wait();
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
        block_partial(active ? part : 0.0, red, &a.partials[(long long)blockIdx.y * gridDim.x + blockIdx.x]);
    }
}

template <int FORM, int MODE, bool NL, bool P3, int P, typename T>
cudaError_t go_x(const SplitPlan &p, const SplitArgs<T> &a, cudaStream_t st)
{
    auto kern = k_split_x<FORM, MODE, NL, P3, P>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(p.after, kern, p.grid_x, p.threads, p.smem, st, a);
}

template <int FORM, int MODE, bool NORM, bool NLOUT, bool P3, int P, typename T>
cudaError_t go_yz(const SplitPlan &p, const SplitArgs<T> &a, cudaStream_t st)
{
    auto kern = k_split_yz<FORM, MODE, NORM, NLOUT, P3, P>;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(p.after, kern, dim3(p.grid_x, p.grid_y), p.threads, p.smem, st, a);
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
    const auto a = split_args<FORM>(p, mode, psi, ax, g, nl, norm_out);
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
    const size_t tables = d ? coef_bytes<double>(conv) + (p.increment ? inc_extra_smem(conv) : 0)
                            : coef_bytes<float>(conv);
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
        while (per > 2 && (lanes * per > (p.increment && d ? 256 : kSplitThreads) || per * line > 64 * 1024)) per /= 2;
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
    p.after = ax.settled;
    if (d) {
        // float-float increments where kappa allows them, whatever the number
        // of lines
        p.increment = increment && inc_applies(ax);
        if (p.increment && shape_plan(p, 8, conv, m, d, g)) return true;
        p.increment = false;
    }
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
    if (prec == kC128 && p.increment)
        return launch_sweep_inc(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
    if (prec == kC128) return launch<kFp64>(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
    if (p.increment) return launch<kIncrement>(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
    return launch<kTwoEnded>(p, mode, psi, ax, g, nl, nl_at_output, norm_out, st);
}

}  // namespace gp
