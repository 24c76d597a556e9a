// Even-odd Wilson hopping kernel (Sec. 5, the unimproved Wilson-Dirac
// operator; Eq. domdec for the intra-/inter-block restrictions).
//
// One thread per output site of parity p:
//   out(x) = a * xin(x) + b * G5out( sum_hops (1 -+ gamma_a) U psi(x +- a) ),
// psi read from the opposite parity, optionally gamma5-multiplied on load.
// MASK = 0: all hops; 1: hops inside a block only (Dirichlet D_b); 2: only
// hops that cross a block face (D_bw, D_wb).  Links are stored per parity:
// the forward hop of x uses U_a(x) (parity p), the backward hop the link
// U_a(x - a) stored at the neighbour (parity 1 - p).
#pragma once

#include <algorithm>
#include <type_traits>

#include "dd_internal.h"
#include "reduce.cuh"
#include "xfix.cuh"

// per-rhs shifted copies of storage descriptors (contiguous per-rhs blocks)
DD_DEV SpinorF64 at_rhs(SpinorF64 s, int r) {
    s.p += (long long)r * 12 * s.stride;
    return s;
}
DD_DEV SpinorF32 at_rhs(SpinorF32 s, int r) {
    s.p += (long long)r * 6 * s.stride;
    return s;
}
DD_DEV SpinorF16 at_rhs(SpinorF16 s, int r) {
    s.p += (long long)r * 3 * s.stride;
    s.nrm += (long long)r * s.stride;
    return s;
}

// canonical FP64 spinors of the caller, stride sites a rhs: the whole lattice,
// or (half) the sites of one parity; AL: on 16-byte boundaries (the C ABI asks
// only for those of a double)
template <bool AL>
struct SpinorC {
    static constexpr bool aligned = AL;
    double* p;
    long long stride;
    int half;
};
template <bool AL>
DD_DEV SpinorC<AL> at_rhs(SpinorC<AL> s, int r) {
    s.p += (long long)r * 24 * s.stride;
    return s;
}
DD_DEV double2 load_entry(const SpinorF64& f, long long i) { return f.p[i]; }
DD_DEV void store_entry(const SpinorF64& f, long long i, double2 v) { f.p[i] = v; }
template <bool AL>
DD_DEV double2 load_entry(const SpinorC<AL>& f, long long i) {
    return load_c(f.p, i, AL);
}
template <bool AL>
DD_DEV void store_entry(const SpinorC<AL>& f, long long i, double2 v) {
    if (AL) {
        reinterpret_cast<double2*>(f.p)[i] = v;
    } else {
        f.p[2 * i] = v.x;
        f.p[2 * i + 1] = v.y;
    }
}
template <class S>
struct is_canonical : std::false_type {};
template <bool AL>
struct is_canonical<SpinorC<AL>> : std::true_type {};
// entry k of the site with even-odd index h and canonical index s
DD_DEV long long entry_at(const SpinorF64& f, int k, int h, int s) { return k * f.stride + h; }
template <bool AL>
DD_DEV long long entry_at(const SpinorC<AL>& f, int k, int h, int s) { return (long long)(f.half ? h : s) * 12 + k; }
DD_DEV long long entry_at(const SpinorX& f, int k, int h, int s) { return k * f.stride + h; }

template <class SIn, class SX, class SOut, class LK>
struct HopArgs {
    Geo g;
    int p;                    // output parity
    SIn in;                   // input field (parity 1 - p)
    SX xin;                   // a * xin term (parity p), used when has_x
    SOut out;                 // output (parity p)
    LK lk;                    // gauge field, both parities: [parity][dir][chunk][Vh]
    long long lk_rhs_stride;  // elements between the fields of consecutive rhs (0: shared)
    double a = 1.0;           // the FP64 hops take 1
    double b;
    int has_x;
    int g5in, g5out;
    int colour_mask;          // 3 = every site; else zero the output outside these block colours
    const CGState* st;        // per-rhs activity (may be null)
    Reduce red;               // |out|^2 reduction (red.op == FIN_NONE: off)
    unsigned long long* sites;  // timed launches: output sites processed (may be null)
    // BiCGStab's sums: 0 off; 1: <rhat, out>; 2: <out, xin>, |out|^2, <rh2, out>, |xin|^2 and <rh2, xin>
    int red3 = 0;
    SIn rh2;                    // red3 == 2: the shadow residual (hop storage)
    SX rhat;                    // red3 == 1: the shadow residual; resid: the right-hand side
    SiteSet S = {nullptr, -1};  // output sites (n < 0: all Vh sites of parity p)
    int resid = 0;              // FP64 hops: out = rhat - (xin + b * hops)
    int has2 = 0;               // FP64 hops: a second copy of out
    SOut out2;
    int both = 0;               // FP64 hops: both output parities in one launch (blockIdx.z), in2: the input of parity 1
    SIn in2;
    int ob[4] = {0, 0, 0, 0};   // MASK 2: hops that leave a block of these extents are dropped too (0: none)
    const double* U = nullptr;  // FP64 hops on canonical fields: the caller's links and the hop's input, for sites
    SX src;                     // with neighbours that are not finite (null: such a site is NaN as a whole)
};

template <class LK>
DD_DEV LK link_parity(LK lk, int par, long long Vh) {
    lk.p += (long long)par * 4 * LK::chunks * Vh;
    return lk;
}

template <class R, class SIn, class LK, int MASK>
DD_DEV void hop_site(const Geo& g, int p, int h, const int x[4], const SIn& in, const LK& lk_p, const LK& lk_q,
                     int g5in, Spinor<R>& acc) {
    zero(acc);
    const int s = canon_index(g, x);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        // local coordinate in the block (multiply-high division: b_a is not a compile-time constant)
        const int loc = x[a] - fast_div(x[a], g.b[a], g.mb[a]) * g.b[a];
        // forward: (1 - gamma_a) U_a(x) psi(x + a)
        bool okf = true, okb = true;
        if (MASK == 1) {
            okf = loc != g.b[a] - 1;
            okb = loc != 0;
        } else if (MASK == 2) {
            okf = loc == g.b[a] - 1;
            okb = loc == 0;
        }
        if (okf) {
            int yh = neighbour_index(g, s, x, a, +1) >> 1;
            Spinor<R> s;
            R w = in.load_unscaled(yh, s);
            if (g5in) gamma5(s);
            Half<R> hf, uh;
            project<R>(a, +1, s, hf);
            Link<R> u;
            lk_p.load(h, a, u);
            mul_link(u, hf, uh);
            R sc = (a == 3 && x[3] == g.L[3] - 1) ? (R)g.bc * w : w;
            accumulate<R>(a, +1, uh, sc, acc);
        }
        if (okb) {
            int yh = neighbour_index(g, s, x, a, -1) >> 1;
            Spinor<R> s;
            R w = in.load_unscaled(yh, s);
            if (g5in) gamma5(s);
            Half<R> hf, uh;
            project<R>(a, -1, s, hf);
            Link<R> u;
            lk_q.load(yh, a, u);
            mul_link_dag(u, hf, uh);
            R sc = (a == 3 && x[3] == 0) ? (R)g.bc * w : w;
            accumulate<R>(a, -1, uh, sc, acc);
        }
    }
}

// Each thread block covers SPT * blockDim.x consecutive entries of the site
// set (SPT passes of blockDim.x threads; thread block size and SPT are
// chosen by the autotuner, see dd_autotune).
template <class R, class SIn, class SX, class SOut, class LK, int MASK, int RED3, int SPT>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 7 : 0)
    hop_eo_kernel(HopArgs<SIn, SX, SOut, LK> A) {
    const int rhs = blockIdx.y;
    if (A.st && !A.st[rhs].active) return;
    const long long Vh = A.g.Vh;
    const long long tile = (long long)blockDim.x * SPT;
    if (A.sites && threadIdx.x == 0)
        atomicAdd(A.sites, (unsigned long long)min(tile, A.S.n - (long long)blockIdx.x * tile));
    double v3[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double nrm = 0.0;
#pragma unroll
    for (int pass = 0; pass < SPT; ++pass) {
        const long long t = (long long)blockIdx.x * tile + (long long)pass * blockDim.x + threadIdx.x;
        if (t >= A.S.n) break;
        int x[4];
        int h;
        if (A.S.colour >= 0) {
            h = colour_site(A.g, A.S.colour, (int)t, A.p, x);
        } else {
            h = (int)A.S.at(t);
            eo_coords(A.g, A.p, h, x);
        }
        const SIn in = at_rhs(A.in, rhs);
        LK lk = A.lk;
        lk.p += (long long)rhs * A.lk_rhs_stride;
        const LK lk_p = link_parity(lk, A.p, Vh);
        const LK lk_q = link_parity(lk, 1 - A.p, Vh);
        Spinor<R> acc;
        hop_site<R, SIn, LK, MASK>(A.g, A.p, h, x, in, lk_p, lk_q, A.g5in, acc);
        if (A.g5out) gamma5(acc);
        Spinor<R> res, xv;
        const R bb = (R)A.b;
        if (A.has_x) {
            at_rhs(A.xin, rhs).load(h, xv);
            const R aa = (R)A.a;
#pragma unroll
            for (int k = 0; k < 12; ++k) res.c[k] = aa * xv.c[k] + bb * acc.c[k];
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) res.c[k] = bb * acc.c[k];
        }
        if (A.colour_mask != 3 && !((A.colour_mask >> block_colour_of(A.g, x)) & 1)) zero(res);
        at_rhs(A.out, rhs).store(h, res);
        // per-site sums in the arithmetic precision, accumulated across sites
        // in FP64 by the grid reduction (FP64 adds per component would cost
        // more than the stencil on GB300's FP64 pipe)
        if (RED3 == 1) {
            Spinor<R> rv;
            at_rhs(A.rhat, rhs).load(h, rv);
            R d0 = 0, d1 = 0;
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                d0 += rv.c[k].x * res.c[k].x + rv.c[k].y * res.c[k].y;
                d1 += rv.c[k].x * res.c[k].y - rv.c[k].y * res.c[k].x;
            }
            v3[0] += (double)d0;
            v3[1] += (double)d1;
        } else if (RED3 == 2) {
            Spinor<R> rv;
            at_rhs(A.rh2, rhs).load(h, rv);
            R d0 = 0, d1 = 0, d2 = 0, d3 = 0, d4 = 0, d5 = 0;
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                d0 += res.c[k].x * xv.c[k].x + res.c[k].y * xv.c[k].y;
                d1 += res.c[k].x * xv.c[k].y - res.c[k].y * xv.c[k].x;
                d2 += rv.c[k].x * res.c[k].x + rv.c[k].y * res.c[k].y;
                d3 += rv.c[k].x * res.c[k].y - rv.c[k].y * res.c[k].x;
                d4 += rv.c[k].x * xv.c[k].x + rv.c[k].y * xv.c[k].y;
                d5 += rv.c[k].x * xv.c[k].y - rv.c[k].y * xv.c[k].x;
            }
            v3[0] += (double)d0;
            v3[1] += (double)d1;
            v3[2] += (double)snorm2(res);
            v3[3] += (double)d2;
            v3[4] += (double)d3;
            v3[5] += (double)snorm2(xv);
            v3[6] += (double)d4;
            v3[7] += (double)d5;
        } else {
            nrm += (double)snorm2(res);
        }
    }
    if (RED3) {
        grid_reduce_bi<RED3 == 1 ? 2 : 8>(A.red, rhs, v3);
    } else if (A.red.op != FIN_NONE) {
        grid_reduce(A.red, rhs, nrm);
    }
}

// FP64 hop on the two-limb integers of xfix.cuh (in: SpinorX, links: LinkX).
// SOut = SpinorX: out = hops; SOut = SpinorF64: out = (has_x ? xin : 0) + b *
// hops, or rhat - (xin + b * hops) with resid, and |out|^2 to A.red.
//
// A block of four warps takes 32 sites: warp w makes the two hops along axis
// w (a lane a site), leaves their sum and difference in shared memory, and
// all threads add up the axes (four lanes a site, one spin each).  A site is
// a chain of 4000 instructions: with all hops in one lane (128 registers, 16
// warps an SM) 2^20 sites took 537 us, 128 sites 21 us; here 508 and 10 us
// (8 x 16384 sites: 28 -> 15 us).  Two lanes a site with one spin each took
// 2.5 times the instructions and 830 us.  What is left is latency: 20 warps
// an SM (96 registers); at 2^19 sites DRAM at 50% and issue slots at 40% with
// out in limbs, 41% and 29% in the residual form.

// sum kept as a pair of FP64 numbers
struct Pair64 {
    double hi, lo;
    DD_DEV void add(double v, double err) {
        const double s = hi + v, b = s - hi;
        lo += (hi - (s - b)) + (v - b) + err;
        hi = s;
    }
    // + a (h + e)
    DD_DEV void mac(double a, double h, double e) {
        const double p = a * h;
        add(p, fma(a, e, fma(a, h, -p)));
    }
};
// The hops onto spin q of one site in FP64 arithmetic on the caller's fields
// (x: its coordinates).  The integer form has one exponent for a
// neighbourhood: it marks whole sites and links that hold a number that is
// not finite, and leaves few bits for entries far below the largest ones (a
// colour or spin that the links do not mix with a larger one).  For those
// this keeps what FP64 gives each component, of the colours in the bits of
// few.  PAIRS: projections and sums as pairs of FP64 numbers, one rounding of
// the result.
template <int MASK, bool AL, bool PAIRS>
__device__ __noinline__ void hop_canonical(const Geo& g, const int* x, const double* U, const SpinorC<AL>& in, int g5in,
                                           int q, int few, double2* out) {
    const int s = canon_index(g, x);
    const bool al16 = (reinterpret_cast<uintptr_t>(U) & 15) == 0;
    cpx<double> acc[3];
    Pair64 pr[3], pi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        acc[c] = mk<double>(0.0, 0.0);
        pr[c] = pi[c] = Pair64{0.0, 0.0};
    }
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        const int a = d >> 1, dir = (d & 1) ? -1 : 1;
        const int loc = x[a] - fast_div(x[a], g.b[a], g.mb[a]) * g.b[a];
        const bool face = loc == (dir > 0 ? g.b[a] - 1 : 0);
        if (MASK && (MASK == 1 ? face : !face)) continue;
        const int y = shift_index(g, x, a, dir);
        // line r of the projection: upper spin r, and the lower spin that meets it
        const int r = q < 2 ? q : (a < 2 ? 3 - q : q - 2), low = a < 2 ? 3 - r : 2 + r;
        // sign of i sigma_a on that line (times i for a = 0, 2)
        const bool rot = !(a & 1), neg = (a == 1 || a == 2) && r == 1;
        const double sl = (neg != (dir < 0)) != (g5in != 0) ? -1.0 : 1.0;
        cpx<double> h[3], e[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 u = load_entry(in, entry_at(in, 3 * r + c, y >> 1, y)),
                          l = load_entry(in, entry_at(in, 3 * low + c, y >> 1, y));
            const double lx = rot ? -sl * l.y : sl * l.x, ly = rot ? sl * l.x : sl * l.y;
            Pair64 hx{u.x, 0.0}, hy{u.y, 0.0};
            hx.add(lx, 0.0);
            hy.add(ly, 0.0);
            h[c] = mk<double>(hx.hi, hy.hi);
            e[c] = mk<double>(hx.lo, hy.lo);
        }
        const bool wrap = a == 3 && x[3] == (dir > 0 ? g.L[3] - 1 : 0);
        double sc = wrap ? (double)g.bc : 1.0;
        if (q > 1) {
            // lower spin q: - dir i sigma_a of the product, time + dir
            const bool lneg = (a == 1 || a == 2) && q == 3;
            if ((a == 3) == (dir < 0)) sc = -sc;
            if (lneg) sc = -sc;
        }
        const long long lk = ((long long)(dir > 0 ? s : y) * 4 + a) * 9;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (!((few >> i) & 1)) continue;
            cpx<double> v = mk<double>(0.0, 0.0);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const double2 w = load_c(U, lk + (dir > 0 ? 3 * i + j : 3 * j + i), al16);
                const cpx<double> m = mk<double>(w.x, dir > 0 ? w.y : -w.y);
                if (PAIRS) {
                    // sc m h, times i for a rotated lower spin
                    const bool turn = q > 1 && rot;
                    Pair64 &re = turn ? pi[i] : pr[i], &im = turn ? pr[i] : pi[i];
                    const double si = turn ? -sc : sc;
                    re.mac(sc * m.x, h[j].x, e[j].x);
                    re.mac(-sc * m.y, h[j].y, e[j].y);
                    im.mac(si * m.x, h[j].y, e[j].y);
                    im.mac(si * m.y, h[j].x, e[j].x);
                } else {
                    v = cmac(v, m, h[j]);
                }
            }
            if (!PAIRS) {
                if (q > 1 && rot) v = itimes(v);
                acc[i] = acc[i] + sc * v;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if ((few >> c) & 1)
            out[c] = PAIRS ? make_double2(pr[c].hi + pr[c].lo, pi[c].hi + pi[c].lo) : make_double2(acc[c].x, acc[c].y);
}

// Of the entries in the bits of few (hops all below 2^-3 of the largest
// product): those whose products are, too.  The hops may also be small
// because their products cancel, and then the integer form has the smaller
// error.  Sums of |link| |projected spinor|
// from the limbs in FP32, in units of the largest product 2^eout.  Bit 3 of
// the result: some lie above 2^-8, where FP64 products and sums would lose
// to the integer form in the error against the neighbourhood, and pairs of
// FP64 numbers keep both.  Random fields: the hops of one axis alone (sites
// at block corners, hops between blocks) get here, 1e-6 of the others.
template <int MASK>
__device__ __noinline__ int hop_few_bits(const Geo& g, const int* x, const SpinorX& in, const LinkX& lk, int par,
                                         int g5in, int q, int eout, int few) {
    const long long Vh = g.Vh;
    const int s = canon_index(g, x);
    const int* le = lk.exps();
    float sum[3] = {0.f, 0.f, 0.f};
    auto mag = [](int4 v) {
        return fabsf(fmaf((float)v.x, 0x1p30f, (float)v.y)) + fabsf(fmaf((float)v.z, 0x1p30f, (float)v.w));
    };
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        const int a = d >> 1, dir = (d & 1) ? -1 : 1;
        const int loc = x[a] - fast_div(x[a], g.b[a], g.mb[a]) * g.b[a];
        const bool face = loc == (dir > 0 ? g.b[a] - 1 : 0);
        if (MASK && (MASK == 1 ? face : !face)) continue;
        const int y = shift_index(g, x, a, dir) >> 1, row = (dir > 0 ? par : 1 - par) * 4 + a, at = dir > 0 ? s >> 1 : y;
        int e = in.e[y] + le[row * Vh + at];
        e -= x_wide_marks(e) * X_WIDE;
        if (e <= X_ZERO / 2) continue;
        const float scale = scalbnf(0x1p-116f, max(e - eout, -60) + 60);  // of limbs: 2^-57 2^-59, times 2^60
        xlimb h[6];
        x_project(a, (dir < 0) != (g5in != 0), in.p, in.stride, (unsigned)y * 16u, h);
        const int r = q < 2 ? q : (a < 2 ? 3 - q : q - 2);
        float hm[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const xlimb v = r ? h[3 + c] : h[c];
            hm[c] = mag(make_int4(v.rh, v.rl, v.ih, v.il)) * scale;
        }
        for (int c = 0; c < 3; ++c)
            if ((few >> c) & 1)
                for (int j = 0; j < 3; ++j) {
                    const int k = dir > 0 ? 3 * c + j : 3 * j + c;
                    sum[c] = fmaf(mag(x_load(lk.p + (long long)row * 9 * Vh, k * Vh, (unsigned)at * 16u)), hm[j], sum[c]);
                }
    }
    int found = 0;
    for (int c = 0; c < 3; ++c) {
        if (!((few >> c) & 1) || sum[c] >= 0x1p57f) continue;
        found |= 1 << c;
        if (sum[c] > 0x1p52f) found |= 8;
    }
    return found;
}

template <class SX, class SOut, int MASK>
__global__ void __launch_bounds__(128, 5) hop_x_kernel(HopArgs<SpinorX, SX, SOut, LinkX> A) {
    __shared__ long long part[4][24][X_PAD];  // axis; sum (0..11) and difference (12..23) of its hops
    __shared__ int ex[4][X_TILE], hs[X_TILE], ss[X_TILE];
    __shared__ unsigned char wide[4][X_TILE];  // X_WIDE marks of an axis
    constexpr bool canonical = is_canonical<SX>::value;
    const int rhs = blockIdx.y, par = A.both ? (int)blockIdx.z : A.p;
    if (A.st && !A.st[rhs].active) return;
    const Geo& g = A.g;
    const long long Vh = g.Vh;
    const int lane = threadIdx.x & 31, a = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);  // uniform in the warp
    const long long base = (long long)blockIdx.x * X_TILE;
    if (A.sites && threadIdx.x == 0) atomicAdd(A.sites, (unsigned long long)min((long long)X_TILE, A.S.n - base));
    auto site = [&](int i, int x[4]) -> int {  // even-odd index and coordinates of site i of the tile
        const long long t = min(base + i, A.S.n - 1);
        if (A.S.colour >= 0) return colour_site(g, A.S.colour, (int)t, par, x);
        const int h = (int)A.S.at(t);
        eo_coords(g, par, h, x);
        return h;
    };
    {
        int x[4];
        const int h = site(lane, x);
        const int s = canon_index(g, x);
        const SpinorX in = at_rhs((A.both && par) ? A.in2 : A.in, rhs);
        const int4* lk = A.lk.p + (long long)rhs * A.lk_rhs_stride;
        const int* le = LinkX{lk, A.lk.stride}.exps();
        const int xa = a == 0 ? x[0] : a == 1 ? x[1] : a == 2 ? x[2] : x[3];
        const int La = g.L[a], sa = g.st[a];
        const bool top = xa == La - 1, bottom = xa == 0;
        const int yf = (top ? s - (La - 1) * sa : s + sa) >> 1, yb = (bottom ? s + (La - 1) * sa : s - sa) >> 1;
        const long long rf = (long long)(par * 4 + a) * Vh + h, rb = (long long)((1 - par) * 4 + a) * Vh + yb;
        bool okf = true, okb = true;
        if (MASK) {
            const int loc = xa - fast_div(xa, g.b[a], g.mb[a]) * g.b[a];
            const bool ff = loc == g.b[a] - 1, fb = loc == 0;
            okf = MASK == 1 ? !ff : ff;
            okb = MASK == 1 ? !fb : fb;
            if (MASK == 2 && A.ob[a]) {
                const int lo = xa % A.ob[a];
                okf = okf && lo != A.ob[a] - 1;
                okb = okb && lo != 0;
            }
        }
        int ef = okf ? in.e[yf] + le[rf] : 2 * X_ZERO, eb = okb ? in.e[yb] + le[rb] : 2 * X_ZERO;
        if (canonical) {
            const int mf = x_wide_marks(ef), mb = x_wide_marks(eb);
            ef -= mf * X_WIDE;
            eb -= mb * X_WIDE;
            wide[a][lane] = (unsigned char)(mf | mb);
        }
        ex[a][lane] = max(ef, eb);
        if (a == 0) {
            hs[lane] = h;
            ss[lane] = s;
        }
        __syncthreads();
        const int eout = max(max(ex[0][lane], ex[1][lane]), max(ex[2][lane], ex[3][lane]));
        const bool phase = a == 3 && g.bc < 0;
        x_axis(a, A.g5in != 0, okf, eout - ef, in.p, in.stride, (unsigned)yf * 16u, lk + (long long)(par * 4 + a) * 9 * Vh,
               (unsigned)h * 16u, phase && top, okb, eout - eb, (unsigned)yb * 16u,
               lk + (long long)((1 - par) * 4 + a) * 9 * Vh, (unsigned)yb * 16u, phase && bottom, Vh, part[a], lane);
    }
    __syncthreads();
    const int i = 8 * a + (lane & 7), q = lane >> 3;  // spin q of site i
    const bool valid = base + i < A.S.n;
    const int h = hs[i], s = ss[i];
    const int eout = max(max(ex[0][i], ex[1][i]), max(ex[2][i], ex[3][i]));
    xacc v[3];
    int mag[3];
    x_gather<canonical>(part, i, q, v, mag);
    if constexpr (std::is_same<SOut, SpinorX>::value) {
        unsigned long long any = x_mag(v[0]) | x_mag(v[1]) | x_mag(v[2]);
        any |= __shfl_xor_sync(0xffffffffu, any, 8);
        any |= __shfl_xor_sync(0xffffffffu, any, 16);
        if (valid) {
            const SpinorX out = at_rhs(A.out, rhs);
            const int sh = x_norm_shift(any);
            if (q == 0) out.e[h] = x_norm_exponent(any, eout, sh);
#pragma unroll
            for (int c = 0; c < 3; ++c) out.p[(3 * q + c) * out.stride + h] = x_normalise(v[c], sh);
        }
    } else {
        double nrm = 0.0;
        if (valid) {
            bool zeroed = false;
            if (A.colour_mask != 3) {
                int x[4];
                site(i, x);
                zeroed = !((A.colour_mask >> block_colour_of(g, x)) & 1);
            }
            const SX xin = at_rhs(A.xin, rhs), bv = at_rhs(A.rhat, rhs);
            const SOut out = at_rhs(A.out, rhs);
            // sums times 2^(eout - 56) b: one multiplier where it is a normal
            // number (conversion and FMA run on the FP64 pipe beside the
            // integer pipes: 30 clocks a site)
            const double f0 = (q > 1 && A.g5out) ? -A.b : A.b;
            bool usual = abs(eout) < 900;
            double2 other[3];
            int few = 0;
            if constexpr (canonical) {
                if (A.U) {
                    if (eout >= X_BAD_MIN) {
                        few = 7;
                    } else if (min(min(mag[0], mag[1]), mag[2]) < X_SMALL && eout > X_ZERO / 2) {
                        few = x_small(part, i, q, mag, (wide[0][i] | wide[1][i] | wide[2][i] | wide[3][i]) != 0);
                        if (few) {
                            int x[4];
                            site(i, x);
                            few = hop_few_bits<MASK>(g, x, at_rhs((A.both && par) ? A.in2 : A.in, rhs),
                                                     LinkX{A.lk.p + (long long)rhs * A.lk_rhs_stride, A.lk.stride}, par,
                                                     A.g5in, q, eout, few);
                        }
                    }
                    usual = usual && !few;
                }
            }
            if (!usual) {
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    other[c] = make_double2(x_to_double_any(v[c].x, eout), x_to_double_any(v[c].y, eout));
                if constexpr (canonical) {
                    if (few) {
                        int x[4];
                        site(i, x);
                        if (few & 8)
                            hop_canonical<MASK, SX::aligned, true>(g, x, A.U, at_rhs(A.src, rhs), A.g5in, q, few, other);
                        else
                            hop_canonical<MASK, SX::aligned, false>(g, x, A.U, at_rhs(A.src, rhs), A.g5in, q, few, other);
                    }
                }
            }
            const double f = usual ? __hiloint2double((eout - 56 + 1023) << 20, 0) * f0 : f0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const long long k = entry_at(out, 3 * q + c, h, s);
                const double2 w = A.has_x ? load_entry(xin, k) : make_double2(0.0, 0.0);
                double2 z = make_double2((double)v[c].x, (double)v[c].y);
                if (!usual) z = other[c];
                z = make_double2(fma(f, z.x, w.x), fma(f, z.y, w.y));
                if (A.resid) {
                    const double2 w = load_entry(bv, k);
                    z = make_double2(w.x - z.x, w.y - z.y);
                }
                if (zeroed) z = make_double2(0.0, 0.0);
                store_entry(out, k, z);
                if (A.has2) store_entry(at_rhs(A.out2, rhs), k, z);
                if (A.red.op != FIN_NONE) nrm = fma(z.x, z.x, fma(z.y, z.y, nrm));
            }
        }
        if (A.red.op != FIN_NONE) grid_reduce(A.red, rhs, nrm);
    }
}

// timing class of a hop kernel instance (see dd_handle::timer_*), -1: not timed
template <class SIn, class SOut>
constexpr int hop_kind() {
    return std::is_same<SIn, SpinorF16>::value && std::is_same<SOut, SpinorF16>::value   ? 0
           : std::is_same<SIn, SpinorF16>::value && std::is_same<SOut, SpinorF32>::value ? 1
           : std::is_same<SIn, SpinorX>::value                                            ? 2
                                                                                          : -1;
}

template <class R, class SIn, class SX, class SOut, class LK, int MASK>
inline void launch_hop(const HopArgs<SIn, SX, SOut, LK>& A, int nrhs, dd_handle* h) {
    HopArgs<SIn, SX, SOut, LK> B = A;
    if (B.S.n < 0) B.S = SiteSet{nullptr, (long long)A.g.Vh};
    // tile shape from the handle's tuning (threads x sites per thread >= 32,
    // which keeps the grid within the reduction partials)
    constexpr bool f64 = std::is_same<SIn, SpinorX>::value;
    // four warps (hop_x_kernel), or the tuned shape within the kernels' launch bound
    const int tpb = f64 ? 128 : std::min(h->tune.hop_tpb, 128);
    const int spt = (!f64 && h->tune.hop_spt == 2) ? 2 : 1;
    dim3 grid(grid_for(B.S.n, f64 ? X_TILE : (long long)tpb * spt), nrhs, f64 && A.both ? 2 : 1);
    constexpr int kind0 = hop_kind<SIn, SOut>();
    // whole-lattice hops keep kinds 0-2; Dirichlet hops are timed as 4 (FP64),
    // 5, 6 (one block colour's sites) or 8, 9 (every site)
    constexpr int kindm = MASK == 0 ? kind0 : (MASK == 1 && kind0 >= 0 ? (kind0 == 2 ? 4 : 5 + kind0) : -1);
    const int kind = (MASK == 1 && kind0 >= 0 && kind0 < 2 && B.S.colour < 0) ? 8 + kind0 : kindm;
    bool timed = false;
    if (kind >= 0 && h->timer_on && !h->capturing && !dd_stream_capturing(h)) timed = (h->timer_seen[kind]++ % h->timer_every) == 0;
    B.sites = nullptr;
    if (timed) {
        cudaEvent_t e = dd_timer_event(h, kind);
        if (e) cudaEventRecord(e, h->stream);
        B.sites = h->d_sites + kind;
    }
    if constexpr (f64) {
        DD_KLAUNCH(h, hop_x_kernel<SX, SOut, MASK><<<grid, tpb, 0, h->stream>>>(B));
    } else if (A.red3 == 1)
        DD_KLAUNCH(h, (spt == 2 ? hop_eo_kernel<R, SIn, SX, SOut, LK, MASK, 1, 2> : hop_eo_kernel<R, SIn, SX, SOut, LK, MASK, 1, 1>)<<<grid, tpb, 0, h->stream>>>(B));
    else if (A.red3 == 2)
        DD_KLAUNCH(h, (spt == 2 ? hop_eo_kernel<R, SIn, SX, SOut, LK, MASK, 2, 2> : hop_eo_kernel<R, SIn, SX, SOut, LK, MASK, 2, 1>)<<<grid, tpb, 0, h->stream>>>(B));
    else
        DD_KLAUNCH(h, (spt == 2 ? hop_eo_kernel<R, SIn, SX, SOut, LK, MASK, 0, 2> : hop_eo_kernel<R, SIn, SX, SOut, LK, MASK, 0, 1>)<<<grid, tpb, 0, h->stream>>>(B));
    if (timed) {
        cudaEvent_t e = dd_timer_event(h, kind);
        if (e) cudaEventRecord(e, h->stream);
    }
}
