// FP64-accurate fields in two-limb integers, and the Wilson hop on them
// (Sec. 5, the unimproved Wilson-Dirac operator in FP64).
//
// GB300 has two FP64 lanes per SM (1.6 FMA per clock measured) but 64 lanes
// of 32 x 32 + 64 bit integer multiply-add (58 measured), so the FP64 hop
// was bound by its 900 FP64 instructions a site at a twentieth of the HBM
// rate.  Here every spinor is stored as 24 integers of 57 bits with one
// exponent per site, every link as 18 integers of 59 bits with one exponent,
// each integer split into two signed limbs, value = hi 2^30 + lo:
//   spinor  psi = (hi 2^30 + lo) 2^(e - 57),  |hi| <= 2^27, lo in [-2^29, 2^29)
//   link    u   = (hi 2^30 + lo) 2^(e - 59),  |hi| <= 2^29, lo in [-2^29, 2^29)
// A product is hi hi' + (hi lo' + lo hi') 2^-30 in units of 2^-56 of the
// two exponents (lo lo' lies below the last bit): three multiply-adds whose
// 64-bit sums are exact.  With the projection h = psi_upper +- psi_lower
// (limb by limb, |h_hi| <= 2^28, |h_lo| <= 2^30) the six terms of a colour
// sum stay below 6 x 2^57 (hi hi') and 7.5 x 2^59 (cross), and eight hops
// below 8 x 6 x 2^57 < 2^63, for any links and spinors.  Rounding errors are
// below 2^-55 of the largest entry around a site, FP64's own are about 2^-53
// of the summed terms: the integer form is the more accurate one.
// Entries that are not finite mark their site or link (X_BAD): every result
// they enter is NaN.  Subnormal entries count as zero.
//
// hop_x_kernel, one thread per output site, is bound by HBM (links 1184,
// spinors 196 + 192 bytes a site) and the 1728 multiply-adds (27 clocks a
// site of one SM at 64 lanes).  A runtime loop over the hops keeps it inside
// the instruction cache; exponents are read twice (the second time from L1)
// so that every hop is shifted to the largest exponent of the eight.
#pragma once

#include "dd_common.cuh"

constexpr int X_BAD = 1 << 26;      // exponent of a non-finite site or link
constexpr int X_BAD_MIN = 1 << 25;  // a sum of exponents with an X_BAD in it is above
constexpr int X_ZERO = -(1 << 24);  // exponent of an all-zero site or link

// 64-bit integer -> limbs (value = hi 2^30 + lo)
DD_DEV int2 x_split(long long v) {
    const int lo = (int)((unsigned)v << 2) >> 2;
    return make_int2((int)((v - lo) >> 30), lo);
}
// v 2^(bits + 1022 - E) rounded to an integer; E: biased exponent of the
// largest entry, so |result| <= 2^bits (53 <= bits <= 60)
DD_DEV long long x_from_double(double v, int E, int bits) {
    const int hi = __double2hiint(v);
    const int ex = (hi >> 20) & 0x7ff;
    unsigned long long m =
        ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(v);
    const int d = E - ex;
    m = (ex == 0 || d > 60) ? 0ull : (((m << (bits - 53)) + ((1ull << d) >> 1)) >> d);
    return hi < 0 ? -(long long)m : (long long)m;
}
// common exponent of n doubles from the OR-free maximum of their high words
// (sign cleared): the biased exponent E (0: nothing but zeros and
// subnormals) and the stored exponent
DD_DEV int x_exponent(int maxhi, int& E) {
    E = maxhi >> 20;
    return E == 0x7ff ? X_BAD : (E == 0 ? X_ZERO : E - 1022);
}
// acc 2^(e - 56) scaled by b: the multiplier where it is a normal number
// (one rounding), else false
DD_DEV bool x_scale(int e, double b, double& sc) {
    const int k = e - 56;
    if (k < -900 || k > 900) return false;
    sc = __hiloint2double((k + 1023) << 20, 0) * b;
    return true;
}

// Spinor in limbs: chunk k (spin * 3 + colour) of site i at p[k * stride + i]
// as (re.hi, re.lo, im.hi, im.lo), its exponent at e[i]
struct SpinorX {
    int4* p;
    int* e;
    long long stride;
    typedef double real;
    DD_DEV void store(long long i, const Spinor<double>& s) const {
        int m = 0;
#pragma unroll
        for (int k = 0; k < 12; ++k)
            m = max(m, max(__double2hiint(s.c[k].x) & 0x7fffffff, __double2hiint(s.c[k].y) & 0x7fffffff));
        int E;
        e[i] = x_exponent(m, E);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int2 a = x_split(x_from_double(s.c[k].x, E, 57)), b = x_split(x_from_double(s.c[k].y, E, 57));
            p[k * stride + i] = make_int4(a.x, a.y, b.x, b.y);
        }
    }
};
DD_DEV SpinorX at_rhs(SpinorX s, int r) {
    s.p += (long long)r * 12 * s.stride;
    s.e += (long long)r * s.stride;
    return s;
}

// Links in limbs, both parities: entry k (row 3, column) of link (parity,
// direction, h) at p[((parity * 4 + a) * 9 + k) * stride + h]; the exponents
// follow the 72 * stride chunks, at [(parity * 4 + a) * stride + h]
struct LinkX {
    const int4* p;
    long long stride;
    static constexpr int chunks = 9;
    // chunks of a whole field with its exponents
    static long long field_chunks(long long Vh) { return 72 * Vh + 2 * Vh; }
    DD_HD const int* exps() const { return reinterpret_cast<const int*>(p + 72 * stride); }
};
// one link, entries u[0..8] (re, im), into the formatted field
DD_DEV void x_store_link(int4* p, long long stride, int par, int a, long long h, const double* u) {
    int m = 0;
#pragma unroll
    for (int k = 0; k < 18; ++k) m = max(m, __double2hiint(u[k]) & 0x7fffffff);
    int E;
    reinterpret_cast<int*>(p + 72 * stride)[(long long)(par * 4 + a) * stride + h] = x_exponent(m, E);
    int4* o = p + (long long)(par * 4 + a) * 9 * stride + h;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int2 x = x_split(x_from_double(u[2 * k], E, 59)), y = x_split(x_from_double(u[2 * k + 1], E, 59));
        o[k * stride] = make_int4(x.x, x.y, y.x, y.y);
    }
}

// complex numbers of the hop: limbs of one projected component, and a
// 64-bit result
struct xlimb {
    int rh, rl, ih, il;
};
struct xacc {
    long long x, y;
};
DD_DEV long long x_neg_if(long long v, long long m) { return (v ^ m) - m; }  // m = 0 or -1

// a + s b limb by limb (m = 0: s = +1, m = -1: s = -1)
DD_DEV xlimb x_add(int4 a, int br_h, int br_l, int mr, int bi_h, int bi_l, int mi) {
    xlimb o;
    o.rh = a.x + (br_h ^ mr) - mr;
    o.rl = a.y + (br_l ^ mr) - mr;
    o.ih = a.z + (bi_h ^ mi) - mi;
    o.il = a.w + (bi_l ^ mi) - mi;
    return o;
}
// (i sigma_a v) for a = 0, 1, 2 acts on the spin pair by a swap of spins
// (a = 0, 1), a factor i (a = 0, 2) and signs; the time direction (a = 3)
// has the identity.  fac: spin 0 gets f0, spin 1 gets f1 = f0 or -f0.
//   a = 0: (i v1, i v0)   a = 1: (v1, -v0)   a = 2: (i v0, -i v1)   a = 3: (v0, v1)

// h = upper + sg (i sigma_a lower) (a = 3: upper + sg lower), m = 0 / -1 for sg = +1 / -1
DD_DEV void x_project(int a, int m, const SpinorX& in, long long y, xlimb* h) {
    const int4* p = in.p + y;
    const long long cs = in.stride;
    const int s0 = (a < 2) ? 9 : 6, s1 = 15 - s0;    // lower chunks that meet spin 0 and spin 1
    const int m1 = (a == 1 || a == 2) ? ~m : m;      // sign of the spin-1 line
    int4 u[6], l[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        u[c] = p[c * cs];
        u[3 + c] = p[(3 + c) * cs];
        l[c] = p[(s0 + c) * cs];
        l[3 + c] = p[(s1 + c) * cs];
    }
    if (a == 0 || a == 2) {  // + sg i z: (-z.y, z.x)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            h[c] = x_add(u[c], l[c].z, l[c].w, ~m, l[c].x, l[c].y, m);
            h[3 + c] = x_add(u[3 + c], l[3 + c].z, l[3 + c].w, ~m1, l[3 + c].x, l[3 + c].y, m1);
        }
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            h[c] = x_add(u[c], l[c].x, l[c].y, m, l[c].z, l[c].w, m);
            h[3 + c] = x_add(u[3 + c], l[3 + c].x, l[3 + c].y, m1, l[3 + c].z, l[3 + c].w, m1);
        }
    }
}

// acc += v on the upper spins, and the lower spins that belong to it:
// a = 3: + sg v, else - sg i sigma_a v
DD_DEV void x_accumulate(int a, long long m, const xacc* v, xacc* acc) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        acc[k].x += v[k].x;
        acc[k].y += v[k].y;
    }
    if (a == 3) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            acc[6 + k].x += x_neg_if(v[k].x, m);
            acc[6 + k].y += x_neg_if(v[k].y, m);
        }
    } else if (a == 1) {  // -sg (v1, -v0)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc[6 + c].x += x_neg_if(v[3 + c].x, ~m);
            acc[6 + c].y += x_neg_if(v[3 + c].y, ~m);
            acc[9 + c].x += x_neg_if(v[c].x, m);
            acc[9 + c].y += x_neg_if(v[c].y, m);
        }
    } else if (a == 0) {  // -sg (i v1, i v0), i z = (-z.y, z.x)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc[6 + c].x += x_neg_if(v[3 + c].y, m);
            acc[6 + c].y += x_neg_if(v[3 + c].x, ~m);
            acc[9 + c].x += x_neg_if(v[c].y, m);
            acc[9 + c].y += x_neg_if(v[c].x, ~m);
        }
    } else {  // -sg (i v0, -i v1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc[6 + c].x += x_neg_if(v[c].y, m);
            acc[6 + c].y += x_neg_if(v[c].x, ~m);
            acc[9 + c].x += x_neg_if(v[3 + c].y, ~m);
            acc[9 + c].y += x_neg_if(v[3 + c].x, m);
        }
    }
}

// One hop onto acc (24 integers in units of 2^(e_out - 56)).  lp: the link's
// first entry, cs its chunk stride; fwd: U h, else U^dag h; mg5: -1 when the
// input is taken with gamma5; flip: the hop carries the fermion phase -1;
// shift = e_out - (exponents of the link and the site).
DD_DEV void x_hop(int a, bool fwd, int mg5, bool flip, int shift, const SpinorX& in, long long y, const int4* lp,
                  long long cs, xacc* acc) {
    const int m = fwd ? 0 : -1;
    xlimb h[6];
    x_project(a, m ^ mg5, in, y, h);
    xacc v[6];
    const long long half = (1ll << shift) >> 1;  // the shift rounds to nearest (shift <= 62, |sums| < 2^61)
    const int mre = ~m, mim = m;  // signs of the link's imaginary part in the real and imaginary sums
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        xlimb u[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int4 w = lp[(fwd ? 3 * i + j : 3 * j + i) * cs];
            u[j] = xlimb{w.x, w.y, w.z, w.w};
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            long long hr = half, hi = half, cr = 1 << 29, ci = 1 << 29;  // cross sums rounded to nearest
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const xlimb w = h[3 * s + j];
                const int rih = (u[j].ih ^ mre) - mre, ril = (u[j].il ^ mre) - mre;
                const int iih = (u[j].ih ^ mim) - mim, iil = (u[j].il ^ mim) - mim;
                hr += (long long)u[j].rh * w.rh;
                hr += (long long)rih * w.ih;
                cr += (long long)u[j].rh * w.rl;
                cr += (long long)u[j].rl * w.rh;
                cr += (long long)rih * w.il;
                cr += (long long)ril * w.ih;
                hi += (long long)u[j].rh * w.ih;
                hi += (long long)iih * w.rh;
                ci += (long long)u[j].rh * w.il;
                ci += (long long)u[j].rl * w.ih;
                ci += (long long)iih * w.rl;
                ci += (long long)iil * w.rh;
            }
            v[3 * s + i].x = (hr + (cr >> 30)) >> shift;
            v[3 * s + i].y = (hi + (ci >> 30)) >> shift;
        }
    }
    if (flip) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            v[k].x = -v[k].x;
            v[k].y = -v[k].y;
        }
    }
    x_accumulate(a, m, v, acc);
}

// acc 2^(e - 56) -> limbs and exponent of an output spinor
DD_DEV void x_store_acc(const SpinorX& out, long long i, const xacc* acc, int e) {
    unsigned long long any = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k)
        any |= (unsigned long long)(acc[k].x ^ (acc[k].x >> 63)) | (unsigned long long)(acc[k].y ^ (acc[k].y >> 63));
    const int sh = any ? 7 - __clzll((long long)any) : 0;  // bits above 57
    const int r = max(sh, 0), l = max(-sh, 0);
    const long long half = r ? 1ll << (r - 1) : 0;
    out.e[i] = e >= X_BAD_MIN ? X_BAD : (any == 0 ? X_ZERO : e + 1 + sh);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int2 x = x_split(((acc[k].x + half) >> r) << l), y = x_split(((acc[k].y + half) >> r) << l);
        out.p[k * out.stride + i] = make_int4(x.x, x.y, y.x, y.y);
    }
}
