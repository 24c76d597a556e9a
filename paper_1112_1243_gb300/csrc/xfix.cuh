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
// below 8 x 6 x 2^57 < 2^63, for any links and spinors.
// Error, in units of 2^-56 of the largest product of a link and a spinor entry
// around a site: a hop drops at most 3 (lo lo'), rounds 1 away and takes 3.75
// from the rounding of its inputs, so eight hops stay below 62 units, 7.8 x
// 2^-53, in the worst case.  Relative to a component's own products random
// fields give at most 0.6 x 2^-53 (0.92 for the FP64 stencil).  This is a
// bound against the neighbourhood's largest numbers; a component far below
// them that the links do not mix with them has fewer bits.  The operators of
// the interface find such components and take them from FP64 arithmetic
// (hop_x_kernel, hop_canonical); inside the solvers, whose targets are norms,
// the bound serves as it is.
// Entries that are not finite mark their site or link (X_BAD): every result
// they enter is NaN.
#pragma once

#include "dd_common.cuh"

constexpr int X_BAD = 1 << 26;      // exponent of a non-finite site or link
constexpr int X_BAD_MIN = 1 << 25;  // a sum of exponents with an X_BAD in it is above
constexpr int X_ZERO = -(1 << 24);  // exponent of an all-zero site or link
constexpr int X_WIDE = 1 << 20;     // added where entries lie far below the largest (fields of the FP64 operators)
// marks in a sum of two exponents (0, 1 or 2), none in the special values
DD_DEV int x_wide_marks(int e) {
    const int k = (e + X_WIDE / 2) / X_WIDE;
    return e > 0 && k <= 2 ? k : 0;
}

// 64-bit integer -> limbs (value = hi 2^30 + lo)
DD_DEV int2 x_split(long long v) {
    const int lo = (int)((unsigned)v << 2) >> 2;
    return make_int2((int)((v - lo) >> 30), lo);
}
// v 2^(bits + 1022 - E) rounded to an integer; E: biased exponent of the
// largest entry, so |result| <= 2^bits (53 <= bits <= 60).  A subnormal number
// has the exponent 1 and no leading bit; E is below 1 where all entries are.
DD_DEV long long x_from_double(double v, int E, int bits) {
    const int hi = __double2hiint(v);
    const int ex = (hi >> 20) & 0x7ff;
    unsigned long long m =
        ((unsigned long long)((unsigned)(hi & 0xfffff) | (ex ? 0x100000u : 0u)) << 32) | (unsigned)__double2loint(v);
    const int d = max(E, 1) - max(ex, 1);
    m = d > 60 ? 0ull : (((m << (bits - 53 + max(1 - E, 0))) + ((1ull << d) >> 1)) >> d);
    return hi < 0 ? -(long long)m : (long long)m;
}
// Magnitude of the largest of a set of doubles: its high word (sign cleared);
// where all high words are 0, -32..-1 by the leading bit of the low words;
// X_NONE where every number is 0.  Larger values are larger numbers.
constexpr int X_NONE = -(1 << 30);
constexpr int X_WIDE_BITS = 24;
struct XTop {
    int m = 0;
    unsigned lo = 0;
    unsigned least = ~0u;  // add_wide: smallest high word of a number that is not 0, less 1
    DD_DEV void add(double v) {
        m = max(m, __double2hiint(v) & 0x7fffffff);
        lo |= (unsigned)__double2loint(v);
    }
    DD_DEV void add_wide(double v) {
        const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
        least = min(least, (hi | min((unsigned)__double2loint(v), 1u)) - 1u);
        add(v);
    }
    // entries that are not 0 far below the largest one: limbs of few bits, or 0
    DD_DEV bool wide() const {
        return least != ~0u && (least < (1u << 20) || (m >> 20) - (int)(least >> 20) > X_WIDE_BITS);
    }
    DD_DEV int get() const { return m ? m : (lo ? -1 - __clz((int)lo) : X_NONE); }
};
// biased exponent E of that magnitude (below 1: subnormal) and the stored exponent
DD_DEV int x_exponent(int top, int& E) {
    E = top >> 20;
    if (E < 1) E = top > 0 ? 12 - __clz(top) : (top == X_NONE ? 1 : top - 19);
    return E == 0x7ff ? X_BAD : (top == X_NONE ? X_ZERO : E - 1022);
}
// Spinor in limbs: chunk k (spin * 3 + colour) of site i at p[k * stride + i]
// as (re.hi, re.lo, im.hi, im.lo), its exponent at e[i]
struct SpinorX {
    int4* p;
    int* e;
    long long stride;
    typedef double real;
    // WIDE: mark a site with entries far below its largest (X_WIDE)
    template <bool WIDE = false>
    DD_DEV void store(long long i, const Spinor<double>& s) const {
        XTop top;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            if (WIDE) {
                top.add_wide(s.c[k].x);
                top.add_wide(s.c[k].y);
            } else {
                top.add(s.c[k].x);
                top.add(s.c[k].y);
            }
        }
        int E;
        e[i] = x_exponent(top.get(), E) + (WIDE && top.wide() ? X_WIDE : 0);
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
// one link, entries u[0..8] (re, im): entry k at p[k * stride], exponent at *e
DD_DEV void x_store_entries(int4* p, long long stride, int* e, const double* u, bool wide = false) {
    XTop top;
#pragma unroll
    for (int k = 0; k < 18; ++k) top.add_wide(u[k]);
    int E;
    *e = x_exponent(top.get(), E) + (wide && top.wide() ? X_WIDE : 0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int2 x = x_split(x_from_double(u[2 * k], E, 59)), y = x_split(x_from_double(u[2 * k + 1], E, 59));
        p[k * stride] = make_int4(x.x, x.y, y.x, y.y);
    }
}
// ... of a field in the layout of LinkX
DD_DEV void x_store_link(int4* p, long long stride, int par, int a, long long h, const double* u, bool wide) {
    x_store_entries(p + (long long)(par * 4 + a) * 9 * stride + h, stride,
                    reinterpret_cast<int*>(p + 72 * stride) + (long long)(par * 4 + a) * stride + h, u, wide);
}

// ------------------------------------------------------------ one hop
struct xlimb {
    int rh, rl, ih, il;
};
struct xacc {
    long long x, y;
};
DD_DEV long long x_neg_if(long long v, long long m) { return (v ^ m) - m; }  // m = 0 or -1

// line of three projected components: u + l or u - l (NEG), ROT: u +- i l
// with i z = (-z.y, z.x)
template <bool ROT>
DD_DEV void x_line(bool neg, const int4* u, const int4* l, xlimb* h) {
    if (neg) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            h[c] = ROT ? xlimb{u[c].x + l[c].z, u[c].y + l[c].w, u[c].z - l[c].x, u[c].w - l[c].y}
                       : xlimb{u[c].x - l[c].x, u[c].y - l[c].y, u[c].z - l[c].z, u[c].w - l[c].w};
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            h[c] = ROT ? xlimb{u[c].x - l[c].z, u[c].y - l[c].w, u[c].z + l[c].x, u[c].w + l[c].y}
                       : xlimb{u[c].x + l[c].x, u[c].y + l[c].y, u[c].z + l[c].z, u[c].w + l[c].w};
    }
}
// entry k of a field of entries 16 bytes wide: a uniform base plus a 32-bit
// lane offset (a parity has less than 2^28 sites), one address register a lane
DD_DEV int4 x_load(const int4* base, long long k, unsigned off) {
    return *reinterpret_cast<const int4*>(reinterpret_cast<const char*>(base + k) + off);
}
// (i sigma_a v) is, for a = 0: (i v1, i v0), 1: (v1, -v0), 2: (i v0, -i v1);
// the time direction (a = 3) has the identity: (v0, v1).

// h = upper + sg (i sigma_a lower) (a = 3: upper + sg lower), neg: sg = -1;
// entry k of the source spinor is x_load(base, k * cs, off).  a and neg are
// uniform in a warp.
DD_DEV void x_project(int a, bool neg, const int4* base, long long cs, unsigned off, xlimb* h) {
    const int s0 = (a < 2) ? 9 : 6, s1 = 15 - s0;            // lower entries that meet spin 0 and spin 1
    const bool neg1 = (a == 1 || a == 2) ? !neg : neg;       // sign of the spin-1 line
    int4 u[6], l[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        u[c] = x_load(base, c * cs, off);
        u[3 + c] = x_load(base, (3 + c) * cs, off);
        l[c] = x_load(base, (s0 + c) * cs, off);
        l[3 + c] = x_load(base, (s1 + c) * cs, off);
    }
    if (a & 1) {
        x_line<false>(neg, u, l, h);
        x_line<false>(neg1, u + 3, l + 3, h + 3);
    } else {
        x_line<true>(neg, u, l, h);
        x_line<true>(neg1, u + 3, l + 3, h + 3);
    }
}

// One row of the product of a link with one spin of h, in units of
// 2^(e_out - 56), e_out = shift + the exponents of link and source (shift
// 0..62).  u: the row's three entries; f, q: h's partners of the imaginary
// part in the real and imaginary sums, (-im, re) for U and (im, -re) for its
// adjoint; half = 2^(shift - 1): the shift rounds to nearest (|sums| < 2^61).
DD_DEV xacc x_row(const int4* u, const xlimb* h, const int2* f, const int2* q, long long half, int shift) {
    long long hr = half, hi = half, cr = 1 << 29, ci = 1 << 29;  // cross sums rounded to nearest
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        hr += (long long)u[j].x * h[j].rh;
        hi += (long long)u[j].x * h[j].ih;
        cr += (long long)u[j].x * h[j].rl;
        ci += (long long)u[j].x * h[j].il;
        hr += (long long)u[j].z * f[j].x;
        hi += (long long)u[j].z * q[j].x;
        cr += (long long)u[j].y * h[j].rh;
        ci += (long long)u[j].y * h[j].ih;
        cr += (long long)u[j].z * f[j].y;
        ci += (long long)u[j].z * q[j].y;
        cr += (long long)u[j].w * f[j].x;
        ci += (long long)u[j].w * q[j].x;
    }
    xacc v;
    v.x = (hr + (cr >> 30)) >> shift;
    v.y = (hi + (ci >> 30)) >> shift;
    return v;
}
// v = U h (FWD) or U^dag h; entry(k) = entry k of the link; put(k, value)
// receives entry k = 3 spin + colour
template <bool FWD, class Entry, class Put>
DD_DEV void x_multiply(int shift, const xlimb* h, Entry entry, Put put) {
    const long long half = (1ll << shift) >> 1;
    int2 f[6], q[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        f[k] = FWD ? make_int2(-h[k].ih, -h[k].il) : make_int2(h[k].ih, h[k].il);
        q[k] = FWD ? make_int2(h[k].rh, h[k].rl) : make_int2(-h[k].rh, -h[k].rl);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        int4 u[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) u[j] = entry(FWD ? 3 * i + j : 3 * j + i);
#pragma unroll
        for (int s = 0; s < 2; ++s) put(3 * s + i, x_row(u, h + 3 * s, f + 3 * s, q + 3 * s, half, shift));
    }
}

// The forward and backward hop along axis a of one site, a lane each site:
// sum (entries 0..11) and difference (12..23) of the products to part.  yf,
// yb: byte offsets of the neighbours in entry 0 of the source; kf, kb: of the
// links in entry 0 of the fields lf, lb; sf, sb: shifts (0 or more); flip:
// the hop carries the fermion phase -1.
constexpr int X_TILE = 32, X_PAD = 36;  // sites of a tile; padded row (two spins' reads meet different banks)
DD_DEV void x_axis(int a, bool g5, bool okf, int sf, const int4* src, long long cs, unsigned yf, const int4* lf,
                   unsigned kf, bool flipf, bool okb, int sb, unsigned yb, const int4* lb, unsigned kb, bool flipb,
                   long long cl, long long (*part)[X_PAD], int lane) {
    xacc vf[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) vf[k].x = vf[k].y = 0;
    if (okf) {
        xlimb h[6];
        x_project(a, g5, src, cs, yf, h);
        x_multiply<true>(min(sf, 62), h, [&](int k) { return x_load(lf, k * cl, kf); },
                         [&](int k, xacc v) { vf[k] = v; });
        if (flipf) {
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                vf[k].x = -vf[k].x;
                vf[k].y = -vf[k].y;
            }
        }
    }
    // a backward hop with the phase enters with the opposite sign: sum and
    // difference trade places
    const int ks = flipb ? 12 : 0, kd = 12 - ks;
    if (okb) {
        xlimb h[6];
        x_project(a, !g5, src, cs, yb, h);
        x_multiply<false>(min(sb, 62), h, [&](int k) { return x_load(lb, k * cl, kb); }, [&](int k, xacc v) {
            part[ks + 2 * k][lane] = vf[k].x + v.x;
            part[ks + 2 * k + 1][lane] = vf[k].y + v.y;
            part[kd + 2 * k][lane] = vf[k].x - v.x;
            part[kd + 2 * k + 1][lane] = vf[k].y - v.y;
        });
    } else {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            part[2 * k][lane] = part[12 + 2 * k][lane] = vf[k].x;
            part[2 * k + 1][lane] = part[13 + 2 * k][lane] = vf[k].y;
        }
    }
}
// high word of |v| (of -v - 1 for a negative one)
DD_DEV int x_mag_hi(long long v) {
    const int h = (int)(v >> 32);
    return h ^ (h >> 31);
}
// spin q of site i from the four axes: the sums of the hops' upper spins, and
// what they give to the lower ones, - i sigma_a (forward - backward), time:
// + the difference.  MAG: mag[c] the OR of the high words of the numbers that
// entry c is made of.
template <bool MAG>
DD_DEV void x_gather(const long long (*part)[24][X_PAD], int i, int q, xacc* v, int* mag) {
    const int r = q & 1;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int own = 2 * (3 * r + c), other = 2 * (3 * (1 - r) + c);
        if (q < 2) {
            xacc p[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) p[a] = xacc{part[a][own][i], part[a][own + 1][i]};
            v[c].x = p[0].x + p[1].x + p[2].x + p[3].x;
            v[c].y = p[0].y + p[1].y + p[2].y + p[3].y;
            if (MAG) {
                mag[c] = 0;
#pragma unroll
                for (int a = 0; a < 4; ++a) mag[c] |= x_mag_hi(p[a].x) | x_mag_hi(p[a].y);
            }
        } else {
            const long long (*d0)[X_PAD] = part[0] + 12, (*d1)[X_PAD] = part[1] + 12, (*d2)[X_PAD] = part[2] + 12,
                            (*d3)[X_PAD] = part[3] + 12;
            const long long m = r ? -1 : 0;
            const xacc p0{d0[other][i], d0[other + 1][i]}, p1{d1[other][i], d1[other + 1][i]},
                p2{d2[own][i], d2[own + 1][i]}, p3{d3[own][i], d3[own + 1][i]};
            v[c].x = p0.y + x_neg_if(p1.x, ~m) + x_neg_if(p2.y, m) + p3.x;
            v[c].y = -p0.x + x_neg_if(p1.y, ~m) + x_neg_if(p2.x, ~m) + p3.y;
            if (MAG)
                mag[c] = x_mag_hi(p0.x) | x_mag_hi(p0.y) | x_mag_hi(p1.x) | x_mag_hi(p1.y) | x_mag_hi(p2.x) |
                         x_mag_hi(p2.y) | x_mag_hi(p3.x) | x_mag_hi(p3.y);
        }
    }
}
// Entries (a bit each) that the common exponent of their neighbourhood leaves
// few bits for: those whose hops are all below 2^53 in units of 2^-56 of the
// largest product, 2^-3 of it (X_SMALL: the high word).  Above the line the
// integer form's error is within a few units of 2^-53 of the entry's own
// hops, as FP64's is.  The sums (upper spins) or differences (lower spins) of
// forward and backward hops that x_gather reads may be small where the hops
// are not, so this looks at both; rarely called (random fields: 4e-4 of the
// sites).  Hops that are all 0 are just that, unless a number near them is so
// far below the others that its limbs are 0 (wide).
constexpr int X_SMALL = 1 << 21;
static __device__ __noinline__ int x_small(const long long (*part)[24][X_PAD], int i, int q, const int* mag, bool wide) {
    const int r = q & 1;
    int found = 0;
    for (int c = 0; c < 3; ++c) {
        if (mag[c] >= X_SMALL) continue;
        int m = 0;
        long long any = 0;
        for (int a = 0; a < 4; ++a) {
            const int k = 2 * (3 * (q > 1 && a < 2 ? 1 - r : r) + c);
            for (int e = 0; e < 2; ++e) {
                m |= x_mag_hi(part[a][k + e][i]) | x_mag_hi(part[a][k + e + 12][i]);
                any |= part[a][k + e][i] | part[a][k + e + 12][i];
            }
        }
        if (m < X_SMALL && (any || wide)) found |= 1 << c;
    }
    return found;
}

// magnitude bits of a set of sums: OR of these, then x_bits
DD_DEV unsigned long long x_mag(xacc v) {
    return (unsigned long long)(v.x ^ (v.x >> 63)) | (unsigned long long)(v.y ^ (v.y >> 63));
}
// right (> 0) or left shift that brings sums with magnitude bits `any` to 57 bits
DD_DEV int x_norm_shift(unsigned long long any) { return any ? 7 - __clzll((long long)any) : 0; }
DD_DEV int x_norm_exponent(unsigned long long any, int e, int sh) {
    return e >= X_BAD_MIN ? X_BAD : (any == 0 ? X_ZERO : e + 1 + sh);
}
DD_DEV int4 x_normalise(xacc v, int sh) {
    const int r = max(sh, 0), l = max(-sh, 0);
    const long long half = (1ll << r) >> 1;
    const int2 x = x_split(((v.x + half) >> r) << l), y = x_split(((v.y + half) >> r) << l);
    return make_int4(x.x, x.y, y.x, y.y);
}

// v 2^(e - 56) for any exponent: subnormal results, and NaN where a source or
// link was not finite
static __device__ __noinline__ double x_to_double_any(long long v, int e) {
    if (e >= X_BAD_MIN) return __longlong_as_double(0x7ff8000000000000ll);
    return e <= X_ZERO / 2 ? 0.0 : scalbn((double)v, e - 56);
}
