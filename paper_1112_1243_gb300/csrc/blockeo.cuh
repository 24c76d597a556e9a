// Persistent block solver of the block filter (Eq. 4step step 1): per work
// item (block, factor) d = D_b[U_{i+1}]^{-1} (D_b[U_i] - D_b[U_{i+1}]) eta and
// -(2 Re<eta, d> + |d|^2), one thread block an item, items from a queue.
//
// D_b is solved in even-odd form inside the block: Dtilde = 1 - kappa^2 H_eo
// H_oe on the even sites, b~ = b_e + kappa H_eo b_o, x_o = b_o + kappa H_oe x_e;
// an FP32 BiCGStab inside a refinement whose residual b~ - Dtilde x has FP64
// accuracy (two-limb integers, xfix.cuh), relative to the whole right-hand
// side.  Half the sites and about half the iterations of the same solver on
// D_b itself.
//
// What bounded the form before (one FP32 BiCGStab on D_b, FP64 residual and
// FP64 sums; 2.8 ms a 4^4 block on two thread blocks an SM) was the FP64 pipe,
// 1.6 lanes a clock: sums converted and added component by component, the
// residual's stencil, the source from two FP64 links a hop, the noise.  Here
// the stencils are integer, sums are kept as pairs of FP32 numbers (48 bits)
// until the block has one, and only the noise, the vector updates of the
// refinement, the differences of links and the final sum are FP64.  4^4: 1024
// items 8.0 -> 4.7 ms (noise 9%, source 18%, FP32 iterations 53%, refinement
// 17%; at 25% of its issue slots, 15 warps an SM waiting for L2 and barriers).
//
// Vectors live in the thread block's scratch slot, component-major (component
// k of site i at [k * half + i]); FP32 work runs two lanes a site, lane pair
// (l, l + 16) of a warp holding spins 0 and 1 of the half spinors: a 4^4
// block has 128 sites a parity and fills 256 threads.
#pragma once

#include <cooperative_groups.h>

#include "blocksolve.cuh"
#include "dfhop.cuh"
#include "dslash.cuh"

// The thread blocks that work on one item: one, or the whole cluster of a
// large block (EO_COOP_SITES).  Warps are numbered through the team.
struct EoTeam {
    int rank, size;
    DD_DEV int warp() const { return rank * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5); }
    DD_DEV int warps() const { return size * (int)(blockDim.x >> 5); }
    // barrier of the team; writes before it, also to global memory, are visible after it
    DD_DEV void sync() const {
        if (size > 1)
            cooperative_groups::this_cluster().sync();
        else
            __syncthreads();
    }
};

struct EoSite {
    int l[4];
    int j;    // local lexicographic index
    int idx;  // storage index
};
// t-th site of parity par; false when there is none
DD_DEV bool eo_site(const EoCtx& c, int par, int t, EoSite& s) {
    if (t >= c.count) return false;
    const int q = fast_div(t, c.d0, c.m0), r0 = t - q * c.d0;
    const int q1 = fast_div(q, c.bd[1], c.m1);
    s.l[1] = q - q1 * c.bd[1];
    s.l[3] = fast_div(q1, c.bd[2], c.m2);
    s.l[2] = q1 - s.l[3] * c.bd[2];
    const int odd = (par + s.l[1] + s.l[2] + s.l[3]) & 1;
    s.l[0] = c.sh ? 2 * r0 + odd : r0;
    s.j = s.l[0] + c.bd[0] * q;
    s.idx = s.j >> c.sh;
    return c.sh || (s.l[0] & 1) == odd;
}
// index of site idx of parity par in arrays over the whole block
DD_DEV int eo_full(const EoCtx& c, int par, int idx) { return c.sh ? par * c.half + idx : idx; }

// ---------------------------------------------------------------- FP32 hops
// one hop of lane sp onto its sums: up (upper spin sp), lo / cross (lower
// spin 2 + sp of this line / of the other lane's line); see xfix.cuh for the
// spin structure.  Entries are read at a uniform base plus a 32-bit lane
// offset (bytes): ou / ol of the first upper / lower component, om of the
// link's first entry.
DD_DEV cpx<float> load32(const float2* base, int k, unsigned off) {
    const float2 v = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(base + k) + off);
    return mk<float>(v.x, v.y);
}
template <int AXIS, bool FWD>
DD_DEV void hop32_lane(int sp, const float2* in, int n, unsigned ou, unsigned ol, const float2* lk, int nb, unsigned om,
                       cpx<float>* up, cpx<float>* lo, cpx<float>* cross) {
    constexpr bool swap = AXIS < 2, rot = !(AXIS & 1);
    const float sg = FWD ? 1.f : -1.f;
    const float s1 = (AXIS == 1 || AXIS == 2) ? (sp ? -sg : sg) : sg;
    cpx<float> h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cpx<float> u = load32(in, c * n, ou), l = load32(in, c * n, ol);
        h[c] = rot ? mk<float>(fmaf(-s1, l.y, u.x), fmaf(s1, l.x, u.y)) : mk<float>(fmaf(s1, l.x, u.x), fmaf(s1, l.y, u.y));
    }
    cpx<float> m[3][3];
#pragma unroll
    for (int k = 0; k < 9; ++k) m[k / 3][k % 3] = load32(lk, (AXIS * 9 + k) * nb, om);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        cpx<float> v = mk<float>(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 3; ++j) v = FWD ? cmac(v, m[i][j], h[j]) : cmacc(v, m[j][i], h[j]);
        up[i] = up[i] + v;
        cpx<float>& d = swap ? cross[i] : lo[i];
        if (AXIS == 3)
            d = d + sg * v;
        else if (AXIS == 1)  // lower spins - sg (v1, -v0)
            d = d + (sp ? -sg : sg) * v;
        else {  // - sg i v (line 1 of axis 2 reversed)
            d.x = fmaf(s1, v.y, d.x);
            d.y = fmaf(-s1, v.x, d.y);
        }
    }
}

// the eight hops inside the block of one lane: res[0..2] upper spin sp,
// res[3..5] lower spin 2 + sp (both lanes of a site call this)
DD_DEV void hops32(const EoCtx& c, bool ok, int par, const EoSite& s, int sp, const float2* in, const float2* lk,
                   cpx<float>* res) {
    cpx<float> cross[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) res[i] = res[3 + i] = cross[i] = mk<float>(0.f, 0.f);
    const unsigned row = (unsigned)c.half * 8u;
    const unsigned up0 = 3u * sp * row, lo0 = 3u * (3 - sp) * row, lo1 = 3u * (2 + sp) * row;  // swapped, straight
    const unsigned own = (unsigned)eo_full(c, par, s.idx) * 8u, other = (unsigned)eo_full(c, 1 - par, 0) * 8u;
#define DD_HOP32(AXIS)                                                                                               \
    if (ok && s.l[AXIS] < c.bd[AXIS] - 1) {                                                                          \
        const unsigned y = (unsigned)((s.j + c.st[AXIS]) >> c.sh) * 8u;                                              \
        hop32_lane<AXIS, true>(sp, in, c.half, up0 + y, (AXIS < 2 ? lo0 : lo1) + y, lk, c.nb, own, res, res + 3,     \
                               cross);                                                                               \
    }                                                                                                                \
    if (ok && s.l[AXIS] > 0) {                                                                                       \
        const unsigned y = (unsigned)((s.j - c.st[AXIS]) >> c.sh) * 8u;                                              \
        hop32_lane<AXIS, false>(sp, in, c.half, up0 + y, (AXIS < 2 ? lo0 : lo1) + y, lk, c.nb, other + y, res,       \
                                res + 3, cross);                                                                     \
    }
    DD_HOP32(0)
    DD_HOP32(1)
    DD_HOP32(2)
    DD_HOP32(3)
#undef DD_HOP32
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        res[3 + i].x += __shfl_xor_sync(0xffffffffu, cross[i].x, 16);
        res[3 + i].y += __shfl_xor_sync(0xffffffffu, cross[i].y, 16);
    }
}

// component of lane sp: 0..2 upper, 3..5 lower
DD_DEV int lane_comp(int sp, int k) { return k < 3 ? 3 * sp + k : 3 + 3 * sp + k; }

// sums over the lanes' sites kept as (hi, lo) pairs of FP32 numbers
// (a CPU model of the sums at 4^4, 6^4 and 8^4: the bits of FP64 sums of the
// same FP32 products, whose own rounding leaves 1e-9 of the summed terms)
DD_DEV void df_acc(dfl& a, float t) {
    const float s = a.hi + t, bb = s - a.hi;
    a.lo += (a.hi - (s - bb)) + (t - bb);
    a.hi = s;
}
struct EoSums {
    dfl v[8];  // Re, Im <rhat, out>; Re, Im <out, in>; |out|^2; |in|^2; Re, Im <rhat, in>
};

// out = Dtilde in (th: odd temporary); with all all eight sums, else the first
// two.  Every thread of the team calls this; in is complete, out is written
// by the lanes that own its entries (no barrier at the end).
DD_DEV void eo_dtilde(const EoCtx& c, const EoTeam& T, const float2* in, float2* th, float2* out, const float2* lk,
                                       const float2* rhat, bool all, EoSums& S) {
    const int lane = threadIdx.x & 31, sp = lane >> 4, step = 16 * T.warps();
    const int first = 16 * T.warp();
    for (int t0 = first; t0 < c.count; t0 += step) {
        EoSite s;
        const bool ok = eo_site(c, 1, t0 + (lane & 15), s);
        cpx<float> r[6];
        hops32(c, ok, 1, s, sp, in, lk, r);
        if (ok)
#pragma unroll
            for (int k = 0; k < 6; ++k) th[lane_comp(sp, k) * c.half + s.idx] = make_float2(r[k].x, r[k].y);
    }
    T.sync();
#pragma unroll
    for (int k = 0; k < 8; ++k) S.v[k] = dfl{0.f, 0.f};
    for (int t0 = first; t0 < c.count; t0 += step) {
        EoSite s;
        const bool ok = eo_site(c, 0, t0 + (lane & 15), s);
        cpx<float> r[6];
        hops32(c, ok, 0, s, sp, th, lk, r);
        if (!ok) continue;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int at = lane_comp(sp, k) * c.half + s.idx;
            const float2 x = in[at], h = rhat[at];
            const float2 o = make_float2(fmaf(-c.kappa2, r[k].x, x.x), fmaf(-c.kappa2, r[k].y, x.y));
            out[at] = o;
            df_acc(S.v[0], h.x * o.x + h.y * o.y);
            df_acc(S.v[1], h.x * o.y - h.y * o.x);
            if (all) {
                df_acc(S.v[2], o.x * x.x + o.y * x.y);
                df_acc(S.v[3], o.x * x.y - o.y * x.x);
                df_acc(S.v[4], o.x * o.x + o.y * o.y);
                df_acc(S.v[5], x.x * x.x + x.y * x.y);
                df_acc(S.v[6], h.x * x.x + h.y * x.y);
                df_acc(S.v[7], h.x * x.y - h.y * x.x);
            }
        }
    }
}

constexpr int EO_CLUSTER = 8;  // thread blocks of a team
struct EoShared {
    dfl part[8][8];
    double tot[8];
    double all[EO_CLUSTER][8];  // the team's totals, by rank
    double sh[34];
    int ex[2][4][X_TILE], hs[2][X_TILE];
    int item;
};
// totals of the team from every thread block's M.tot (n values, set by the
// first threads), in a fixed order; valid in every thread
DD_DEV void eo_team_total(EoShared& M, const EoTeam& T, int n, double* out) {
    if (T.size > 1) {
        auto cl = cooperative_groups::this_cluster();
        for (int k = threadIdx.x; k < n * T.size; k += blockDim.x)
            cl.map_shared_rank(&M, k / n)->all[T.rank][k % n] = M.tot[k % n];
        cl.sync();
        for (int k = 0; k < n; ++k) {
            double t = 0.0;
            for (int r = 0; r < T.size; ++r) t += M.all[r][k];
            out[k] = t;
        }
        cl.sync();  // every rank has read before the next totals arrive
    } else {
        for (int k = 0; k < n; ++k) out[k] = M.tot[k];
    }
}
// sums of n pairs over the team, in FP64
DD_DEV void eo_total(EoShared& M, const EoTeam& T, const EoSums& S, int n, double* out) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k = 0; k < n; ++k) {
        dfl a = S.v[k];
        for (int o = 16; o; o >>= 1) {
            const dfl b{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
            df_acc(a, b.hi);
            a.lo += b.lo;
        }
        if (lane == 0) M.part[k][wid] = a;
    }
    __syncthreads();
    if (threadIdx.x < n) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += (double)M.part[threadIdx.x][w].hi + (double)M.part[threadIdx.x][w].lo;
        M.tot[threadIdx.x] = t;
    }
    __syncthreads();
    eo_team_total(M, T, n, out);
}
// sum of one FP64 value a thread over the team
DD_DEV double eo_sum(EoShared& M, const EoTeam& T, double v) {
    v = block_sum(v, M.sh);
    if (T.size == 1) return v;
    if (threadIdx.x == 0) M.tot[0] = v;
    __syncthreads();
    eo_team_total(M, T, 1, &v);
    return v;
}

// ------------------------------------------------ BiCGStab on Dtilde (FP32)
// x = 0, r holds the right-hand side.  Per iteration two operator
// applications with their sums, one pass for s and one for x, r and p: rho
// of the next iteration follows from <rhat, s> and <rhat, t>, |r|^2 from
// |s|^2, <t, s> and |t|^2, so the vector updates need no sums of their own.
// (<rhat, s> carried on as rho - alpha <rhat, v> kept the rounding of all
// iterations: near the critical mass, 8^4 blocks at kappa 0.16, some solves
// ran to their cap of 2000 iterations where 40 are enough.  The two sums more
// cost 4%: batch of 4^4, 6^4 and 8^4 blocks 15.06 -> 15.72 ms.)  Stops when
// |r|^2 <= tol2rel |r0|^2, after maxit iterations or at a breakdown (the
// refinement around it restarts from the true residual).
struct EoVecs {
    float2 *x, *r, *rhat, *p, *v, *s, *t, *th;
};
template <class F>
DD_DEV void eo_each(const EoCtx& c, const EoTeam& T, F f) {  // f(offset of a component of an even site owned by this lane)
    const int lane = threadIdx.x & 31, sp = lane >> 4, step = 16 * T.warps();
    for (int t0 = 16 * T.warp(); t0 < c.count; t0 += step) {
        EoSite s;
        if (!eo_site(c, 0, t0 + (lane & 15), s)) continue;
#pragma unroll
        for (int k = 0; k < 6; ++k) f(lane_comp(sp, k) * c.half + s.idx);
    }
}
DD_DEV int eo_bicgstab(const EoCtx& c, const EoTeam& T, EoShared& M, const EoVecs& V, const float2* lk, double tol2rel, int maxit) {
    EoSums S;
    dfl rr0{0.f, 0.f};
    eo_each(c, T, [&](int at) {
        const float2 r = V.r[at];
        V.x[at] = make_float2(0.f, 0.f);
        V.rhat[at] = V.p[at] = r;
        df_acc(rr0, r.x * r.x + r.y * r.y);
    });
    S.v[0] = rr0;
    double d[8];
    eo_total(M, T, S, 1, d);
    if (!(d[0] > 0.0)) return 0;
    T.sync();  // p complete
    const double target = tol2rel * d[0];
    cpx<double> rho = mk<double>(d[0], 0.0), alpha = mk<double>(0.0, 0.0);
    cpx<float> aR = mk<float>(0.f, 0.f);
    int it = 0;
    // two passes an iteration, v = Dtilde p and t = Dtilde s, with one copy
    // of the operator in the code
#pragma unroll 1
    for (bool second = false; second || it < maxit; second = !second) {
        eo_dtilde(c, T, second ? V.s : V.p, V.th, second ? V.t : V.v, lk, V.rhat, second, S);
        eo_total(M, T, S, second ? 8 : 2, d);
        if (!second) {
            const cpx<double> rv = mk<double>(d[0], d[1]);
            if (!(norm2(rv) > 0.0)) break;
            alpha = (1.0 / norm2(rv)) * cmul(rho, conj(rv));
            aR = mk<float>((float)alpha.x, (float)alpha.y);
            eo_each(c, T, [&](int at) {
                const float2 r = V.r[at], v = V.v[at];
                const cpx<float> w = mk<float>(r.x, r.y) - cmul(aR, mk<float>(v.x, v.y));
                V.s[at] = make_float2(w.x, w.y);
            });
            T.sync();
            continue;
        }
        ++it;
        const cpx<double> rt = mk<double>(d[0], d[1]), ts = mk<double>(d[2], d[3]);
        const double tt = d[4], ss = d[5];
        const bool stop_s = !(tt > 0.0) || ss <= target;  // s is the residual: x += alpha p
        const cpx<double> omega = stop_s ? mk<double>(0.0, 0.0) : (1.0 / tt) * ts;
        const cpx<float> wR = mk<float>((float)omega.x, (float)omega.y);
        const cpx<double> wd = mk<double>((double)wR.x, (double)wR.y);
        const double rr = ss - 2.0 * (wd.x * ts.x + wd.y * ts.y) + norm2(wd) * tt;
        const cpx<double> rho_new = mk<double>(d[6], d[7]) - cmul(wd, rt);
        cpx<double> beta = mk<double>(0.0, 0.0);
        bool last = stop_s || !(rr > target) || !(norm2(omega) > 0.0) || !(norm2(rho_new) > 0.0);
        if (!last) {
            // (rho_new / rho) (alpha / omega)
            beta = (1.0 / (norm2(rho) * norm2(omega))) * cmul(cmul(rho_new, conj(rho)), cmul(alpha, conj(omega)));
            last = !isfinite(beta.x) || !isfinite(beta.y);
        }
        const cpx<float> bR = mk<float>((float)beta.x, (float)beta.y);
        eo_each(c, T, [&](int at) {
            const float2 x2 = V.x[at], p2 = V.p[at], s2 = V.s[at];
            const cpx<float> p = mk<float>(p2.x, p2.y), s = mk<float>(s2.x, s2.y);
            const cpx<float> x = mk<float>(x2.x, x2.y) + cmul(aR, p) + cmul(wR, s);
            V.x[at] = make_float2(x.x, x.y);
            if (last) return;
            const float2 t2 = V.t[at], v2 = V.v[at];
            const cpx<float> r = s - cmul(wR, mk<float>(t2.x, t2.y));
            V.r[at] = make_float2(r.x, r.y);
            const cpx<float> q = r + cmul(bR, p - cmul(wR, mk<float>(v2.x, v2.y)));
            V.p[at] = make_float2(q.x, q.y);
        });
        if (last) break;
        rho = rho_new;
        T.sync();
    }
    return it;
}

// ------------------------------------------ FP64-accurate half hop (limbs)
struct EoX {
    int4* p;
    int* e;
};
// hops of in (parity 1 - par) onto the sites of parity par, four warps a tile
// of 32 sites (as hop_x_kernel): to limbs (xo.p given), or out = b1 - b2 +
// coef * hops (b2 may be null).  lx: links of the block, entries [a][9][nb],
// le: exponents [a][nb].  In is complete on entry, out on return (team barrier).
typedef long long EoPart[4][24][X_PAD];
__device__ __noinline__ void eo_xhop(const EoCtx c, const EoTeam T, EoShared& M, EoPart* part, int par, EoX in, const int4* lx,
                                     const int* le, EoX xo, double2* out, const double2* b1, const double2* b2,
                                     double coef) {
    const int lane = threadIdx.x & 31, wid = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), a = wid & 3;
    const int grp = wid >> 2, grp0 = T.rank * (blockDim.x >> 7), ngrp = T.size * (blockDim.x >> 7);
    const int ntile = (c.count + X_TILE - 1) / X_TILE;
    for (int tile0 = 0; tile0 < ntile; tile0 += ngrp) {
        const int tile = tile0 + grp0 + grp;
        EoSite s;
        const bool ok = eo_site(c, par, tile * X_TILE + lane, s);
        const int la = a == 0 ? s.l[0] : a == 1 ? s.l[1] : a == 2 ? s.l[2] : s.l[3];
        const bool okf = ok && la < c.bd[a] - 1, okb = ok && la > 0;
        const int yf = (s.j + c.st[a]) >> c.sh, yb = (s.j - c.st[a]) >> c.sh;
        const int kf = eo_full(c, par, s.idx), kb = eo_full(c, 1 - par, yb);
        const int ef = okf ? in.e[yf] + le[a * c.nb + kf] : 2 * X_ZERO, eb = okb ? in.e[yb] + le[a * c.nb + kb] : 2 * X_ZERO;
        M.ex[grp][a][lane] = max(ef, eb);
        if (a == 0) M.hs[grp][lane] = ok ? s.idx : -1;
        __syncthreads();
        {
            const int eout = max(max(M.ex[grp][0][lane], M.ex[grp][1][lane]), max(M.ex[grp][2][lane], M.ex[grp][3][lane]));
            const int4* lk = lx + (long long)a * 9 * c.nb;
            x_axis(a, false, okf, eout - ef, in.p, c.half, (unsigned)yf * 16u, lk, (unsigned)kf * 16u, false, okb,
                   eout - eb, (unsigned)yb * 16u, lk, (unsigned)kb * 16u, false, c.nb, part[grp][a], lane);
        }
        __syncthreads();
        const int i = 8 * a + (lane & 7), q = lane >> 3, idx = M.hs[grp][i];
        const int eout = max(max(M.ex[grp][0][i], M.ex[grp][1][i]), max(M.ex[grp][2][i], M.ex[grp][3][i]));
        xacc v[3];
        x_gather<false>(part[grp], i, q, v, nullptr);
        if (xo.p) {
            unsigned long long any = x_mag(v[0]) | x_mag(v[1]) | x_mag(v[2]);
            any |= __shfl_xor_sync(0xffffffffu, any, 8);
            any |= __shfl_xor_sync(0xffffffffu, any, 16);
            if (idx >= 0) {
                const int sh = x_norm_shift(any);
                if (q == 0) xo.e[idx] = x_norm_exponent(any, eout, sh);
#pragma unroll
                for (int k = 0; k < 3; ++k) xo.p[(3 * q + k) * c.half + idx] = x_normalise(v[k], sh);
            }
        } else if (idx >= 0) {
            const bool usual = abs(eout) < 900;
            const double f = usual ? __hiloint2double((eout - 56 + 1023) << 20, 0) * coef : coef;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int at = (3 * q + k) * c.half + idx;
                double2 w = b1[at];
                if (b2) {
                    const double2 u = b2[at];
                    w = make_double2(w.x - u.x, w.y - u.y);
                }
                const double2 z = usual ? make_double2((double)v[k].x, (double)v[k].y)
                                        : make_double2(x_to_double_any(v[k].x, eout), x_to_double_any(v[k].y, eout));
                out[at] = make_double2(fma(f, z.x, w.x), fma(f, z.y, w.y));
            }
        }
        __syncthreads();
    }
    T.sync();
}

// limbs of a spinor held by a lane pair (6 components each); every lane of
// the warp calls this
DD_DEV void eo_store_limbs(EoX x, int stride, int idx, int sp, bool ok, const cpx<double>* v) {
    XTop top;
    if (ok)
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            top.add(v[k].x);
            top.add(v[k].y);
        }
    int m = top.get();
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
    if (!ok) return;
    int E;
    const int e = x_exponent(m, E);
    if (sp == 0) x.e[idx] = e;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int2 a = x_split(x_from_double(v[k].x, E, 57)), b = x_split(x_from_double(v[k].y, E, 57));
        x.p[lane_comp(sp, k) * stride + idx] = make_int4(a.x, a.y, b.x, b.y);
    }
}

// ------------------------------------------------------------ the source
// (H_b[U_src] - H_b[U_sol]) eta at one site: only hops whose links differ
// contribute (the proposal changes active links only).  The difference of two
// links is taken in FP64 from the canonical fields and then put into limbs of
// its own scale: for a small rotation it lies far below the links, and limbs
// of the links (59 bits of the largest entry) would have few bits of it.  One
// lane a site.
struct EoSource {
    const double2 *u1, *u2;  // the two fields, canonical
    const uint8_t* active;   // [V * 4]
    Geo g;
    int org[4];
};
DD_DEV double2 link_diff(const EoSource& Q, long long k) {
    const double2 a = Q.u1[k], b = Q.u2[k];
    return make_double2(a.x - b.x, a.y - b.y);
}
__device__ __noinline__ void eo_source(const EoCtx c, const EoSource& Q, bool ok, int par, const EoSite& s, EoX eta,
                                       cpx<double>* b) {
    xacc acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k].x = acc[k].y = 0;
    int x[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) x[a] = Q.org[a] + s.l[a];
    const int site = ok ? canon_index(Q.g, x) : 0;
    auto hop_at = [&](int d, int& y, long long& lk) {  // eta index of the neighbour, first entry of the link
        const int a = d >> 1;
        const int la = a == 0 ? s.l[0] : a == 1 ? s.l[1] : a == 2 ? s.l[2] : s.l[3];
        if ((d & 1) ? la == 0 : la == c.bd[a] - 1) return false;
        const long long l = (long long)((d & 1) ? site - Q.g.st[a] : site) * 4 + a;
        if (!Q.active[l]) return false;
        y = eo_full(c, 1 - par, ((d & 1) ? s.j - c.st[a] : s.j + c.st[a]) >> c.sh);
        lk = l * 9;
        return true;
    };
    int eout = 2 * X_ZERO;
    int de[8];  // exponents of the differences, X_ZERO: no hop
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        int y;
        long long lk;
        de[d] = X_ZERO;
        if (!ok || !hop_at(d, y, lk)) continue;
        XTop top;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double2 v = link_diff(Q, lk + k);
            top.add(v.x);
            top.add(v.y);
        }
        int E;
        de[d] = x_exponent(top.get(), E);
        if (de[d] != X_ZERO) eout = max(eout, de[d] + eta.e[y]);
    }
    const bool use = eout != 2 * X_ZERO;
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        int y;
        long long lk;
        if (de[d] == X_ZERO || !hop_at(d, y, lk)) continue;
        const int a = d >> 1;
        const bool fwd = !(d & 1);
        xlimb h[6];
        x_project(a, !fwd, eta.p, c.nb, (unsigned)y * 16u, h);
        const int shift = min(eout - (de[d] + eta.e[y]), 62), E = de[d] + 1022;
        xacc v[6];
        // one body for U h and U^dag h: the adjoint's entries, conjugated
        x_multiply<true>(
            shift, h,
            [&](int k) {
                const double2 v = link_diff(Q, lk + (fwd ? k : 3 * (k % 3) + k / 3));
                const int2 re = x_split(x_from_double(v.x, E, 59));
                const int2 im = x_split(x_from_double(fwd ? v.y : -v.y, E, 59));
                return make_int4(re.x, re.y, im.x, im.y);
            },
            [&](int k, xacc w) { v[k] = w; });
        // upper spins, and the lower spins that belong to them (xfix.cuh)
        const long long m = fwd ? 0 : -1;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            acc[k].x += v[k].x;
            acc[k].y += v[k].y;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (a == 3) {
                acc[6 + k].x += x_neg_if(v[k].x, m);
                acc[6 + k].y += x_neg_if(v[k].y, m);
                acc[9 + k].x += x_neg_if(v[3 + k].x, m);
                acc[9 + k].y += x_neg_if(v[3 + k].y, m);
            } else if (a == 1) {
                acc[6 + k].x += x_neg_if(v[3 + k].x, ~m);
                acc[6 + k].y += x_neg_if(v[3 + k].y, ~m);
                acc[9 + k].x += x_neg_if(v[k].x, m);
                acc[9 + k].y += x_neg_if(v[k].y, m);
            } else {
                const int f0 = a == 0 ? 3 + k : k, f1 = a == 0 ? k : 3 + k;
                const long long m1 = a == 0 ? m : ~m;
                const xacc w0 = f0 < 3 ? v[k] : v[3 + k], w1 = f1 < 3 ? v[k] : v[3 + k];
                acc[6 + k].x += x_neg_if(w0.y, m);
                acc[6 + k].y += x_neg_if(w0.x, ~m);
                acc[9 + k].x += x_neg_if(w1.y, m1);
                acc[9 + k].y += x_neg_if(w1.x, ~m1);
            }
        }
    }
    const bool usual = abs(eout) < 900;
    const double f = usual ? __hiloint2double((eout - 56 + 1023) << 20, 0) * -c.kappa : -c.kappa;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 z = !use ? make_double2(0.0, 0.0)
                          : usual ? make_double2((double)acc[k].x, (double)acc[k].y)
                                  : make_double2(x_to_double_any(acc[k].x, eout), x_to_double_any(acc[k].y, eout));
        b[k] = mk<double>(f * z.x, f * z.y);
    }
}

template <bool BATCH>
__global__ void __launch_bounds__(256, 2) block_eo_kernel(BlockArgs A) {
    __shared__ EoShared M;
    extern __shared__ long long dyn[];
    EoPart* part = reinterpret_cast<EoPart*>(dyn);
    const int lane = threadIdx.x & 31, sp = lane >> 4;
    auto cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
    bool coop = A.nbig > 0;  // the items of the large blocks come first
    // every thread block of the cluster runs before one writes into another's
    // shared memory (the first item below)
    if (coop) cluster.sync();
    for (;;) {
        if (coop) {
            if (rank == 0 && threadIdx.x == 0) {
                const int u = atomicAdd(A.queue, 1);
                for (int r = 0; r < csize; ++r) cluster.map_shared_rank(&M, r)->item = u;
            }
            cluster.sync();
        } else {
            if (threadIdx.x == 0) M.item = A.nbig + atomicAdd(A.queue + 1, 1);
            __syncthreads();
        }
        const int item = M.item;
        const EoTeam T{coop ? rank : 0, coop ? csize : 1};
        T.sync();
        if (coop && item >= A.nbig) {
            coop = false;  // the same decision in every block of the cluster
            continue;
        }
        if (item >= A.nitems) break;
        const int wid = T.warp(), step = 16 * T.warps();
        char* base = A.scratch + (long long)(coop ? (int)blockIdx.x - rank : (int)blockIdx.x) * A.slot_bytes;
        const BlockItem it = BATCH ? A.items[item]
                                   : BlockItem{A.item_pos0 + item / A.item_n, item % A.item_n, item % A.item_n + 1,
                                               item % A.item_n, 0};
        const LatDesc& L = BATCH ? A.lats[it.lat] : A.lat;
        const EoCtx c = L.eo;
        const long long nb = c.nb, half = c.half;
        char* w = base;
        auto take = [&](size_t bytes) {
            char* p = w;
            w += (bytes + 15) & ~(size_t)15;
            return p;
        };
        double2* eta = (double2*)take(12 * nb * 16);
        double2 *bt = (double2*)take(12 * half * 16), *bo = (double2*)take(12 * half * 16),
                *x64 = (double2*)take(12 * half * 16), *r64 = (double2*)take(12 * half * 16);
        EoX px{(int4*)take(12 * half * 16), (int*)take(half * 4)}, tx{(int4*)take(12 * half * 16), (int*)take(half * 4)};
        EoVecs V;
        float2* f = (float2*)take(8 * 12 * half * 8);
        // limbs of eta, used before the FP32 vectors: their first half
        EoX ex{(int4*)f, (int*)(f + 2 * 12 * nb)};
        V.x = f;
        V.r = f + 12 * half;
        V.rhat = f + 24 * half;
        V.p = f + 36 * half;
        V.v = f + 48 * half;
        V.s = f + 60 * half;
        V.t = f + 72 * half;
        V.th = f + 84 * half;
        const long long lo = (long long)it.block_pos * 36 * nb, leo = (long long)it.block_pos * 4 * nb;
        const int4* lx = L.ddx + (long long)it.f_sol * L.ddx_fs + lo;
        const int* le = reinterpret_cast<const int*>(L.ddx + (long long)it.f_sol * L.ddx_fs + 36LL * L.g.V) + leo;
        const float2* l32 = L.dd32 + (long long)it.f_sol * L.dd32_fs + lo;
        int colour;
        const int id = block_id_at(L.g, it.block_pos, &colour);
        EoSource Q;
        Q.u1 = reinterpret_cast<const double2*>(L.canon + (long long)it.f_src * L.canon_fs);
        Q.u2 = reinterpret_cast<const double2*>(L.canon + (long long)it.f_sol * L.canon_fs);
        Q.active = L.active;
        Q.g = L.g;
        block_origin(L.g, id, Q.org);
        // ---- noise: two lanes a site, six complex Gaussians each
        for (int par = 0; par < 2; ++par)
            for (int t0 = 16 * wid; t0 < c.count; t0 += step) {
                EoSite s;
                const bool ok = eo_site(c, par, t0 + (lane & 15), s);
                cpx<double> v[6];
                const int at = ok ? eo_full(c, par, s.idx) : 0;
                if (ok) {
                    int x[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) x[a] = Q.org[a] + s.l[a];
                    const uint32_t site = (uint32_t)canon_index(L.g, x);
                    const uint64_t ctr = stream_ctr(A.ctr, A.ctr_off);
#pragma unroll 1
                    for (int k = 0; k < 6; ++k) {
                        const cpx<double> z = gaussian(site * 12u + lane_comp(sp, k), (uint32_t)A.purpose,
                                                       (uint32_t)it.vec, A.seed, ctr);
                        eta[lane_comp(sp, k) * nb + at] = make_double2(z.x, z.y);
                    }
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        const double2 z = eta[lane_comp(sp, k) * nb + at];
                        v[k] = mk<double>(z.x, z.y);
                    }
                }
                eo_store_limbs(ex, (int)nb, at, sp, ok, v);
            }
        T.sync();
        // ---- b = -kappa (H[src] - H[sol]) eta, |b|^2
        double bb = 0.0;
        for (int par = 0; par < 2; ++par)
            for (int t0 = 32 * wid; t0 < c.count; t0 += 2 * step) {
                EoSite s;
                const bool ok = eo_site(c, par, t0 + lane, s);
                if (!ok) continue;
                cpx<double> b[12];
                eo_source(c, Q, ok, par, s, ex, b);
                double2* o = par ? bo : bt;
                Spinor<double> sv;
#pragma unroll
                for (int k = 0; k < 12; ++k) {
                    o[k * half + s.idx] = make_double2(b[k].x, b[k].y);
                    sv.c[k] = b[k];
                    bb += norm2(b[k]);
                }
                if (par) SpinorX{tx.p, tx.e, half}.store(s.idx, sv);
            }
        bb = eo_sum(M, T, bb);
        T.sync();  // bt, bo and tx complete
        // ---- b~ = b_e + kappa H_eo b_o; x = 0, r = b~
        eo_xhop(c, T, M, part, 0, tx, lx, le, EoX{nullptr, nullptr}, bt, bt, nullptr, c.kappa);
        double rr = 0.0;
        eo_each(c, T, [&](int at) {
            const double2 v = bt[at];
            r64[at] = v;
            x64[at] = make_double2(0.0, 0.0);
            rr = fma(v.x, v.x, fma(v.y, v.y, rr));
        });
        for (int i = T.rank * (int)blockDim.x + threadIdx.x; i < half; i += T.size * (int)blockDim.x) px.e[i] = X_ZERO;
        rr = eo_sum(M, T, rr);
        int outer = 0;
        long long inner_its = 0;
        while (rr > A.tol2 * bb && outer < A.max_outer) {
            // inner right-hand side: the residual, normalised to unit norm
            const double rn = sqrt(rr), rinv = 1.0 / rn;
            eo_each(c, T, [&](int at) {
                const double2 v = r64[at];
                V.r[at] = make_float2((float)(rinv * v.x), (float)(rinv * v.y));
            });
            inner_its += eo_bicgstab(c, T, M, V, l32, A.tol2_inner, A.maxit_inner);
            // x += |r| e; r = b~ - Dtilde x
            for (int t0 = 16 * wid; t0 < c.count; t0 += step) {
                EoSite s;
                const bool ok = eo_site(c, 0, t0 + (lane & 15), s);
                cpx<double> v[6];
                if (ok)
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        const int at = lane_comp(sp, k) * (int)half + s.idx;
                        const double2 a = x64[at];
                        const float2 e = V.x[at];
                        v[k] = mk<double>(fma(rn, (double)e.x, a.x), fma(rn, (double)e.y, a.y));
                        x64[at] = make_double2(v[k].x, v[k].y);
                    }
                eo_store_limbs(px, (int)half, s.idx, sp, ok, v);
            }
            T.sync();
            eo_xhop(c, T, M, part, 1, px, lx, le, tx, nullptr, nullptr, nullptr, 0.0);
            eo_xhop(c, T, M, part, 0, tx, lx, le, EoX{nullptr, nullptr}, r64, bt, x64, c.kappa * c.kappa);
            rr = 0.0;
            eo_each(c, T, [&](int at) {
                const double2 v = r64[at];
                rr = fma(v.x, v.x, fma(v.y, v.y, rr));
            });
            rr = eo_sum(M, T, rr);
            ++outer;
        }
        if (T.rank == 0 && threadIdx.x == 0) {
            if (rr > A.tol2 * bb) raise_status(A.status, DD_ERR_NOT_CONVERGED);
            if (!isfinite(rr)) raise_status(A.status, DD_ERR_NUMERIC);
            if (A.stats) {
                atomicAdd(A.stats, 1ull);
                atomicAdd(A.stats + 1, (unsigned long long)inner_its);
                atomicAdd(A.stats + 2, (unsigned long long)outer);
                atomicAdd(A.stats + 3, (unsigned long long)inner_its * (unsigned long long)nb);
            }
        }
        // ---- x_o = b_o + kappa H_oe x_e, and the result
        if (bb == 0.0) {  // an unchanged block: d = 0
            if (T.rank == 0 && threadIdx.x == 0) L.item_out[item] = 0.0;
            T.sync();
            continue;
        }
        eo_xhop(c, T, M, part, 1, px, lx, le, EoX{nullptr, nullptr}, bt, bo, nullptr, c.kappa);
        double sum = 0.0;
        for (int par = 0; par < 2; ++par)
            for (int t0 = 16 * wid; t0 < c.count; t0 += step) {
                EoSite s;
                if (!eo_site(c, par, t0 + (lane & 15), s)) continue;
                const double2* d = par ? bt : x64;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const double2 e = eta[lane_comp(sp, k) * nb + eo_full(c, par, s.idx)],
                                  v = d[lane_comp(sp, k) * half + s.idx];
                    sum += 2.0 * (e.x * v.x + e.y * v.y) + (v.x * v.x + v.y * v.y);
                }
            }
        sum = eo_sum(M, T, sum);
        if (T.rank == 0 && threadIdx.x == 0) L.item_out[item] = -sum;
        T.sync();
    }
}

// The same items with everything in FP64 (dd_params.block_prec DD_PREC_F64):
// CG on the normal equations of D_b.
__global__ void __launch_bounds__(256, 2) block_solve64_kernel(BlockArgs A) {
    __shared__ double sh[34];
    __shared__ int s_item;
    // scratch slot of this thread block: vectors eta, b, x, r and the inner x, r, p, q, z
    char* base = A.scratch + (long long)blockIdx.x * A.slot_bytes;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(A.queue, 1);  // one queue
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= A.nitems) break;
        const BlockItem it = A.items ? A.items[item]
                                     : BlockItem{A.item_pos0 + item / A.item_n, item % A.item_n,
                                                 item % A.item_n + 1, item % A.item_n, 0};
        const LatDesc& L = A.lats ? A.lats[it.lat] : A.lat;
        const BlockCtx c = L.c;
        const long long nb = c.nb;
        auto vec = [&](int k) { return SpinorF64{(double2*)base + (long long)k * 12 * nb, nb}; };
        const SpinorF64 eta = vec(0), bv = vec(1), xv = vec(2), rv = vec(3), xi = vec(4), ri = vec(5), pi = vec(6),
                        qi = vec(7), zi = vec(8);
        int colour;
        int id = block_id_at(L.g, it.block_pos, &colour);
        int org[4];
        block_origin(L.g, id, org);
        const LinkCanonF64 lsol{L.canon + (long long)it.f_sol * L.canon_fs, L.g, c, {org[0], org[1], org[2], org[3]}};
        const LinkCanonF64 lsrc{L.canon + (long long)it.f_src * L.canon_fs, L.g, c, {org[0], org[1], org[2], org[3]}};
        // ---- right-hand side
        for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
            int l[4];
            local_coords(c, j, l);
            int x[4] = {org[0] + l[0], org[1] + l[1], org[2] + l[2], org[3] + l[3]};
            uint32_t s = (uint32_t)canon_index(L.g, x);
            Spinor<double> e;
#pragma unroll
            for (int k = 0; k < 12; ++k)
                e.c[k] = gaussian(s * 12u + k, (uint32_t)A.purpose, (uint32_t)it.vec, A.seed, stream_ctr(A.ctr, A.ctr_off));
            eta.store(j, e);
        }
        __syncthreads();
        // b = (D_b[src] - D_b[sol]) eta = -kappa (H[src] - H[sol]) eta; x = 0, r = b
        double bb = 0.0;
        for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
            Spinor<double> h1, z;
            dirichlet_hop_diff(c, j, eta, lsrc, lsol, h1);
#pragma unroll
            for (int k = 0; k < 12; ++k) h1.c[k] = (-c.kappa) * h1.c[k];
            bv.store(j, h1);
            rv.store(j, h1);
            zero(z);
            xv.store(j, z);
            bb += snorm2(h1);
        }
        bb = block_sum(bb, sh);
        double rr = bb;
        int outer = 0;
        long long inner_its = 0;
        while (rr > A.tol2 * bb && outer < A.max_outer) {
            // inner right-hand side: the FP64 residual, normalised to unit norm
            const double rn = sqrt(rr), rinv = 1.0 / rn;
            for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
                Spinor<double> v;
                rv.load(j, v);
#pragma unroll
                for (int k = 0; k < 12; ++k) v.c[k] = rinv * v.c[k];
                ri.store(j, v);
            }
            __syncthreads();
            inner_its += block_cgnr<double>(c, xi, ri, pi, qi, zi, lsol, A.tol2_inner, A.maxit_inner, sh);
            // x += |r| e; r = b - D_b x (FP64)
            for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
                Spinor<double> a;
                Spinor<double> e;
                xv.load(j, a);
                xi.load(j, e);
#pragma unroll
                for (int k = 0; k < 12; ++k)
                    a.c[k] = a.c[k] + rn * e.c[k];
                xv.store(j, a);
            }
            __syncthreads();
            rr = 0.0;
            for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
                Spinor<double> acc, v, b;
                dirichlet_hop<double>(c, j, xv, lsol, 0, acc);
                xv.load(j, v);
                bv.load(j, b);
#pragma unroll
                for (int k = 0; k < 12; ++k) b.c[k] = b.c[k] - (v.c[k] + (-c.kappa) * acc.c[k]);
                rv.store(j, b);
                rr += snorm2(b);
            }
            rr = block_sum(rr, sh);
            ++outer;
        }
        if (rr > A.tol2 * bb && threadIdx.x == 0) raise_status(A.status, DD_ERR_NOT_CONVERGED);
        if (A.stats && threadIdx.x == 0) {
            atomicAdd(A.stats, 1ull);
            atomicAdd(A.stats + 1, (unsigned long long)inner_its);
            atomicAdd(A.stats + 2, (unsigned long long)outer);
            atomicAdd(A.stats + 3, (unsigned long long)inner_its * (unsigned long long)nb);
        }
        if (!isfinite(rr) && threadIdx.x == 0) raise_status(A.status, DD_ERR_NUMERIC);
        // ---- result
        double s = 0.0;
        for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
            Spinor<double> e, d;
            eta.load(j, e);
            xv.load(j, d);
#pragma unroll
            for (int k = 0; k < 12; ++k) s += 2.0 * (e.c[k].x * d.c[k].x + e.c[k].y * d.c[k].y) + norm2(d.c[k]);
        }
        s = block_sum(s, sh);
        if (threadIdx.x == 0) L.item_out[item] = -s;
        __syncthreads();
    }
}
