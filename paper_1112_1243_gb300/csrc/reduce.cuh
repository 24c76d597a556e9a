// Deterministic two-stage grid reduction with a finisher run by the last
// thread block (ticket counter), so that Krylov scalars are formed on the
// device without a host round trip.  Partial sums are FP64; the final sum is
// taken in a fixed order, so results do not depend on block scheduling.
#pragma once

#include "dd_internal.h"

DD_DEV void finish(const Reduce& R, int rhs, double s) {
    switch (R.op) {
        case FIN_STORE:
            R.out[rhs] = s;
            break;
        case FIN_OUTER: {  // defect correction: active while |r|^2 > tol2
            // a non-finite true residual ends the system and is reported as NUMERIC
            CGState& c = R.st[rhs];
            R.out[rhs] = s;
            c.rr = s;
            if (!isfinite(s)) {
                c.active = 0;
                c.flags |= 2;
                raise_status(R.status, DD_ERR_NUMERIC);
            } else {
                c.active = c.active && s > c.tol2;
            }
            break;
        }
        case FIN_ALPHA: {  // alpha = zz / |A p|^2
            CGState& c = R.st[rhs];
            c.qq = s;
            double a = c.zz / s;
            if (!(s > 0.0) || !isfinite(a)) {
                c.alpha = 0.0;
                c.active = 0;
                c.flags |= 2;
                raise_status(R.status, DD_ERR_NUMERIC);
            } else {
                c.alpha = a;
            }
            break;
        }
        case FIN_RR: {  // convergence test on the recursive residual
            CGState& c = R.st[rhs];
            c.rr = s;
            c.iters += 1;
            if (!isfinite(s)) {
                c.active = 0;
                c.flags |= 2;
                raise_status(R.status, DD_ERR_NUMERIC);
            } else if (s <= c.tol2) {
                c.active = 0;
            } else if (c.iters >= c.maxit) {
                c.active = 0;
                c.flags |= 1;
            }
            break;
        }
        case FIN_BETA: {  // beta = |z_new|^2 / |z_old|^2
            CGState& c = R.st[rhs];
            c.beta = (c.zz > 0.0) ? s / c.zz : 0.0;
            c.zz = s;
            break;
        }
        case FIN_ZZ_INIT: {  // first z: p = z, beta = 0
            CGState& c = R.st[rhs];
            c.zz = s;
            c.beta = 0.0;
            if (!(s > 0.0)) c.active = 0;  // zero right-hand side: nothing to do
            break;
        }
        default:
            break;
    }
}

// BiCGStab finishers on two, three or eight sums; complex scalars z = (re, im)
DD_DEV void cdiv(double ar, double ai, double br, double bi, double& cr, double& ci) {
    double d = br * br + bi * bi;
    cr = (ar * br + ai * bi) / d;
    ci = (ai * br - ar * bi) / d;
}
// A zero denominator (Lanczos breakdown) ends the inner solve quietly: the
// outer FP64 loop restarts from the true residual.  Non-finite values are
// reported in the status word.
DD_DEV void bicg_fail(const Reduce& R, CGState& c, bool numeric = false) {
    c.active = 0;
    c.flags |= 4;
    if (numeric) {
        c.flags |= 2;
        raise_status(R.status, DD_ERR_NUMERIC);
    }
}
DD_DEV void finish3(const Reduce& R, int rhs, const double* s) {
    CGState& c = R.st[rhs];
    switch (R.op) {
        case FIN_BI_RHO: {  // s = (Re<rh,r>, Im<rh,r>, |r|^2) of the start; counts as the first iteration
            c.rr = s[2];
            c.iters += 1;
            c.rho_re = s[0];
            c.rho_im = s[1];
            if (!isfinite(s[2]) || !isfinite(s[0]) || !isfinite(s[1])) {
                bicg_fail(R, c, true);
            } else if (s[2] <= c.tol2) {
                c.active = 0;
            } else if (c.iters >= c.maxit) {
                c.active = 0;
                c.flags |= 1;
            } else if (!(s[0] * s[0] + s[1] * s[1] > 0.0)) {
                bicg_fail(R, c);
            }
            break;
        }
        case FIN_BI_ALPHA: {  // s = (Re<rh,v>, Im<rh,v>): alpha = rho / <rh,v>
            double ar, ai;
            if (!isfinite(s[0]) || !isfinite(s[1])) {
                bicg_fail(R, c, true);
                break;
            }
            if (!(s[0] * s[0] + s[1] * s[1] > 0.0)) {
                bicg_fail(R, c);
                break;
            }
            cdiv(c.rho_re, c.rho_im, s[0], s[1], ar, ai);
            c.al_re = ar;
            c.al_im = ai;
            if (!isfinite(ar) || !isfinite(ai)) bicg_fail(R, c);
            break;
        }
        // omega = <t,s> / |t|^2, then everything of the next iteration that
        // the vector updates x += alpha p + omega s, r = s - omega t, p = r +
        // beta (p - omega v) need: |r|^2 = |s|^2 - 2 Re(conj(omega) <t,s>) +
        // |omega|^2 |t|^2 and rho' = <rh,s> - omega <rh,t>, with omega as the
        // updates take it (rounded to FP32).  The updates then need no sums of
        // their own.  <rh,s> is a sum of the vectors, not rho - alpha <rh,v>:
        // rho then kept the rounding of every iteration before, and solves
        // asked for 1e-7 and less in one cycle did not end.
        case FIN_BI_OMEGA: {
            for (int k = 0; k < 8; ++k)
                if (!isfinite(s[k])) {
                    bicg_fail(R, c, true);
                    return;
                }
            if (!(s[2] > 0.0)) {
                bicg_fail(R, c);
                break;
            }
            c.om_re = s[0] / s[2];
            c.om_im = s[1] / s[2];
            if (!isfinite(c.om_re) || !isfinite(c.om_im)) {
                bicg_fail(R, c);
                break;
            }
            const double wr = (double)(float)c.om_re, wi = (double)(float)c.om_im;
            c.rr = s[5] - 2.0 * (wr * s[0] + wi * s[1]) + (wr * wr + wi * wi) * s[2];
            c.iters += 1;
            c.last = 1;
            if (c.rr <= c.tol2) {
                c.active = 0;
                break;
            }
            if (c.iters >= c.maxit) {
                c.active = 0;
                c.flags |= 1;
                break;
            }
            const double nr = s[6] - (wr * s[3] - wi * s[4]);
            const double ni = s[7] - (wr * s[4] + wi * s[3]);
            // beta = (rho' / rho) (alpha / omega)
            double qr, qi, er, ei;
            cdiv(nr, ni, c.rho_re, c.rho_im, qr, qi);
            cdiv(c.al_re, c.al_im, c.om_re, c.om_im, er, ei);
            c.be_re = qr * er - qi * ei;
            c.be_im = qr * ei + qi * er;
            c.rho_re = nr;
            c.rho_im = ni;
            if (!(nr * nr + ni * ni > 0.0) || !isfinite(c.be_re) || !isfinite(c.be_im))
                bicg_fail(R, c);
            else
                c.last = 0;
            break;
        }
        default:
            break;
    }
}

// Sum of N values a thread over the grid row of rhs; the last thread block
// runs the finisher.  Every thread of the block calls this (at most 128
// threads).  Deterministic: all sums are taken in a fixed order.
//
// FP64 additions are the scarce resource (1.6 lanes a clock): the block sum
// goes through shared memory, 32 lanes a value, about 8 warp additions a
// value instead of 5 a warp.  Above 4096 partial sums the reduction has two
// levels: the last block of a group of DD_REDUCE_GROUP adds its members, the
// last group the groups.  With one level the last block of a grid of 6144
// had 18432 additions to make: the three-value kernels of a solve at
// 32^3 x 48 took 100 us instead of 66.  Below the line the second ticket
// costs more than it saves (135 blocks of one value: 1.5 us a launch).
template <int N>
DD_DEV void grid_reduce_n(const Reduce& R, int rhs, const double* v, void (*fin)(const Reduce&, int, const double*)) {
    __shared__ double buf[N][128];
    __shared__ double tot[N];
    __shared__ int last;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = (blockDim.x + 31) >> 5;
    const int nblk = gridDim.x;
    auto block_total = [&](const double* w) {  // tot[k] = sum of w[k] over the block
#pragma unroll
        for (int k = 0; k < N; ++k) buf[k][tid] = w[k];
        __syncthreads();
        for (int k = wid; k < N; k += nw) {
            double s = 0.0;
            for (int j = lane; j < (int)blockDim.x; j += 32) s += buf[k][j];
            s = warp_sum(s);
            if (lane == 0) tot[k] = s;
        }
        __syncthreads();
    };
    // true in every thread of the block that arrives last at a counter
    auto ticket = [&](unsigned* c, unsigned members) {
        if (tid == 0) {
            __threadfence();
            last = atomicAdd(c, 1u) == members - 1;
            if (last) *c = 0;
        }
        __syncthreads();
        const bool l = last;
        if (l) __threadfence();
        return l;
    };
    // partial sums p[k * n + i], i in [lo, hi), added up by the whole block
    auto gather = [&](const double* p, int n, int lo, int hi) {
        double s[N];
#pragma unroll
        for (int k = 0; k < N; ++k) s[k] = 0.0;
#pragma unroll 4
        for (int i = lo + tid; i < hi; i += blockDim.x)
#pragma unroll
            for (int k = 0; k < N; ++k) s[k] += __ldcg(p + (long long)k * n + i);
        block_total(s);
    };
    block_total(v);
    double* part = R.partials + (long long)rhs * N * nblk;
    if (tid < N) part[(long long)tid * nblk + blockIdx.x] = tot[tid];
    if (tid < N) __threadfence();
    __syncthreads();
    const int ngrp = (nblk + DD_REDUCE_GROUP - 1) / DD_REDUCE_GROUP;
    if (N * nblk > 4096) {
        const int grp = blockIdx.x / DD_REDUCE_GROUP, lo = grp * DD_REDUCE_GROUP, hi = min(lo + DD_REDUCE_GROUP, nblk);
        if (!ticket(R.groups + (long long)rhs * R.gmax + grp, (unsigned)(hi - lo))) return;
        gather(part, nblk, lo, hi);
        double* gpart = R.partials + (long long)gridDim.y * N * nblk + (long long)rhs * N * ngrp;
        if (tid < N) gpart[(long long)tid * ngrp + grp] = tot[tid];
        if (tid < N) __threadfence();
        __syncthreads();
        if (!ticket(&R.counters[rhs], (unsigned)ngrp)) return;
        gather(gpart, ngrp, 0, ngrp);
    } else {
        if (!ticket(&R.counters[rhs], (unsigned)nblk)) return;
        gather(part, nblk, 0, nblk);
    }
    if (tid == 0) fin(R, rhs, tot);
}

DD_DEV void finish1(const Reduce& R, int rhs, const double* s) { finish(R, rhs, s[0]); }
template <int N>
DD_DEV void grid_reduce_bi(const Reduce& R, int rhs, const double* v) { grid_reduce_n<N>(R, rhs, v, finish3); }
DD_DEV void grid_reduce(const Reduce& R, int rhs, double v) { grid_reduce_n<1>(R, rhs, &v, finish1); }
