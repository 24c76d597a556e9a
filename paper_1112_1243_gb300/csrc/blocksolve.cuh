// Block-local Dirichlet operator and the persistent launch of the block filter
// (Eq. 4step step 1): its items, lattices and arguments, and CG on the
// normal equations of one block.  The launches are in blockeo.cuh.
//
// Every thread block of the grid takes work items (block, factor) from an
// atomic queue and runs a complete solve of D_b x = src for that item with
// the whole thread block, all vectors in a per-thread-block scratch slot.
//
// D_b = 1 - kappa * H restricted to hops with both ends in block b (Dirichlet
// boundary: hops leaving the block are dropped).  Blocks never straddle the
// time edge (at least two blocks per direction), so no boundary phase occurs
// inside a block.  Block data (links, vectors) are stored in block order:
// block position, then sites of the block (FP64 vectors lexicographic; links
// by parity, then lexicographic, see format_gauge_kernel).
#pragma once

#include <type_traits>

#include "dd_internal.h"
#include "reduce.cuh"

struct BlockCtx {
    int bd[4];    // block extents
    int st[4];    // local strides
    int nb;       // sites per block
    double kappa;
};

DD_DEV void local_coords(const BlockCtx& c, int j, int l[4]) {
    l[0] = j % c.bd[0];
    int r = j / c.bd[0];
    l[1] = r % c.bd[1];
    r /= c.bd[1];
    l[2] = r % c.bd[2];
    l[3] = r / c.bd[2];
}

// acc = H_b in at local site j (hops inside the block only)
template <class R, class SIn, class LK>
DD_DEV void dirichlet_hop(const BlockCtx& c, int j, const SIn& in, const LK& lk, int g5in, Spinor<R>& acc) {
    int l[4];
    local_coords(c, j, l);
    zero(acc);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        if (l[a] < c.bd[a] - 1) {
            int jn = j + c.st[a];
            Spinor<R> s;
            in.load(jn, s);
            if (g5in) gamma5(s);
            Half<R> hf, uh;
            project<R>(a, +1, s, hf);
            Link<R> u;
            lk.load(j, a, u);
            mul_link(u, hf, uh);
            accumulate<R>(a, +1, uh, (R)1, acc);
        }
        if (l[a] > 0) {
            int jn = j - c.st[a];
            Spinor<R> s;
            in.load(jn, s);
            if (g5in) gamma5(s);
            Half<R> hf, uh;
            project<R>(a, -1, s, hf);
            Link<R> u;
            lk.load(jn, a, u);
            mul_link_dag(u, hf, uh);
            accumulate<R>(a, -1, uh, (R)1, acc);
        }
    }
}

// acc = (H_b[lk1] - H_b[lk2]) in at local site j: only hops whose two links
// differ contribute (the proposal changes the active links only)
template <class SIn, class LK>
DD_DEV void dirichlet_hop_diff(const BlockCtx& c, int j, const SIn& in, const LK& lk1, const LK& lk2,
                               Spinor<double>& acc) {
    int l[4];
    local_coords(c, j, l);
    zero(acc);
    for (int a = 0; a < 4; ++a) {
        for (int dir = +1; dir >= -1; dir -= 2) {
            if (dir > 0 ? (l[a] >= c.bd[a] - 1) : (l[a] <= 0)) continue;
            const int jn = j + dir * c.st[a];
            const int jl = dir > 0 ? j : jn;  // the link sits at the lower end
            Link<double> u1, u2;
            lk1.load(jl, a, u1);
            lk2.load(jl, a, u2);
            bool same = true;
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    u1.m[r][s] = u1.m[r][s] - u2.m[r][s];
                    same = same && u1.m[r][s].x == 0.0 && u1.m[r][s].y == 0.0;
                }
            if (same) continue;
            Spinor<double> sp;
            in.load(jn, sp);
            Half<double> hf, uh;
            project<double>(a, dir, sp, hf);
            if (dir > 0)
                mul_link(u1, hf, uh);
            else
                mul_link_dag(u1, hf, uh);
            accumulate<double>(a, dir, uh, 1.0, acc);
        }
    }
}

// out = D_b in (dag: gamma5 D_b gamma5); returns this thread's |out|^2 (block-reduce it)
template <class R, class SIn, class SOut, class LK>
DD_DEV double dirichlet_apply(const BlockCtx& c, const SIn& in, const SOut& out, const LK& lk, int dag) {
    double n2 = 0.0;
    for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
        Spinor<R> acc, v;
        dirichlet_hop<R>(c, j, in, lk, dag, acc);
        in.load(j, v);
        if (dag) gamma5(v);
        const R mk_ = (R)(-c.kappa);
#pragma unroll
        for (int k = 0; k < 12; ++k) v.c[k] = v.c[k] + mk_ * acc.c[k];
        if (dag) gamma5(v);
        out.store(j, v);
        n2 += (double)snorm2(v);
    }
    return n2;
}

// Inner CG on the normal equations D_b^dag D_b x = D_b^dag r0 (x starts at 0,
// r holds r0 on entry).  Stops when |r|^2 <= tol2rel |r0|^2 or after maxit.
template <class R, class S, class LK>
DD_DEV int block_cgnr(const BlockCtx& c, const S& x, const S& r, const S& p, const S& q, const S& z, const LK& lk,
                      double tol2rel, int maxit, double* sh) {
    double rr0 = 0.0;
    for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
        Spinor<R> zz;
        zero(zz);
        x.store(j, zz);
        Spinor<R> v;
        r.load(j, v);
        rr0 += (double)snorm2(v);
    }
    rr0 = block_sum(rr0, sh);  // includes a barrier: r and x complete
    if (!(rr0 > 0.0)) return 0;
    double zz = block_sum(dirichlet_apply<R>(c, r, z, lk, 1), sh);
    for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
        Spinor<R> v;
        z.load(j, v);
        p.store(j, v);
    }
    __syncthreads();
    const double target = tol2rel * rr0;
    int it = 0;
    while (it < maxit) {
        double qq = block_sum(dirichlet_apply<R>(c, p, q, lk, 0), sh);
        if (!(qq > 0.0)) break;
        const R alpha = (R)(zz / qq);
        double rr = 0.0;
        for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
            Spinor<R> a, b;
            x.load(j, a);
            p.load(j, b);
#pragma unroll
            for (int k = 0; k < 12; ++k) a.c[k] = a.c[k] + alpha * b.c[k];
            x.store(j, a);
            r.load(j, a);
            q.load(j, b);
#pragma unroll
            for (int k = 0; k < 12; ++k) a.c[k] = a.c[k] - alpha * b.c[k];
            r.store(j, a);
            rr += (double)snorm2(a);
        }
        rr = block_sum(rr, sh);
        ++it;
        if (rr <= target) break;
        double zn = block_sum(dirichlet_apply<R>(c, r, z, lk, 1), sh);
        const R beta = (R)(zn / zz);
        zz = zn;
        for (int j = threadIdx.x; j < c.nb; j += blockDim.x) {
            Spinor<R> a, b;
            z.load(j, a);
            p.load(j, b);
#pragma unroll
            for (int k = 0; k < 12; ++k) a.c[k] = a.c[k] + beta * b.c[k];
            p.store(j, a);
        }
        __syncthreads();
    }
    return it;
}

// ----------------------------------------------------------- the launch
struct BlockItem {
    int block_pos;  // position of the block in block order
    int f_src;      // field slot of the source operator
    int f_sol;      // field slot of the solve
    int vec;        // factor index (noise sub)
    int lat;        // lattice of the item in a multi-lattice launch (0 otherwise)
};

// block shape of the even-odd solver (blockeo.cuh)
struct EoCtx {
    int bd[4], st[4];
    int nb;     // sites of the block
    int half;   // stride of one parity's vectors: nb / 2, or nb for an odd extent along axis 0
    int sh;     // storage index of local site j: j >> sh
    int count;  // sites to visit for one parity (an odd extent along axis 0: all, the wrong parity skipped)
    int d0;     // extent along axis 0 in visited sites
    unsigned m0, m1, m2;
    float kappa2;
    double kappa;
};

// one lattice of a launch (blocks of different shapes)
struct LatDesc {
    Geo g;
    BlockCtx c;
    EoCtx eo;
    const double* canon;  // canonical FP64 links, field slot 0
    long long canon_fs;   // doubles between consecutive slots
    const int4* ddx;      // links in limbs, block order
    long long ddx_fs;
    const float2* dd32;
    long long dd32_fs;
    const uint8_t* active;  // active links [V * 4]
    double* item_out;
};

struct BlockArgs {
    const LatDesc* lats;  // multi-lattice launch: per-item lattice
    LatDesc lat;          // single-lattice launch (lats null)
    const BlockItem* items;  // null: block-filter items k -> (block position item_pos0 + k / item_n, vector k % item_n)
    int nitems;
    int nbig;  // leading items of large blocks, each solved by a cluster of thread blocks (block_eo_kernel)
    int item_pos0, item_n;
    int* queue;  // heads of the two queues: large items, the others
    char* scratch;
    long long slot_bytes;
    uint64_t seed, ctr;
    const unsigned long long* ctr_off;  // added to ctr (graph replays; may be null)
    int purpose;
    double tol2;       // relative target of the FP64 residual (squared)
    double tol2_inner; // relative target of one inner solve (squared)
    int maxit_inner;
    int max_outer;
    int inner_f64;
    int* status;
    unsigned long long* stats;  // items, inner iterations, outer cycles, site-iterations (may be null)
};

// block id of the block at position pos of the block order
DD_DEV int block_id_at(const Geo& g, int pos, int* colour) {
    int half = g.nblocks / 2;
    int col = pos >= half ? 1 : 0;
    int rank = pos - col * half;
    int id = 2 * rank;
    int B1 = (id / g.nbk[0]) % g.nbk[1], B2 = (id / (g.nbk[0] * g.nbk[1])) % g.nbk[2],
        B3 = id / (g.nbk[0] * g.nbk[1] * g.nbk[2]);
    if (((B1 + B2 + B3) & 1) != col) id += 1;
    *colour = col;
    return id;
}
DD_DEV void block_origin(const Geo& g, int id, int o[4]) {
    o[0] = (id % g.nbk[0]) * g.b[0];
    int r = id / g.nbk[0];
    o[1] = (r % g.nbk[1]) * g.b[1];
    r /= g.nbk[1];
    o[2] = (r % g.nbk[2]) * g.b[2];
    o[3] = (r / g.nbk[2]) * g.b[3];
}

// links of one block, read from a canonical FP64 field (V x 4 x 3 x 3 complex)
struct LinkCanonF64 {
    const double* U;
    Geo g;
    BlockCtx c;
    int org[4];
    template <class R>
    DD_DEV void load(long long j, int a, Link<R>& u) const {
        int l[4];
        local_coords(c, (int)j, l);
        int x[4] = {org[0] + l[0], org[1] + l[1], org[2] + l[2], org[3] + l[3]};
        const double* p = U + ((long long)canon_index(g, x) * 4 + a) * 18;
#pragma unroll
        for (int k = 0; k < 9; ++k) u.m[k / 3][k % 3] = mk<R>((R)p[2 * k], (R)p[2 * k + 1]);
    }
};
