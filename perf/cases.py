"""Performance cases: what a program that uses this package asks of it, through its public entry points.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what the program has in hand
(fields, spinors, the handle with its workspace), run() is one pass, work() the bytes and operations that a pass
cannot do without and exact() the outputs in plain torch, 64 bits, without the package.

Sizes: the workloads c1-c5 of the benchmark (4^4 with 2^4 blocks; 8^4 with 4^4 blocks and 16 factors; 16^4 with 8^4
blocks and 8 factors; 4^4, 6^4 and 8^4 blocks in one batched filter; 32^3 x 64 and 32^3 x 48), and lattices with
other even extents around them.  Fields are exp(i eps H) with Gaussian H, proposals rotate every active link by
about the angle of a heat-bath hit.
"""
import math

import numpy as np
import torch

from paper_1112_1243_gb300 import api
from paper_1112_1243_gb300.chain import HierarchicalStep

BETA = 5.3
ROTATION = 0.2  # a heat-bath hit at beta 5.3 turns each SU(2) subgroup by about 0.4
HOP_FLOPS = 1368  # one Wilson hopping term on one site, with the sum onto the result
PRECS = {"f64": api.DD_PREC_F64, "f32": api.DD_PREC_F32, "f16": api.DD_PREC_F16}
KRYLOV = {"cgnr": api.DD_KRYLOV_CGNR, "bicgstab": api.DD_KRYLOV_BICGSTAB}


def listed():
    return [
        # one application of D on the smallest lattice: all latency and launches (tests, smoke)
        {"name": "apply_4", "path": "apply", "dims": "4x4x4x4", "block": "2x2x2x2", "n": 1},
        # one application of D at the benchmark's volume: the Dslash of the headline metric in FP64
        {"name": "apply_32x64", "path": "apply", "dims": "32x32x32x64", "block": "8x8x8x8", "n": 1},
        # one mixed-precision propagator column on a small lattice
        {"name": "solve_8", "path": "solve", "dims": "8x8x8x8", "block": "4x4x4x4", "n": 1, "prec": "f16",
         "krylov": "bicgstab", "eps": 0.3, "kappa": 0.13},
        # a batch of right-hand sides with FP32 storage, the default Krylov method, extents that are no powers of 2
        {"name": "solve_12x20_f32", "path": "solve", "dims": "12x12x12x20", "block": "6x6x6x10", "n": 5, "prec": "f32",
         "krylov": "cgnr", "eps": 0.3, "kappa": 0.13},
        # the single global solve of the benchmark (its solve mode): beyond the L2 cache
        {"name": "solve_32x48", "path": "solve", "dims": "32x32x32x48", "block": "8x8x8x8", "n": 1, "prec": "f16",
         "krylov": "bicgstab", "eps": 0.2, "kappa": 0.1355},
        # the global estimate of c2 in mixed precision, and on the plain FP64 path it is compared with
        {"name": "estimate_8", "path": "estimate", "dims": "8x8x8x8", "block": "4x4x4x4", "n": 16, "prec": "f16",
         "krylov": "bicgstab", "eps": 0.3, "kappa": 0.13},
        {"name": "estimate_8_f64", "path": "estimate", "dims": "8x8x8x8", "block": "4x4x4x4", "n": 16, "prec": "f64",
         "krylov": "cgnr", "eps": 0.3, "kappa": 0.13},
        # the global estimate of c3: 8^4 blocks, 8 factors
        {"name": "estimate_16", "path": "estimate", "dims": "16x16x16x16", "block": "8x8x8x8", "n": 8, "prec": "f16",
         "krylov": "bicgstab", "eps": 0.25, "kappa": 0.135},
        # the batched block filter of c4: blocks of 4^4, 6^4 and 8^4, 4 noise vectors each
        {"name": "filter_batch", "path": "filter", "n": 4, "eps": 0.3, "kappa": 0.13,
         "lattices": "16x16x16x16/4x4x4x4 12x12x12x12/6x6x6x6 16x16x16x16/8x8x8x8"},
        # the whole Markov step: proposal, block filter, global estimate, accept (with enough factors for the
        # filter to let blocks through, as a run that is to move needs)
        {"name": "chain_16x32", "path": "chain", "dims": "16x16x16x32", "block": "4x4x4x4", "n": 12, "eps": 0.2,
         "kappa": 0.1355},
        # ln |det D| by dense LU, the exact check of c1
        {"name": "logdet_4", "path": "logdet", "dims": "4x4x4x4", "block": "2x2x2x2", "which": 0},
        # thermalisation of a pure-gauge field: one heat-bath and two over-relaxation sweeps over every link
        {"name": "thermalise_16", "path": "update", "dims": "16x16x16x16", "block": "4x4x4x4", "n_or": 2},
    ]


def draw(rng):
    path = rng.choice(["apply", "solve", "solve", "estimate", "estimate", "filter", "chain", "logdet", "update"])

    def lattice(low, high, blocks=(2, 3, 4, 5, 6, 8), counts=(2, 4)):
        """Extents block x count whose volume lies in [low, high], spread over its logarithm."""
        goal = math.exp(rng.uniform(math.log(low), math.log(high)))
        best = None
        for _ in range(200):
            b = [rng.choice(blocks) for _ in range(4)]
            d = [x * rng.choice(counts) for x in b]
            off = abs(math.log(math.prod(d) / goal))
            if low <= math.prod(d) <= high and (best is None or off < best[0]):
                best = (off, d, b)
                if off < 0.1:
                    break
        return {"dims": "x".join(map(str, best[1])), "block": "x".join(map(str, best[2]))}

    if path == "apply":
        return {"path": path, **lattice(256, 2 << 20, (2, 3, 4, 5, 6, 8, 10, 16)), "n": rng.randint(1, 3)}
    if path == "solve":
        prec = rng.choice(["f16", "f16", "f32", "f64"])
        return {"path": path, **lattice(1024, 1 << 18, (3, 4, 5, 6, 8)), "n": rng.randint(1, 6), "prec": prec,
                "krylov": rng.choice(["bicgstab", "cgnr"]) if prec != "f64" else "cgnr", "eps": 0.3, "kappa": 0.13}
    if path == "estimate":
        return {"path": path, **lattice(4096, 65536, (4, 6, 8)), "n": rng.randint(2, 12), "prec": "f16",
                "krylov": rng.choice(["bicgstab", "bicgstab", "cgnr"]), "eps": 0.3, "kappa": rng.choice([0.125, 0.13])}
    if path == "filter":
        one = [lattice(4096, 65536, (4, 5, 6, 8)) for _ in range(rng.randint(1, 3))]
        return {"path": path, "n": rng.randint(1, 4), "eps": 0.3, "kappa": 0.13,
                "lattices": " ".join(c["dims"] + "/" + c["block"] for c in one)}
    if path == "chain":
        return {"path": path, **lattice(16384, 131072, (4,), (2, 4, 6, 8)), "n": rng.randint(8, 12), "eps": 0.2,
                "kappa": rng.choice([0.13, 0.1355])}
    if path == "logdet":
        return {"path": path, **lattice(300, 512, (2, 3)), "which": rng.choice([0, 1, 2])}
    return {"path": path, **lattice(4096, 1 << 18, (4, 5, 6, 8)), "n_or": rng.randint(0, 4)}


# ------------------------------------------------------------------ inputs
def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def _lattices(case):
    if case["path"] == "filter":
        return [tuple(_ints(t) for t in p.split("/")) for p in case["lattices"].split()]
    return [(_ints(case["dims"]), _ints(case["block"]))]


def _mul(a, b):
    """Product of stacked small matrices (element by element: no batched library calls)."""
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _su3(shape, eps, gen, device):
    """exp(i eps H), H traceless Hermitian with N(0, 1) parts off the diagonal; rows made orthonormal again."""
    total = math.prod(shape)
    out = torch.empty((total, 3, 3), dtype=torch.complex128, device=device)
    step = 1 << 20
    for k in range(0, total, step):
        m = min(step, total - k)
        w = torch.randn((8, m), dtype=torch.float64, device=device, generator=gen)
        h = torch.zeros((m, 3, 3), dtype=torch.complex128, device=device)
        for e, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
            h[:, i, j] = torch.complex(w[2 * e], -w[2 * e + 1])
            h[:, j, i] = h[:, i, j].conj()
        h[:, 0, 0] = w[6] + w[7] / math.sqrt(3)
        h[:, 1, 1] = -w[6] + w[7] / math.sqrt(3)
        h[:, 2, 2] = -2 * w[7] / math.sqrt(3)
        x = (0.25j * eps) * h
        u = torch.eye(3, dtype=torch.complex128, device=device) + x
        t = x
        for r in range(2, 15):
            t = _mul(t, x) / r
            u = u + t
        u = _mul(u, u)
        u = _mul(u, u)
        a = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=-1, keepdim=True)
        b = u[:, 1] - (a.conj() * u[:, 1]).sum(-1, keepdim=True) * a
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
        out[k:k + m] = torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=1)
    return out.view(*shape, 3, 3)


def _active(dims, block):
    """Active links (V, 4) of the blocks: at most one end on the boundary of the block (of the block without its outer
    layer for extents of 8 and more; every link inside a block for extents up to 2)."""
    x = np.stack([g.reshape(-1, order="F") for g in np.meshgrid(*(np.arange(d) for d in dims), indexing="ij")], axis=1)
    b, size = np.array(block), np.array(dims)
    shrink = 1 if min(block) >= 8 else 0

    def region(y):
        loc = y % b
        inside = np.all((loc >= shrink) & (loc <= b - 1 - shrink), axis=1)
        at = (y // b) @ np.cumprod([1] + [d // e for d, e in zip(dims, block)][:3])
        return np.where(inside, at, -1)

    def on_boundary(y):
        r, edge = region(y), np.zeros(len(y), dtype=bool)
        for a in range(4):
            for s in (1, -1):
                z = y.copy()
                z[:, a] = (z[:, a] + s) % size[a]
                edge |= region(z) != r
        return edge & (r >= 0)

    act = np.zeros((len(x), 4), dtype=bool)
    here, edge = region(x), on_boundary(x)
    for a in range(4):
        y = x.copy()
        y[:, a] = (y[:, a] + 1) % size[a]
        act[:, a] = (here >= 0) & (region(y) == here)
        if min(block) > 2:
            act[:, a] &= ~(edge & on_boundary(y))
    return act


def _fields(case, seed):
    """The gauge field, and the proposal where the path has one, of every lattice of the case."""
    out = []
    for k, (dims, block) in enumerate(_lattices(case)):
        gen = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + k)
        V = math.prod(dims)
        U = _su3((V, 4), case.get("eps", 0.3), gen, "cuda")
        Up = None
        if case["path"] in ("estimate", "filter"):
            act = torch.from_numpy(_active(dims, block)).cuda()
            Up = U.clone()
            Up[act] = _mul(U[act], _su3((int(act.sum()),), ROTATION, gen, "cuda"))
        out.append((dims, block, U, Up, gen))
    return out


def _spinors(n, V, gen):
    re = torch.randn((n, V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen)
    return torch.view_as_complex(re) / math.sqrt(2)


def prepare(case, seed):
    fields = _fields(case, seed)
    dims, block, U, Up, gen = fields[0]
    path, V = case["path"], math.prod(dims)
    s = {"path": path, "U": U, "ctr": 0, "seed": int(seed)}
    if path == "apply":
        s["h"] = api.dd_init(dims, block, 0.13, max_rhs=case["n"], features=api.DD_FEAT_SOLVE)
        s["in"] = _spinors(case["n"], V, gen)
        s["out"] = torch.empty_like(s["in"])
        s["n"] = case["n"]
    elif path == "solve":
        s["h"] = api.dd_init(dims, block, case["kappa"], max_rhs=case["n"], inner_prec=PRECS[case["prec"]],
                             krylov=KRYLOV[case["krylov"]], features=api.DD_FEAT_SOLVE)
        s["in"] = _spinors(case["n"], V, gen)
        s["out"] = torch.empty_like(s["in"])
        s["n"], s["prec"] = case["n"], PRECS[case["prec"]]
    elif path == "estimate":
        s["h"] = api.dd_init(dims, block, case["kappa"], max_rhs=case["n"], inner_prec=PRECS[case["prec"]],
                             krylov=KRYLOV[case["krylov"]])
        s["Up"], s["n"] = Up, case["n"]
    elif path == "filter":
        s["h"] = [api.dd_init(d, b, case["kappa"], max_rhs=case["n"]) for d, b, _, _, _ in fields]
        s["U"] = [f[2] for f in fields]
        s["proposal"] = [f[3] for f in fields]
        s["Up"] = [torch.empty_like(u) for u in s["U"]]
        s["n"] = case["n"]
    elif path == "chain":
        h = api.dd_init(dims, block, case["kappa"], max_rhs=case["n"], krylov=api.DD_KRYLOV_BICGSTAB)
        s["h"] = h
        s["chain"] = HierarchicalStep(h, BETA, n_block=case["n"], n_global=case["n"], seed=int(seed))
    elif path == "logdet":
        s["h"] = api.dd_init(dims, block, 0.12, features=api.DD_FEAT_EXACT)
        s["which"] = case["which"]
    else:
        s["h"] = api.dd_init(dims, block, 0.125, active_mode=api.DD_ACTIVE_ALL, features=api.DD_FEAT_SOLVE)
        s["n_or"] = case["n_or"]
    return s


def run(s):
    path, h, U = s["path"], s["h"], s["U"]
    ctr = s["ctr"]
    s["ctr"] += 1  # every pass draws its own random numbers
    if path == "apply":
        api.dd_apply_D(h, s["out"], s["in"], U, api.DD_OP_D, api.DD_PREC_F64, s["n"])
        return s["out"]
    if path == "solve":
        # the iteration counts and residuals that the call also returns are no results: any solver's differ
        api.dd_solve(h, s["out"], s["in"], U, s["n"], s["prec"])
        return s["out"]
    if path == "estimate":
        return api.dd_det_ratio_estimate(h, U, s["Up"], s["n"], s["seed"], ctr)
    if path == "filter":
        for up, p in zip(s["Up"], s["proposal"]):
            up.copy_(p)
        ln_b, accept = api.dd_block_filter_batch(h, U, s["Up"], 3, s["n"], s["seed"], ctr)
        return {"ln_b": ln_b, "accept": accept, "U": s["Up"]}
    if path == "chain":
        c = s["chain"]
        c.step(U, ctr)
        return {"U": U, "ln_b": c.ln_b, "accept_b": c.acc_b, "ln_g": c.ln_g, "accept_g": c.acc_g, "margin": c.margin}
    if path == "logdet":
        return api.dd_logdet_exact(h, U, s["which"])
    api.dd_gauge_update(h, U, 3, 5.8, 1, s["n_or"], s["seed"], ctr)
    return U


def work(case):
    """Inputs read and outputs written once; the arithmetic of the method with the iterations that its solves need to
    their targets at these masses (Krylov steps of two even-odd operators, so many Wilson applications a system)."""
    path, n = case["path"], case.get("n", 1)
    V = sum(math.prod(d) for d, _ in _lattices(case))
    field, spinor = 576 * V, 192 * V
    heavy = case.get("kappa", 0.13) <= 0.13
    solve, dirichlet = (100, 60) if heavy else (250, 75)
    if path == "apply":
        return {"bytes": field + 2 * n * spinor, "flops": n * V * HOP_FLOPS}
    if path == "solve":
        return {"bytes": field + 2 * n * spinor, "flops": n * V * HOP_FLOPS * solve}
    if path == "estimate":  # three block solves on half of the sites and one global solve a factor
        return {"bytes": 2 * field + 8 * n, "flops": n * V * HOP_FLOPS * (solve + 1.5 * dirichlet)}
    if path == "filter":
        return {"bytes": 3 * field, "flops": n * V * HOP_FLOPS * dirichlet}
    if path == "chain":
        return {"bytes": 2 * field, "flops": n * V * HOP_FLOPS * (solve + 2.5 * dirichlet)}
    if path == "logdet":
        order = {0: 12 * V, 1: 12 * math.prod(_ints(case["block"])), 2: 6 * V}[case["which"]]
        count = V // math.prod(_ints(case["block"])) if case["which"] == 1 else 1
        return {"bytes": field, "flops": count * 8 * order ** 3 / 3}
    # six staples of three matrix products (two of them shared by no other link) and three subgroup updates a link
    return {"bytes": 2 * field, "flops": 4 * V * (1 + case["n_or"]) * (12 * 198 + 6 * 18 + 3 * 150)}


# --------------------------------------------- the outputs in plain 64 bits
# gamma of the lattice axes 0..3 as a permutation of the spins and a phase (chiral basis, axis 3 = time)
GAMMA = (((3, 2, 1, 0), (-1j, -1j, 1j, 1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
         ((2, 3, 0, 1), (-1j, 1j, 1j, -1j)), ((2, 3, 0, 1), (-1, -1, -1, -1)))
ALL, INTRA, INTER = 0, 1, 2


class Plain:
    """The Wilson operator D = 1 - kappa H (antiperiodic in time) and its block pieces on (n, V, 4, 3) spinors with
    gauge fields (n or 1, V, 4, 3, 3)."""

    def __init__(self, dims, block, kappa):
        self.dims, self.kappa = dims, kappa
        V = math.prod(dims)
        s = torch.arange(V, device="cuda")
        x, stride = [], 1
        for d in dims:
            x.append((s // stride) % d)
            stride *= d
        self.x = x
        self.B = [c // b for c, b in zip(x, block)]
        self.colour = sum(self.B) % 2
        count = [d // b for d, b in zip(dims, block)]
        self.block_id = self.B[0] + count[0] * (self.B[1] + count[1] * (self.B[2] + count[2] * self.B[3]))
        self.nblocks = math.prod(count)
        self.fwd, self.bwd, stride = [], [], 1
        for a, d in enumerate(dims):
            self.fwd.append(torch.where(x[a] == d - 1, s - (d - 1) * stride, s + stride))
            self.bwd.append(torch.where(x[a] == 0, s + (d - 1) * stride, s - stride))
            stride *= d
        self.sign = (1.0 - 2.0 * (x[3] == dims[3] - 1).double(), 1.0 - 2.0 * (x[3] == 0).double())
        self.phase = [torch.tensor(p, dtype=torch.complex128, device="cuda")[:, None] for _, p in GAMMA]

    def hop(self, U, v, which):
        out = torch.zeros_like(v)
        for a in range(4):
            for dirn, at in ((0, self.fwd[a]), (1, self.bwd[a])):
                w = v[:, at]
                g = self.phase[a] * w[:, :, list(GAMMA[a][0])]
                w = w + g if dirn else w - g
                # the projected spinor has two free spins; the other two follow from (1 -+ gamma) w = 2 w
                u = _dag(U[:, at, a]) if dirn else U[:, :, a]
                top = _mul(w[:, :, :2], u.transpose(-1, -2))
                src = GAMMA[a][0]
                # w = -+ gamma w on the lower spins
                low = self.phase[a][2:] * top[:, :, [src[2], src[3]]]
                t = torch.cat([top, low if dirn else -low], dim=2)
                f = torch.ones_like(self.sign[0])
                if a == 3:
                    f = f * self.sign[dirn]
                if which != ALL:
                    f = f * ((self.block_id[at] == self.block_id) == (which == INTRA))
                out += f[:, None, None] * t
        return out

    def D(self, U, v, which=ALL):
        h = -self.kappa * self.hop(U, v, which)
        return h if which == INTER else v + h

    def solve(self, U, b, which=ALL, tol=2e-14):
        """BiCGStab on D, all systems at once, started again from the true residual until it stays below tol."""
        x, norm = torch.zeros_like(b), _dot(b, b).real.sqrt()
        norm = torch.where(norm > 0, norm, torch.ones_like(norm))
        for _ in range(6):
            r = b - self.D(U, x, which)
            if bool((_dot(r, r).real.sqrt() <= 4 * tol * norm).all()):
                break
            goal = torch.clamp(tol * norm / 2, min=1e-300)
            rh, p, rho = r.clone(), r.clone(), _dot(r, r)
            for it in range(2000):
                on = _dot(r, r).real.sqrt() > goal
                if it % 8 == 0 and not bool(on.any()):
                    break
                v = self.D(U, p, which)
                alpha = _safe(rho, _dot(rh, v), on)
                s = r - _up(alpha) * v
                t = self.D(U, s, which)
                omega = _safe(_dot(t, s), _dot(t, t), on)
                x = x + _up(alpha) * p + _up(omega) * s
                r = torch.where(_up(on), s - _up(omega) * t, r)
                new = _dot(rh, r)
                beta = _safe(new * alpha, rho * omega, on)
                p, rho = r + _up(beta) * (p - _up(omega) * v), torch.where(on, new, rho)
        return x


def _dot(a, b):
    return (a.conj() * b).flatten(1).sum(1)


def _up(a):
    return a[:, None, None, None]


def _safe(a, b, on):
    ok = on & (b.abs() > 0)
    return torch.where(ok, a / torch.where(ok, b, torch.ones_like(b)), torch.zeros_like(a))


def _philox(element, purpose, sub, seed, ctr):
    """Philox4x32-10 words of the stream (element, purpose, sub, seed, ctr), in 64-bit integers."""
    mask = 0xFFFFFFFF
    c = [element & mask, torch.full_like(element, (purpose << 24) | (sub & 0xFFFFFF)),
         torch.full_like(element, ctr & mask), torch.full_like(element, (ctr >> 32) & mask)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def wide(m, v):
        high, low = m * (v >> 16), m * (v & 0xFFFF)
        return (high + (low >> 16)) >> 16, (((high & 0xFFFF) << 16) + low) & mask

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = wide(0xD2511F53, c[0])
        h1, l1 = wide(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


def _uniforms(element, purpose, sub, seed, ctr):
    w = _philox(element, purpose, sub, seed, ctr)
    return [(((w[k] << 21) | (w[k + 1] >> 11)).double() + 0.5) * 2.0 ** -53 for k in (0, 2)]


def _noise(V, purpose, sub, seed, ctr):
    u1, u2 = _uniforms(torch.arange(12 * V, device="cuda"), purpose, sub, seed, ctr)
    return torch.polar(torch.sqrt(-torch.log(u1)), 2 * math.pi * u2).view(V, 4, 3)


def _path_fields(U, Up, act, n):
    """U (U^dag U')^(i/n) on the active links, i = 0 .. n."""
    a, b = U[act], Up[act]
    lam, vec = np.linalg.eig(_mul(_dag(a), b).cpu().numpy())
    th = np.angle(lam)
    total = th.sum(1)
    for rows, pick, turn in ((total > math.pi, np.argmax, -2 * math.pi), (total < -math.pi, np.argmin, 2 * math.pi)):
        at = np.nonzero(rows)[0]
        th[at, pick(th[at], axis=1)] += turn
    inv = np.linalg.inv(vec)
    fields = [U]
    for i in range(1, n):
        w = (vec * np.exp(1j * i / n * th)[:, None, :]) @ inv
        f = U.clone()
        f[act] = _mul(a, torch.from_numpy(w).cuda())
        fields.append(f)
    last = U.clone()
    last[act] = b
    return torch.stack(fields + [last])


def _exact_estimate(case, seed):
    dims, block, U, Up, _ = _fields(case, seed)[0]
    n, P = case["n"], Plain(dims, block, case["kappa"])
    F = _path_fields(U, Up, torch.from_numpy(_active(dims, block)).cuda(), n)
    old, new = F[:-1], F[1:]
    black = (P.colour == 0)[:, None, None]
    eta = torch.stack([_noise(math.prod(dims), api.DD_PURPOSE_GLOBAL_NOISE, i, int(seed), 0) for i in range(n)]) * black

    def inner(f):  # B E^-1 C eta
        w = P.D(f, eta, INTER) * ~black
        return P.D(f, P.solve(f, w, INTRA), INTER) * black

    a = P.solve(old, inner(old), INTRA)
    s = (inner(new) - P.D(new, a, INTRA)) * black
    d = P.solve(new, s) * black
    return -(2 * _dot(eta, d).real + _dot(d, d).real)


def _exact_filter(case, seed):
    n, res = case["n"], {"ln_b": [], "accept": [], "U": []}
    for dims, block, U, Up, _ in _fields(case, seed):
        P = Plain(dims, block, case["kappa"])
        act = torch.from_numpy(_active(dims, block)).cuda()
        F = _path_fields(U, Up, act, n)
        eta = torch.stack([_noise(math.prod(dims), api.DD_PURPOSE_BLOCK_NOISE, i, int(seed), 0) for i in range(n)])
        d = P.solve(F[1:], P.D(F[:-1], eta, INTRA) - P.D(F[1:], eta, INTRA), INTRA)
        per_site = -(2 * (eta.conj() * d).real + (d.conj() * d).real).sum((0, 2, 3))
        ln_b = torch.zeros(P.nblocks, dtype=torch.float64, device="cuda").index_add_(0, P.block_id, per_site)
        u = _uniforms(torch.arange(P.nblocks, device="cuda"), api.DD_PURPOSE_BLOCK_ACCEPT, 0, int(seed), 0)[0]
        accept = torch.log(u) < ln_b
        res["ln_b"].append(ln_b)
        res["accept"].append(accept.to(torch.uint8))
        back = act & ~accept[P.block_id][:, None]
        res["U"].append(torch.where(back[:, :, None, None], U, Up))
    return res


def _exact_logdet(case, seed):
    dims, block, U, _, _ = _fields(case, seed)[0]
    V, P = math.prod(dims), Plain(dims, block, 0.12)

    def dense(which):
        unit = torch.eye(12 * V, dtype=torch.complex128, device="cuda").view(12 * V, V, 4, 3)
        return torch.cat([P.D(U[None], unit[k:k + 512], which).view(-1, 12 * V) for k in range(0, 12 * V, 512)]).T

    def ln(m):
        return float(np.linalg.slogdet(m.cpu().numpy())[1])

    if case["which"] == 0:
        return torch.tensor([ln(dense(ALL))], dtype=torch.float64)
    blocks = dense(INTRA)
    of = torch.arange(V, device="cuda")

    def rows(sites):
        return (12 * sites[:, None] + torch.arange(12, device="cuda")).reshape(-1)

    per = []
    for k in range(P.nblocks):
        r = rows(of[P.block_id == k])
        per.append(ln(blocks[r][:, r]))
    if case["which"] == 1:
        return torch.tensor(per, dtype=torch.float64)
    # det D = det A det E det Dhat
    return torch.tensor([ln(dense(ALL)) - sum(per)], dtype=torch.float64)


def _exact_update(case, seed):
    dims, block, U, _, _ = _fields(case, seed)[0]
    P, U, beta = Plain(dims, block, 0.125), U.clone(), 5.8
    parity = sum(P.x) % 2
    sites = torch.arange(math.prod(dims), device="cuda")

    def su2(a):
        return torch.stack([torch.stack([torch.complex(a[0], a[3]), torch.complex(a[2], a[1])], -1),
                            torch.stack([torch.complex(-a[2], a[1]), torch.complex(a[0], -a[3])], -1)], -2)

    def group(a, s, heatbath):
        staples = torch.zeros((len(s), 3, 3), dtype=torch.complex128, device="cuda")
        sa = P.fwd[a][s]
        for b in range(4):
            if b != a:
                sb, sm, sam = P.fwd[b][s], P.bwd[b][s], P.bwd[b][sa]
                staples += _mul(_mul(U[sa, b], _dag(U[sb, a])), _dag(U[s, b]))
                staples += _mul(_dag(_mul(U[sm, a], U[sam, b])), U[sm, b])
        u, element = U[s, a], 4 * s + a
        for sg, (i, j) in enumerate(((0, 1), (1, 2), (0, 2))):
            w = _mul(u, staples)
            q = torch.stack([w[:, i, i].real + w[:, j, j].real, w[:, i, j].imag + w[:, j, i].imag,
                             w[:, i, j].real - w[:, j, i].real, w[:, i, i].imag - w[:, j, j].imag]) / 2
            k = torch.linalg.vector_norm(q, dim=0)
            v = _dag(su2(q / k))
            if heatbath:
                alpha, x0, done = 2 * beta * k / 3, torch.ones_like(k), torch.zeros_like(k, dtype=torch.bool)
                for t in range(64):
                    if bool(done.all()):
                        break
                    u1, u2 = _uniforms(element, api.DD_PURPOSE_HEATBATH, (sg << 12) + 2 * t, int(seed), 0)
                    u3, u4 = _uniforms(element, api.DD_PURPOSE_HEATBATH, (sg << 12) + 2 * t + 1, int(seed), 0)
                    lam = -(torch.log(u1) + torch.cos(2 * math.pi * u2) ** 2 * torch.log(u3)) / (2 * alpha)
                    take = ~done & (u4 * u4 <= 1 - lam)
                    x0 = torch.where(take, 1 - 2 * lam, x0)
                    done |= take
                u5, u6 = _uniforms(element, api.DD_PURPOSE_HEATBATH, (sg << 12) + 200, int(seed), 0)
                r = torch.sqrt(torch.clamp(1 - x0 * x0, min=0))
                cth = 2 * u5 - 1
                sth = torch.sqrt(torch.clamp(1 - cth * cth, min=0))
                turn = _mul(su2([x0, r * sth * torch.cos(2 * math.pi * u6), r * sth * torch.sin(2 * math.pi * u6),
                                 r * cth]), v)
                turn = torch.where(done[:, None, None], turn, torch.eye(2, dtype=turn.dtype, device="cuda"))
            else:
                turn = _mul(v, v)
            u = u.clone()
            u[:, [i, j]] = _mul(turn, u[:, [i, j]])
        U[s, a] = u

    for kind in range(1 + case["n_or"]):
        for a in range(4):
            for par in (0, 1):
                group(a, sites[parity == par], kind == 0)
    return U


def exact(case, seed):
    path = case["path"]
    if path in ("apply", "solve"):
        dims, block, U, _, gen = _fields(case, seed)[0]
        b = _spinors(case["n"], math.prod(dims), gen)
        if path == "apply":
            return Plain(dims, block, 0.13).D(U[None], b)
        return Plain(dims, block, case["kappa"]).solve(U[None], b)
    if path == "estimate":
        return _exact_estimate(case, seed)
    if path == "filter":
        return _exact_filter(case, seed)
    if path == "logdet":
        return _exact_logdet(case, seed)
    if path == "update":
        return _exact_update(case, seed)
    return None  # the whole step: some hundred operator applications a factor, over 20 seconds in plain torch
