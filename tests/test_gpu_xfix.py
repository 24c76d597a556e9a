"""The FP64 operator on two-limb integers (hop_x_kernel): against the same
stencil in extended precision (numpy longdouble), at ragged extents, one and
several right-hand sides, entries over many orders of magnitude, sparse
fields and links that are not unitary."""
import numpy as np
import pytest

from gpu_util import dev, host, lib_api
from oracle import geometry
from oracle.gamma import GAMMA_AXIS
from paper_1112_1243_gb300 import synthetic

pytestmark = pytest.mark.gpu
LD = np.clongdouble


@pytest.fixture(scope="module")
def api():
    return lib_api()


def hop_extended(U, psi, lat):
    """H psi and the sum of the magnitudes of its terms, in extended precision."""
    out, mag = np.zeros(psi.shape, dtype=LD), np.zeros(psi.shape[0])
    U, psi = U.astype(LD), psi.astype(LD)
    for a in range(4):
        for y, sign, links, g in ((lat.fwd[:, a], lat.sign_fwd[:, a], U[:, a], -1),
                                  (lat.bwd[:, a], lat.sign_bwd[:, a], np.conj(np.swapaxes(U[lat.bwd[:, a], a], 1, 2)), 1)):
            w = psi[y]
            gam = GAMMA_AXIS[a]
            p = w + g * sum(gam[:, k].astype(LD)[None, :, None] * w[:, k:k + 1] for k in range(4))
            t = sum(links[:, :, j][:, None, :] * p[:, :, j][:, :, None] for j in range(3))
            out += sign[:, None, None] * t
            mag += (np.abs(links).max((1, 2)) * np.abs(w).max((1, 2))).astype(np.float64)
    return out, mag


@pytest.mark.parametrize("dims,block,nrhs,kind", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 1, "plain"),
    ((6, 4, 10, 12), (3, 2, 5, 6), 3, "plain"),
    ((8, 8, 8, 8), (4, 4, 4, 4), 2, "spread"),
    ((10, 6, 4, 8), (5, 3, 2, 4), 1, "sparse"),
    ((4, 8, 6, 4), (2, 4, 3, 2), 2, "links"),
    ((2, 4, 6, 2), (1, 2, 3, 1), 2, "plain"),
])
def test_against_extended_precision(api, dims, block, nrhs, kind):
    """Per site: one rounding of the result (2^-53), the rounding of the hop
    sum (2^-53) and the integer form's 2^-54 of every hop's largest product."""
    kappa = 0.13
    lat = geometry.Lattice(dims, block)
    rng = np.random.default_rng(11)
    U = synthetic.random_gauge(dims, 0.4, 2)
    psi = synthetic.random_spinor(dims, 5, nrhs=nrhs)
    if kind == "spread":
        psi = psi * np.exp(6 * rng.standard_normal(psi.shape))
    elif kind == "sparse":
        psi = psi * (rng.random(psi.shape) < 0.03)
    elif kind == "links":
        U = U * np.exp(3 * rng.standard_normal(U.shape[:2]))[:, :, None, None]
    h = api.dd_init(dims, block, kappa, max_rhs=nrhs)
    out = dev(np.zeros_like(psi))
    api.dd_apply_D(h, out, dev(psi), dev(U), api.DD_OP_D, api.DD_PREC_F64, nrhs)
    got = host(out)
    for r in range(nrhs):
        hop, mag = hop_extended(U, psi[r], lat)
        ref = psi[r].astype(LD) - LD(kappa) * hop
        err = np.abs(got[r].astype(LD) - ref).max((1, 2)).astype(np.float64)
        top = (np.abs(ref).max((1, 2)) + kappa * np.abs(hop).max((1, 2))).astype(np.float64)
        assert np.all(err <= np.sqrt(2) * (2.0 ** -53 * top + kappa * 2.0 ** -54 * mag))


def test_scales_far_from_one(api):
    """Exponents beyond the range of one multiplier take the general scaling:
    powers of two pass through exactly."""
    dims, block = (4, 4, 4, 4), (2, 2, 2, 2)
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5)
    h = api.dd_init(dims, block, 0.125)
    res = {}
    for k in (0, -960, 960):
        out = dev(np.zeros_like(psi))
        api.dd_apply_D(h, out, dev(psi * 2.0 ** k), dev(U), api.DD_OP_D, api.DD_PREC_F64, 1)
        res[k] = host(out)
    for k in (-960, 960):
        assert np.allclose(res[k] * 2.0 ** -k, res[0], rtol=1e-14, atol=1e-14)
    out = dev(np.ones_like(psi))
    api.dd_apply_D(h, out, dev(0 * psi), dev(U), api.DD_OP_D, api.DD_PREC_F64, 1)
    assert np.all(host(out) == 0)


def test_non_finite_numbers_stay_in_their_components(api):
    """An infinity or NaN in a spinor or link entry reaches exactly the
    components that the FP64 stencil takes it to."""
    dims, block, kappa = (4, 4, 6, 4), (2, 2, 3, 2), 0.13
    lat = geometry.Lattice(dims, block)
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5)
    psi[17, 2, 1] = np.inf
    U[200, 3, 1, 2] = np.nan
    h = api.dd_init(dims, block, kappa)
    out = dev(np.zeros_like(psi))
    api.dd_apply_D(h, out, dev(psi), dev(U), api.DD_OP_D, api.DD_PREC_F64, 1)
    got = host(out)
    # sites next to neither are finite, and equal to those of the clean fields
    touched = {17, 200, int(lat.fwd[200, 3])} | {int(n[17, a]) for n in (lat.fwd, lat.bwd) for a in range(4)}
    clean = np.array([s not in touched for s in range(lat.V)])
    assert np.all(np.isfinite(got[clean]))
    bad = ~np.isfinite(got)
    # the link's row 1 (forward, at its site) and column 2 (backward, at its far end); the rest stays finite
    assert bad[200, :, 1].all() and not bad[200, :, 0].any() and not bad[200, :, 2].any()
    far = int(lat.fwd[200, 3])
    assert bad[far, :, 2].all() and not bad[far, :, 0].any() and not bad[far, :, 1].any()
    # a spinor component: its own at its site; two of the four spins of every neighbour, all colours
    assert bad[17].sum() == 1 and bad[17, 2, 1]
    for n in touched - {17, 200, far}:
        assert bad[n].all(axis=1).sum() >= 2


@pytest.mark.parametrize("shift", [0, 8])
def test_fields_on_8_byte_boundaries(api, shift):
    """The C ABI asks for the alignment of a double: the same numbers through
    the paths for 16-byte and for 8-byte boundaries."""
    import torch
    dims, block = (4, 4, 4, 6), (2, 2, 2, 3)
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5, nrhs=2)
    h = api.dd_init(dims, block, 0.13, max_rhs=2)
    ref = dev(np.zeros_like(psi))
    api.dd_apply_D(h, ref, dev(psi), dev(U), api.DD_OP_DDAG, api.DD_PREC_F64, 2)

    def at(a):
        flat = torch.zeros(2 * a.size + 2, dtype=torch.float64, device="cuda")
        flat[shift // 8:shift // 8 + 2 * a.size] = dev(a).view(torch.float64).reshape(-1)
        return flat, flat.data_ptr() + shift
    bufs = [at(np.zeros_like(psi)), at(psi), at(U)]
    api.dd_apply_D(h, bufs[0][1], bufs[1][1], bufs[2][1], api.DD_OP_DDAG, api.DD_PREC_F64, 2)
    got = host(bufs[0][0])[shift // 8:shift // 8 + 2 * psi.size].view(np.complex128).reshape(psi.shape)
    assert np.array_equal(got, host(ref))


def hop_bad(bad_u, bad_psi, lat):
    """Which components of H psi a number that is not finite reaches: the projection joins two spins of a neighbour,
    the link all colours whose entry or whose component is not finite."""
    out = np.zeros_like(bad_psi)
    for a in range(4):
        pair = np.abs(GAMMA_AXIS[a]).argmax(1)
        for y, links in ((lat.fwd[:, a], bad_u[:, a]), (lat.bwd[:, a], np.swapaxes(bad_u[lat.bwd[:, a], a], 1, 2))):
            w = bad_psi[y]
            w = w | w[:, pair]
            out |= (links[:, None, :, :] | w[:, :, None, :]).any(3)
    return out


@pytest.mark.parametrize("shift", [0, 8])
@pytest.mark.parametrize("op", ["D", "DDAG", "HEO", "DTILDE", "DTILDE_DAG"])
def test_non_finite_numbers_of_every_operator(api, op, shift):
    """The same components for every operator, on 16- and on 8-byte
    boundaries; all others equal to those of the clean fields."""
    import torch
    dims, block = (4, 4, 6, 4), (2, 2, 3, 2)
    lat = geometry.Lattice(dims, block)
    parity = geometry_parity(lat)
    sites = {"HEO": np.flatnonzero(parity == 1), "DTILDE": np.flatnonzero(parity == 0)}.get(op.split("_")[0],
                                                                                           np.arange(lat.V))
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5)
    mask = np.zeros(lat.V, dtype=bool)
    mask[sites] = True
    psi[~mask] = 0
    h = api.dd_init(dims, block, 0.13)

    def at(a):
        flat = torch.zeros(2 * a.size + 2, dtype=torch.float64, device="cuda")
        flat[shift // 8:shift // 8 + 2 * a.size] = dev(a).view(torch.float64).reshape(-1)
        return flat, flat.data_ptr() + shift

    def apply(U, psi):
        bufs = [at(np.zeros_like(psi[sites])), at(psi[sites]), at(U)]
        api.dd_apply_D(h, bufs[0][1], bufs[1][1], bufs[2][1], getattr(api, "DD_OP_" + op), api.DD_PREC_F64, 1)
        n = 2 * psi[sites].size
        return host(bufs[0][0])[shift // 8:shift // 8 + n].view(np.complex128).reshape(psi[sites].shape)

    clean = apply(U, psi)
    U[200, 3, 1, 2] = np.nan
    psi[sites[17], 2, 1] = np.inf
    got = apply(U, psi)
    bad_u, bad_psi = ~np.isfinite(U), ~np.isfinite(psi)
    hop = hop_bad(bad_u, bad_psi, lat)
    if op == "HEO":
        want = hop[parity == 0]
    elif op.startswith("DTILDE"):
        hop[parity == 0] = False
        want = (hop_bad(bad_u, hop, lat) | bad_psi)[parity == 0]
    else:
        want = hop | bad_psi
    assert np.array_equal(~np.isfinite(got), want)
    assert want.any() and not want.all()
    ok = ~want
    assert np.abs(got[ok] - clean[ok]).max() <= 1e-14 * np.abs(clean).max()


@pytest.mark.parametrize("op", ["D", "HEO", "DTILDE"])
def test_output_over_the_input(api, op):
    """Not promised by the interface, but it works as it always has."""
    dims, block = (4, 4, 4, 6), (2, 2, 2, 3)
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5)
    if op != "D":
        psi = psi[: psi.shape[0] // 2]
    h = api.dd_init(dims, block, 0.13)
    ref, io, Ud = dev(np.zeros_like(psi)), dev(psi), dev(U)
    api.dd_apply_D(h, ref, dev(psi), Ud, getattr(api, "DD_OP_" + op), api.DD_PREC_F64, 1)
    api.dd_apply_D(h, io, io, Ud, getattr(api, "DD_OP_" + op), api.DD_PREC_F64, 1)
    assert np.array_equal(host(io), host(ref))


def geometry_parity(lat):
    x = np.stack(np.meshgrid(*(np.arange(d) for d in lat.dims), indexing="ij"))
    return x.sum(0).reshape(-1, order="F") % 2


@pytest.mark.parametrize("kind", ["spinor", "spinor mixed", "link"])
def test_subnormal_numbers(api, kind):
    """Subnormal entries are numbers like all others: the hops between blocks
    (their sum alone) against extended precision, to the bound above and half
    a unit of the smallest number for a subnormal result."""
    dims, block, kappa = (4, 4, 6, 4), (1, 1, 1, 1), 0.125
    lat = geometry.Lattice(dims, block)
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5)
    if kind == "spinor":
        psi = psi * 2.0 ** -1060
    elif kind == "spinor mixed":  # largest entries normal, others below the normal range
        psi = psi * 2.0 ** -1020
        psi[:, 1::2] *= 2.0 ** -14
    else:
        U, psi = U * 2.0 ** -1050, psi * 2.0 ** 600
    h = api.dd_init(dims, block, kappa)
    out = dev(np.zeros_like(psi))
    api.dd_apply_D(h, out, dev(psi), dev(U), api.DD_OP_INTER, api.DD_PREC_F64, 1)
    got = host(out)
    hop, mag = hop_extended(U, psi, lat)
    ref = -LD(kappa) * hop
    err = np.abs(got.astype(LD) - ref).max((1, 2)).astype(np.longdouble)
    top = np.abs(ref).max((1, 2))
    assert np.abs(ref).max() > 0 and np.all(err <= np.sqrt(2) * (2.0 ** -53 * top + kappa * 2.0 ** -54 * mag
                                                               + np.longdouble(2.0) ** -1075 * 2))


def own_terms(U, psi, lat):
    """Per component of H psi the sum of |link entry| (|upper| + |lower|) over its own products."""
    out, U, psi = np.zeros(psi.shape, dtype=np.longdouble), np.abs(U.astype(LD)), np.abs(psi.astype(LD))
    for a in range(4):
        pair = np.abs(GAMMA_AXIS[a]).argmax(1)
        for y, links in ((lat.fwd[:, a], U[:, a]), (lat.bwd[:, a], np.swapaxes(U[lat.bwd[:, a], a], 1, 2))):
            w = psi[y]
            out += np.einsum("sij,skj->ski", links, w + w[:, pair])
    return out


@pytest.mark.parametrize("op", ["D", "INTER", "HEO", "DTILDE"])
@pytest.mark.parametrize("kind", ["colour 1e-6", "colour 1e-18", "colour 1e-200", "spin 1e-9", "links", "one spin",
                                  "spread", "plain"])
def test_each_component_keeps_the_accuracy_of_fp64(api, op, kind):
    """Entries far below the largest of their site, where no link mixes them
    with larger ones.  Per component, relative to its own terms: FP64 has one
    rounding for the projection, six for a colour product and eight for the
    hops; the integer form up to 8.5 units of 2^-56 of the largest product a
    hop (3 dropped, 1 rounded, 4.5 of the inputs), eight hops, for a component
    whose largest hop is above 2^-3 of it: 68 x 2^-53."""
    dims, block, kappa = (4, 6, 4, 8), (2, 3, 2, 4), 0.125
    lat = geometry.Lattice(dims, block)
    parity = geometry_parity(lat)
    rng = np.random.default_rng(3)
    U, psi = synthetic.random_gauge(dims, 0.4, 2), synthetic.random_spinor(dims, 5)
    if kind.startswith("colour") or kind == "spin 1e-9":
        if kind.startswith("colour"):
            U = np.where(np.eye(3, dtype=bool), np.exp(2j * np.pi * rng.random(U.shape[:2]))[..., None, None], 0)
            psi[:, :, 1] *= float(kind.split()[1])
        else:
            psi[:, 2:] *= 1e-9
    elif kind == "links":
        U = U * np.exp(rng.uniform(-40, 0, U.shape)) + np.eye(3)
        psi[:, :, 2] *= 1e-25
    elif kind == "one spin":
        psi[:, [0, 2, 3]] = 0
    elif kind == "spread":
        psi = psi * np.exp(12 * rng.standard_normal(psi.shape))
    sites = {"HEO": parity == 1, "DTILDE": parity == 0}.get(op, parity >= 0)
    psi[~sites] = 0
    h = api.dd_init(dims, block, kappa)
    out = dev(np.zeros_like(psi[sites]))
    api.dd_apply_D(h, out, dev(psi[sites]), dev(U), getattr(api, "DD_OP_" + op), api.DD_PREC_F64, 1)
    got, k = host(out), LD(kappa)
    if op == "INTER":
        # only the hops that cross block faces: those of the lattice without the ones inside
        inside = api.dd_init(dims, block, kappa)
        blk = dev(np.zeros_like(psi))
        api.dd_apply_D_block(inside, blk, dev(psi), dev(U), 3, api.DD_PREC_F64, 1)
        got = got + host(blk)
        ref, terms = psi - k * hop_extended(U, psi, lat)[0], np.abs(psi) + kappa * own_terms(U, psi, lat)
    else:
        hop, terms = hop_extended(U, psi, lat)[0], own_terms(U, psi, lat)
        if op == "D":
            ref, terms = psi - k * hop, np.abs(psi) + kappa * terms
        elif op == "HEO":
            ref, terms = hop[parity == 0], terms[parity == 0]
        else:
            hop[parity == 0] = 0
            terms[parity == 0] = 0
            ref = (psi - k * k * hop_extended(U, hop, lat)[0])[parity == 0]
            terms = (np.abs(psi) + 2 * kappa * kappa * own_terms(U, terms, lat))[parity == 0]
    err = np.abs(got.astype(LD) - ref).astype(np.longdouble)
    bound = np.sqrt(2) * (68 + 2) * np.longdouble(2.0) ** -53 * terms
    print(op, kind, "largest error in units of 2^-53 of a component's own terms:",
          float((err[terms > 0] / terms[terms > 0]).max() * 2.0 ** 53))
    assert np.all(err <= bound), float((err[terms > 0] / terms[terms > 0]).max() * 2.0 ** 53)
