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
