"""The persistent block solver in even-odd form (block_eo_kernel) against the
oracle: block shapes with odd extents along any axis (vectors kept at full
length for an odd extent along axis 0), one- and two-site extents, more and
fewer sites than threads, every thread-block size, blocks large enough for a
cluster of thread blocks, unchanged blocks."""
import numpy as np
import pytest

from gpu_util import dev, host, lib_api
from oracle import estimator, geometry, heatbath
from oracle.interp import interpolate
from paper_1112_1243_gb300 import synthetic

pytestmark = pytest.mark.gpu
KAPPA = 0.12


@pytest.fixture(scope="module")
def api():
    return lib_api()


def reference(U, Up, lat, n, seed, ctr):
    """ln_b of the oracle (solves to 1e-14) and the error that a relative
    residual of 1e-12 leaves: |delta ln| <= 2 (|eta| + |d|) |D_b^-1| 1e-12 |b|
    per factor, |D_b^-1| <= 1 / (1 - 8 kappa) for unitary links."""
    ln, tol = np.zeros(lat.nblocks), np.zeros(lat.nblocks)
    for i in range(n):
        Pi = estimator.Pieces(interpolate(U, Up, i / n, lat.active), lat, KAPPA)
        Pj = estimator.Pieces(interpolate(U, Up, (i + 1) / n, lat.active), lat, KAPPA)
        eta = estimator.block_noise(lat, i, seed, ctr)
        b = Pi.dirichlet(eta) - Pj.dirichlet(eta)
        d = Pj.dirichlet_solve(b)
        per = lambda v: np.bincount(lat.block_id, weights=v, minlength=lat.nblocks)
        sq = lambda v: np.sqrt(per(np.sum(np.abs(v) ** 2, axis=(1, 2))))
        ln += per(-(2 * np.sum(np.conj(eta) * d, axis=(1, 2)).real + np.sum(np.abs(d) ** 2, axis=(1, 2))))
        tol += 2 * (sq(eta) + sq(d)) / (1 - 8 * KAPPA) * 1e-12 * sq(b)
    return ln, tol + 1e-12


@pytest.mark.parametrize("dims,block,tpb", [
    ((6, 6, 6, 6), (3, 3, 3, 3), 256),
    ((6, 4, 4, 10), (3, 2, 2, 5), 64),
    ((4, 6, 10, 6), (2, 3, 5, 3), 128),
    ((8, 8, 8, 8), (4, 4, 4, 4), 256),
    ((8, 8, 8, 8), (4, 4, 4, 4), 64),
    ((12, 8, 4, 8), (6, 4, 2, 4), 256),
    ((2, 4, 4, 4), (1, 2, 2, 2), 256),
    ((20, 8, 8, 8), (5, 4, 4, 4), 128),
    ((12, 12, 12, 12), (6, 6, 6, 6), 256),
    ((14, 12, 12, 12), (7, 6, 6, 6), 128),
])
def test_block_shapes(api, dims, block, tpb):
    n = 2
    lat = geometry.Lattice(dims, block)
    U = synthetic.random_gauge(dims, 0.3, 4)
    cm = 1 if lat.active_mode == "intra" else 3
    Up, _ = heatbath.gauge_update(U, lat, 5.3, 1, 0, 21, 4, colour_mask=cm)
    h = api.dd_init(dims, block, KAPPA, max_rhs=n)
    api.dd_set_tuning(h, block_tpb=tpb, block_ctas_per_sm=2)
    ref, tol = reference(U, Up, lat, n, 9, 3)
    got = host(api.dd_block_ratios_range(h, dev(U), dev(Up), 0, lat.nblocks, n, 9, 3))
    assert np.all(np.abs(got - ref) <= tol)
    assert api.dd_status(h)[0] == 0
    # nothing proposed: exactly zero
    got = host(api.dd_block_ratios_range(h, dev(U), dev(U), 0, lat.nblocks, n, 9, 3))
    assert np.all(got == 0)


def test_source_of_small_rotations(api):
    """Links that differ only in entries far below their largest one: diagonal
    links with off-diagonal entries near 2^-26, of which the proposal changes
    2^-10 parts.  The reference takes the difference of the links in FP64 and
    scales it up before the operator adds it to the noise; what is left is
    that of the solve (reference(), relative to |b|)."""
    dims, block = (8, 4, 4, 8), (4, 2, 2, 4)
    lat = geometry.Lattice(dims, block)
    rng = np.random.default_rng(3)
    V = int(np.prod(dims))
    U = np.zeros((V, 4, 3, 3), dtype=np.complex128)
    ph = rng.uniform(0, 2 * np.pi, (V, 4, 3))
    ph[..., 2] = -ph[..., 0] - ph[..., 1]
    for k in range(3):
        U[..., k, k] = np.exp(1j * ph[..., k])
    off = rng.standard_normal((2, V, 4, 3, 3))
    off = (off[0] + 1j * off[1]) * (1 - np.eye(3)) * 2.0 ** -26
    change = 1 + 2.0 ** -10 * rng.standard_normal((V, 4, 3, 3))
    Up = U + off * np.where(lat.active[..., None, None], change, 1.0)
    U = U + off
    diff = (U - Up) * 2.0 ** 40  # exact differences, scaled to about 1
    assert 0 < np.abs(U - Up).max() < 2.0 ** -30
    eta = estimator.block_noise(lat, 0, 9, 3)
    b = 2.0 ** -40 * (estimator.Pieces(diff, lat, KAPPA).dirichlet(eta) - eta)
    d = estimator.Pieces(Up, lat, KAPPA).dirichlet_solve(b)
    per = lambda v: np.bincount(lat.block_id, weights=v, minlength=lat.nblocks)
    sq = lambda v: np.sqrt(per(np.sum(np.abs(v) ** 2, axis=(1, 2))))
    ref = per(-(2 * np.sum(np.conj(eta) * d, axis=(1, 2)).real + np.sum(np.abs(d) ** 2, axis=(1, 2))))
    tol = 2 * (sq(eta) + sq(d)) / (1 - 8 * KAPPA) * 1e-12 * sq(b)
    h = api.dd_init(dims, block, KAPPA, max_rhs=1)
    got = host(api.dd_block_ratios_range(h, dev(U), dev(Up), 0, lat.nblocks, 1, 9, 3))
    assert np.all(np.abs(got - ref) <= tol)
    assert api.dd_status(h)[0] == 0


def test_no_item_runs_to_its_iteration_cap(api):
    """Blocks of 8^4 near the critical mass: an inner solve whose rho has lost
    its accuracy goes on to its cap of 2000 iterations, as many as all 16 items
    of a launch need together.  Launches with other noise vectors therefore
    differ by far less than half of their iterations."""
    dims, block, kappa = (16, 16, 16, 16), (8, 8, 8, 8), 0.16
    U = dev(synthetic.random_gauge(dims, 0.2, 4))
    Up = U.clone()
    h = api.dd_init(dims, block, kappa, max_rhs=1)
    api.dd_gauge_update(h, Up, 3, 5.3, 1, 0, 21, 4)
    its = []
    for ctr in range(12):
        api.dd_kernel_timer(h, 1, 0, 1)
        got = host(api.dd_block_ratios_range(h, U, Up, 0, 16, 1, 9, ctr))
        st = api.dd_solver_stats(h, 2)
        assert np.all(np.isfinite(got)) and st["items"] == 16
        its.append(st["inner_iterations"])
    assert max(its) < 1.5 * min(its), its
    assert api.dd_status(h)[0] == 0
