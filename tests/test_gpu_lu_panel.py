"""Panel launch of the dense LU (matrices above 384 rows): candidates exchanged
by tagged messages between its thread blocks.  Sizes: 24, 72 and 192 thread
blocks (one and two rounds of reads a lane), matrices that follow one another
in the same workspace; a number that is not finite ends in a status, for
one-block panels too.

Tolerance: 1e-9 relative against LAPACK, both backward-stable with partial
pivoting (about n 1e-16 times the condition number); the same matrix twice
gives the same bits."""
import numpy as np
import pytest

from gpu_util import dev, host, lib_api
from oracle import dirac, geometry
from paper_1112_1243_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    return lib_api()


@pytest.mark.parametrize("dims,block,check", [((2, 4, 2, 4), (1, 2, 1, 2), True), ((4, 4, 2, 6), (2, 2, 1, 3), True),
                                              ((8, 4, 4, 4), (2, 2, 2, 2), False)])
def test_panels_of_many_blocks(api, dims, block, check):
    lat = geometry.Lattice(dims, block)
    h = api.dd_init(dims, block, 0.12)
    fields = [synthetic.random_gauge(dims, 0.4, k) for k in (1, 2)]
    got = [float(host(api.dd_logdet_exact(h, dev(fields[k]), 0))[0]) for k in (0, 1, 0)]
    assert api.dd_status(h)[0] == 0
    assert got[0] == got[2] and got[0] != got[1]
    api.dd_lu_tensor_cores(h, False)
    fma = float(host(api.dd_logdet_exact(h, dev(fields[0]), 0))[0])
    assert abs(got[0] - fma) < 1e-9 * abs(fma)
    if check:
        for k in (0, 1):
            ref = dirac.logabsdet(dirac.dense_D(fields[k], lat, 0.12))
            assert abs(got[k] - ref) < 1e-9 * abs(ref)


@pytest.mark.parametrize("which", [0, 1, 2])
def test_nan_raises_a_status(api, which):
    """A column of NaN still has a pivot row: the status reads DD_ERR_NUMERIC
    and the next determinant is right."""
    dims, block = (2, 4, 2, 4), (1, 2, 1, 2)
    h = api.dd_init(dims, block, 0.12)
    U = synthetic.random_gauge(dims, 0.4, 1)
    ref = host(api.dd_logdet_exact(h, dev(U), which)).copy()
    bad = U.copy()
    bad[0, 1] = np.nan  # a link inside a block
    api.dd_logdet_exact(h, dev(bad), which)
    assert api.dd_status(h)[0] == api.DD_ERR_NUMERIC
    assert np.array_equal(host(api.dd_logdet_exact(h, dev(U), which)), ref)
    assert api.dd_status(h)[0] == 0
