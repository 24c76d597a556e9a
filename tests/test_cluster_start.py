"""Order of the first accesses to another thread block's shared memory: a
thread block of a cluster may touch it only after a cluster barrier has shown
that the other one runs.  A late start is a matter of scheduling and does not
show in results, so this reads the kernel's source."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1112_1243_gb300", "csrc")


def kernels(text):
    """(name, body) of every __global__ function, comments taken out."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\([^{;]*\)\s*\{", text):
        depth, k = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), text[m.end():k]


def first_accesses():
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as fh:
            for name, body in kernels(fh.read()):
                if "this_cluster" in body:
                    yield f, name, body


def test_a_cluster_barrier_comes_before_the_first_remote_access():
    found = 0
    for f, name, body in first_accesses():
        remote = re.search(r"map_shared_rank|eo_team_total|eo_sum|eo_total|eo_bicgstab", body)
        assert remote, (f, name)
        found += 1
        head = body[:remote.start()]
        barrier = head.rfind("cluster.sync()")
        assert barrier >= 0, (f, name, "no cluster barrier before the first remote access")
        # outside the loop over items: passed before the first item
        assert head.index("for (;;)") > barrier, (f, name)
    assert found == 1


@pytest.mark.gpu
def test_first_items_of_large_blocks_arrive():
    """Few items for many clusters, one launch after another on fresh
    handles: every item is solved once, with the same bits each time."""
    import numpy as np

    from gpu_util import dev, host, lib_api
    from oracle import geometry, heatbath
    from paper_1112_1243_gb300 import synthetic
    api = lib_api()
    dims, block = (12, 12, 12, 12), (6, 6, 6, 6)
    lat = geometry.Lattice(dims, block)
    U = synthetic.random_gauge(dims, 0.3, 4)
    Up, _ = heatbath.gauge_update(U, lat, 5.3, 1, 0, 21, 4, colour_mask=3)
    Ud, Upd, first = dev(U), dev(Up), None
    for _ in range(3):
        h = api.dd_init(dims, block, 0.12, max_rhs=1)
        for npos in (1, 3, lat.nblocks):
            got = host(api.dd_block_ratios_range(h, Ud, Upd, 0, npos, 1, 9, 3))
            if npos == lat.nblocks:
                first = got if first is None else first
                assert np.array_equal(got, first) and np.all(got != 0)
        assert api.dd_status(h)[0] == 0
