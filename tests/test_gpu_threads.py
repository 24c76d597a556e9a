"""Host threads with a handle and a stream each: launch attributes belong to
the process, so a thread with a smaller launch shape must not take the shared
memory from under a larger one between its attribute call and its launch."""
import threading

import numpy as np
import pytest

from gpu_util import dev, host, lib_api
from paper_1112_1243_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    return lib_api()


def in_threads(jobs, rounds):
    """Every job (a callable) `rounds` times in a thread of its own, all at once: their results or errors."""
    import torch
    start, out = threading.Barrier(len(jobs)), [None] * len(jobs)

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                res = [jobs[k]() for _ in range(rounds)]
                torch.cuda.current_stream().synchronize()
                out[k] = [r.cpu().numpy() for r in res]
        except Exception as e:  # noqa: BLE001 - reported by the caller
            out[k] = e

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return out


def check(make, shapes, rounds):
    """make(shape) -> callable; the same bits in threads as one after the other."""
    want = [host(make(s)()) for s in shapes]
    got = in_threads([make(s) for s in shapes], rounds)
    for g, w in zip(got, want):
        assert not isinstance(g, Exception), g
        assert all(np.array_equal(r, w) for r in g)


def test_block_solver_shapes_in_threads(api):
    import torch
    dims, block = (4, 4, 4, 4), (2, 2, 2, 2)
    U = synthetic.random_gauge(dims, 0.3, 4)
    Ud, Upd = dev(U), dev(U)
    api.dd_gauge_update(api.dd_init(dims, block, 0.12), Upd, 1, 5.3, 1, 0, 21, 4)
    torch.cuda.synchronize()

    def make(tpb):
        hs = {}

        def job():
            if not hs:
                hs["h"] = api.dd_init(dims, block, 0.12)
                api.dd_set_tuning(hs["h"], block_tpb=tpb, block_ctas_per_sm=2)
            return api.dd_block_ratios_range(hs["h"], Ud, Upd, 0, 16, 1, 9, 3)
        return job

    check(make, [256, 128, 256, 128], 300)


def test_exact_block_determinants_in_threads(api):
    import torch
    fields = {}
    for block in ((2, 2, 2, 2), (1, 2, 2, 2)):
        dims = tuple(2 * b for b in block)
        fields[block] = (dims, dev(synthetic.random_gauge(dims, 0.3, 4)))
    torch.cuda.synchronize()

    def make(block):
        dims, U = fields[block]
        hs = {}

        def job():
            if not hs:
                hs["h"] = api.dd_init(dims, block, 0.12, features=api.DD_FEAT_EXACT)
            return api.dd_logdet_exact(hs["h"], U, 1)
        return job

    check(make, [(2, 2, 2, 2), (1, 2, 2, 2), (2, 2, 2, 2), (1, 2, 2, 2)], 300)
