"""A server and a batch plan keep the shared-memory size of their launches: a
count with fewer bins in between, which needs less, leaves them working."""
import threading

import numpy as np
import pytest

from paper_1208_3658_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def inputs():
    fp = synth.Patch(120.0, 15.0, 20.0, 35.0)
    d = synth.clustered(fp, 40_000, 800, 3.0, 7, "test", "data")
    r = synth.uniform(fp, 40_001, 7, "test", "random")
    return d, r


def _count(W, dd, rr, e):
    c = torch.zeros((3, len(e) + 1), dtype=torch.int64, device="cuda")
    W.wtheta_count_wtheta(dd, rr, False, e, c)
    torch.cuda.synchronize()
    return c.cpu().numpy().astype(np.uint64)


def test_server_and_plan_after_counts_with_fewer_bins(inputs):
    from paper_1208_3658_gb300 import wtheta as W
    d, r = inputs
    dd, rr = torch.from_numpy(d).cuda(), torch.from_numpy(r).cuda()
    many, one = W.wtheta_edges(1 / 60, 10.0, 60), W.wtheta_edges(1 / 60, 10.0, 1)
    want = _count(W, dd, rr, many)
    plan = W.wtheta_batch_plan([(dd, rr)], many, tune=dict(threads=128))
    out = torch.zeros(3 * (len(many) + 1), dtype=torch.int64, device="cuda")
    srv = W.wtheta_server_create(many, 1 << 30)
    try:
        for _ in range(2):
            _count(W, dd, rr, one)
            q = W.wtheta_server_submit(srv, d, r)
            done, c, _w = W.wtheta_server_wait(srv, q, 60_000)
            assert done and np.array_equal(c, want)
            W.wtheta_server_release(srv, q)
            _count(W, dd, rr, one)
            W.wtheta_batch_run(plan, out)
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy().astype(np.uint64).reshape(want.shape), want)
    finally:
        W.wtheta_server_destroy(srv)
        W.wtheta_batch_free(plan)


def test_threads_with_different_bins(inputs):
    from paper_1208_3658_gb300 import wtheta as W
    d, r = inputs
    sets = [W.wtheta_edges(1 / 60, 10.0, k) for k in (1, 40, 60, 250)]
    bad = []

    def work(e):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                dd, rr = torch.from_numpy(d).cuda(), torch.from_numpy(r).cuda()
                c = torch.zeros((3, len(e) + 1), dtype=torch.int64, device="cuda")
                first = None
                for _ in range(20):
                    W.wtheta_count_wtheta(dd, rr, False, e, c, stream=s)
                    s.synchronize()
                    got = c.cpu().numpy()
                    first = got if first is None else first
                    assert np.array_equal(got, first)
        except Exception as x:  # noqa: BLE001
            bad.append((len(e) - 1, x))

    ts = [threading.Thread(target=work, args=(e,)) for e in sets]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad
