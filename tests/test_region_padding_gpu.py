"""Regions and mocks whose padding outweighs their points, and more counts in one
launch than one pass of the prefix scan takes (1024): counts equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1208_3658_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("R,n_d,n_r", [(33, 900, 1100), (64, 3000, 5000), (2, 5000, 3)])
def test_many_regions(R, n_d, n_r):
    """33 regions are 33 * 34 + 33 * 33 = 2211 region pairs."""
    from paper_1208_3658_gb300 import wtheta as W
    fp = synth.Patch(30.0, 8.0, 10.0, 18.0)
    D = O.radec_to_xyz(synth.clustered(fp, n_d, max(1, n_d // 50), 3.0, 3, "test", "data"))
    Rn = O.radec_to_xyz(synth.uniform(fp, n_r, 3, "test", "random"))
    rng = np.random.default_rng(R)
    ld, lr = (rng.integers(0, R, n).astype(np.int32) for n in (n_d, n_r))
    e = W.wtheta_edges(1.0 / 60, 5.0, 6)
    c = torch.zeros((3, R, R, len(e) + 1), dtype=torch.int64, device="cuda")
    sizes = W.wtheta_count_regions(_dev(D), _dev(ld), _dev(Rn), _dev(lr), e, R, c,
                                   coords_are_xyz=True)
    torch.cuda.synchronize()
    want = O.count_regions(D, ld, Rn, lr, e, R)
    assert np.array_equal(c.cpu().numpy().astype(np.uint64), np.asarray(want).reshape(c.shape))
    assert np.array_equal(np.asarray(sizes).reshape(2, R),
                          [np.bincount(ld, minlength=R), np.bincount(lr, minlength=R)])


def test_many_small_mocks():
    """400 mocks: 1200 counts, each catalogue a fraction of a tile."""
    from paper_1208_3658_gb300 import wtheta as W
    fp = synth.Patch(30.0, 4.0, 10.0, 14.0)
    e = W.wtheta_edges(1.0 / 60, 5.0, 5)
    mocks = [(O.radec_to_xyz(synth.uniform(fp, 5 + i % 37, i, "test", "data")),
              O.radec_to_xyz(synth.uniform(fp, 9 + i % 53, i, "test", "random"))) for i in range(400)]
    cats = [(_dev(d), _dev(r)) for d, r in mocks]
    plan = W.wtheta_batch_plan(cats, e, tune=dict(threads=128), coords_are_xyz=True)
    out = torch.zeros((400, 3, len(e) + 1), dtype=torch.int64, device="cuda")
    for _ in range(2):
        W.wtheta_batch_run(plan, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy().astype(np.uint64)
    W.wtheta_batch_free(plan)
    for m in range(0, 400, 7):
        d, r = mocks[m]
        assert np.array_equal(got[m], [O.count_xyz(d, None, e, True), O.count_xyz(d, r, e, False),
                                       O.count_xyz(r, None, e, True)]), m


def test_plan_memory_per_point():
    from paper_1208_3658_gb300 import wtheta as W
    n = 2_000_000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    p = torch.rand(n, 2, generator=g, device="cuda", dtype=torch.float64) * 20.0
    e = W.wtheta_edges(1.0 / 60, 0.05, 4)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = W.wtheta_batch_plan([(p, p)], e, tune=dict(threads=128, skip_far=2))
    after = torch.cuda.mem_get_info()[0]
    W.wtheta_batch_free(plan)
    # 64.75 B a point and allocation granularity
    assert before - after < 66.5 * 2 * n + (8 << 20)
