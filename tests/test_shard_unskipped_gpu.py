"""Shards of a w(theta) whose far tile pairs are not skipped (a top edge of 180
degrees, or skip_far = 2) add up to the oracle's counts."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1208_3658_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top,K,tune", [(180.0, 12, None), (5.0, 8, dict(skip_far=2))])
def test_unskipped_shards_sum_to_the_oracle(top, K, tune):
    from paper_1208_3658_gb300 import wtheta as W
    fp = synth.Patch(30.0, 8.0, 10.0, 18.0)
    D = O.radec_to_xyz(synth.clustered(fp, 15_001, 300, 3.0, 3, "test", "data"))
    R = O.radec_to_xyz(synth.uniform(fp, 20_002, 3, "test", "random"))
    e = W.wtheta_edges(0.0, top, K, W.BINS_LINEAR)
    want = np.stack([O.count_xyz(D, None, e, True), O.count_xyz(D, R, e, False),
                     O.count_xyz(R, None, e, True)])
    d, r = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (D, R))
    for S in (2, 3, 7):
        acc = np.zeros((3, K + 2), np.uint64)
        for s in range(S):
            c = torch.zeros((3, K + 2), dtype=torch.int64, device="cuda")
            W.wtheta_count_wtheta_shard(d, r, True, e, s, S, c, tune=tune)
            torch.cuda.synchronize()
            acc += c.cpu().numpy().astype(np.uint64)
        assert np.array_equal(acc, want), S
