"""The device scratch of a w(theta) count and of a shard of one (wtheta_layout):
what the launches write lies inside its own part of the allocation, with and
without skipping far tile pairs.  A shard split reads tile caps either way."""
import pytest

from host_calls import run

CAP_BYTES = 32   # a tile cap: four doubles


@pytest.mark.parametrize("shards", [1, 2, 200])
@pytest.mark.parametrize("cull", [0, 1])
@pytest.mark.parametrize("nd,nr", [(1, 0), (700, 5000), (30000, 30011), (1024000, 1024000)])
def test_parts_hold_what_is_written(tmp_path, nd, nr, cull, shards):
    T = 512
    (line,) = run(tmp_path, """
    long long nd = atoll(argv[1]), nr = atoll(argv[2]), T = 512;
    long long pd = round_up(nd, T), pr = round_up(nr, T), td = pd / T, tr = pr / T;
    long long items = td * (td + 1) / 2 + td * tr + tr * (tr + 1) / 2;
    WthetaLayout Y = wtheta_layout(nd, pd, nr, pr, T, atoi(argv[3]) != 0, atoi(argv[4]), items);
    printf("%zu %zu %zu %zu %zu %zu %lld %zu %zu\\n", Y.prep, Y.caps, Y.rows, Y.row0, Y.lists,
           Y.bytes, Y.n_caps, prepare_joint_bytes(nd, pd, nr, pr), sizeof(TileCap));
    """, [nd, nr, cull, shards])
    prep, caps, rows, row0, lists, end, n_caps, prep_bytes, cap_size = (int(x) for x in line)
    td, tr = -(-nd // T), -(-nr // T)
    items = td * (td + 1) // 2 + td * tr + tr * (tr + 1) // 2
    assert cap_size == CAP_BYTES
    need_caps = cull or shards > 1
    assert n_caps == (td + tr if need_caps else 0)
    assert prep >= 256 + 1024 + 1024 + 24 and prep + prep_bytes <= caps
    assert caps + CAP_BYTES * n_caps <= rows
    assert rows + (8 * (2 * td + tr) if shards > 1 else 0) <= row0
    assert row0 + (24 if shards > 1 else 0) <= lists
    assert lists + (4 * items if cull else 0) <= end
    assert all(x % 8 == 0 for x in (prep, caps, rows, row0, lists))
