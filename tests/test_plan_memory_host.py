"""The scratch of a batch plan and of region counts (no GPU): the spheres and local
coordinates lie in buffers that the sort no longer reads, inside their own part,
and a plan takes no more than about 65 bytes per point."""
import pytest

from host_calls import run

BODY = """
    const int nc2 = atoi(argv[1]);
    const long long n = atoll(argv[2]), np = atoll(argv[3]);
    PlanLayout Y = plan_scratch(nc2, n, np);
    unsigned char* base = (unsigned char*)4096;
    Prepared q = regions_layout(base + Y.all, base + Y.lab, base + Y.sort, n, np);
    auto at = [&](const void* p) { return (long long)((const unsigned char*)p - base); };
    printf("%zu %zu %zu %zu %zu %zu %zu %zu\\n", Y.cats, Y.offs, Y.x, Y.lab, Y.sort, Y.all, Y.bytes,
           order_bytes(n, 1));
    printf("%lld %lld %lld %lld %lld %lld\\n", at(q.p32), at(q.c32), at(q.groups), at(q.l32), at(q.kap),
           q.l_stride);
"""


@pytest.mark.parametrize("nc2,n,n_pad", [(2, 4, 512), (2, 10**6, 1000448), (32, 3 * 10**7, 30015488),
                                         (1200, 180000, 1228800), (65536, 131072, 16777216),
                                         (4, 4100, 5120)])
def test_plan_parts(tmp_path, nc2, n, n_pad):
    (off, view) = run(tmp_path, BODY, [nc2, n, n_pad])
    cats, offs, x, lab, sort, all_, end, order = (int(v) for v in off)
    p32, c32, groups, l32, kap, stride = (int(v) for v in view)
    a4 = -(-4 * n // 256) * 256
    assert cats >= 8 and cats + 16 * nc2 <= offs and offs + 16 * (nc2 + 1) <= x
    assert x + 24 * n <= lab and lab + 4 * n <= sort and sort + order <= all_
    assert groups == lab and groups + 2 * n_pad <= sort          # in the labels' place
    assert l32 == sort + 2 * a4                                  # after both index buffers
    assert stride == n_pad and l32 + 12 * n_pad <= kap and kap + n_pad // 4 <= all_
    assert p32 == all_ and p32 + 16 * n_pad <= c32 and c32 + n_pad // 2 <= end
    assert all(v % 256 == 0 for v in (x, lab, sort, all_, groups, l32, kap, p32, c32))
    if n >= 10**6:
        assert end <= 65.5 * n_pad + 2e5
