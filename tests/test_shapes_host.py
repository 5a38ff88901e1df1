"""Which build of the pair kernel a tuning request gets (pick_variant, host only):
without span binning, hist_mode 3 is the build with a column per thread and no
span code, in every tile size that bins spans, and a plan's reported tuning
picks the same build again."""
import pytest

from host_calls import run

BODY = """
    wtheta_tune t = {};
    t.threads = atoi(argv[1]); t.points_per_thread = 8; t.hist_mode = atoi(argv[2]);
    t.deferred = atoi(argv[3]); t.span_bins = atoi(argv[4]);
    const Variant* v = pick_variant(&t, atoi(argv[5]), 700, 232448);
    if (!v) { printf("none\\n"); return 0; }
    printf("%d %d %d %d %zu\\n", v->nt, v->r, v->hm, v->def, v->smem(atoi(argv[5]), 700));
"""


@pytest.mark.parametrize("threads", [32, 64, 128])
@pytest.mark.parametrize("hist_mode", [0, 3])
@pytest.mark.parametrize("deferred", [0, 1])
@pytest.mark.parametrize("K", [1, 24])
def test_no_spans_means_a_column_per_thread(tmp_path, threads, hist_mode, deferred, K):
    (no,), (yes,) = (run(tmp_path, BODY, [threads, hist_mode, deferred, s, K]) for s in (2, 1))
    assert [int(x) for x in no[:4]] == [threads, 8, 3, 2]
    assert [int(x) for x in yes[:4]] == [threads, 8, 3, 0]
    # as reported by a plan (hist_mode 3, deferred 1) and asked for again
    (again,) = run(tmp_path, BODY, [threads, 3, 1, 2, K])
    assert again == no


def test_no_request_without_spans_gets_span_code(tmp_path):
    """Every combination of the tuning's fields: what is refused is refused with and
    without spans alike, and without them the build has no span jobs (deferred 0
    with hist_mode 3 or 4 is a span build)."""
    out = run(tmp_path, """
    for (int K : {1, 24, 100, 256}) for (int n_lut : {20, 1000}) for (int t : {0, 32, 64, 128, 256, 512})
    for (int r : {0, 8, 16}) for (int h = 0; h <= 4; ++h) for (int j = 0; j <= 2; ++j)
    for (int d = 0; d <= 2; ++d) {
        wtheta_tune u = {};
        u.threads = t; u.points_per_thread = r; u.hist_mode = h; u.j_per_screen = j; u.deferred = d;
        u.span_bins = 2;
        const Variant* no = pick_variant(&u, K, n_lut, 232448);
        u.span_bins = 1;
        const Variant* yes = pick_variant(&u, K, n_lut, 232448);
        const bool spans = no && no->def == 0 && no->hm != kHistWarp;
        printf("%d %d %d %d %d\\n", !no == !yes, spans, no ? no->nt * no->r : 0,
               yes ? yes->nt * yes->r : 0, no && no->smem(K, n_lut) > 232448);
    }""")
    assert len(out) == 4 * 2 * 6 * 3 * 5 * 3 * 3
    for same, spans, tile, tile_yes, too_big in out:
        assert same == "1" and spans == "0" and tile == tile_yes and too_big == "0"


def test_other_requests_without_spans(tmp_path):
    deferred, warp, red, plain = (run(tmp_path, BODY, [128, h, d, 2, 24])[0]
                                  for h, d in ((3, 2), (2, 0), (4, 0), (1, 0)))
    assert deferred[:4] == ["128", "8", "3", "1"]
    assert warp[:4] == ["128", "8", "2", "0"]
    assert red[:4] == ["128", "8", "4", "2"]
    assert plain[:4] == ["128", "8", "4", "2"]   # (mode 1 is built deferred only)
    # 256 bins: a column per thread only if it is asked for
    (chosen,), (asked,) = (run(tmp_path, BODY, [128, h, 0, 2, 256]) for h in (0, 3))
    assert chosen[2:4] == ["4", "2"] and asked[2:4] == ["3", "2"]
