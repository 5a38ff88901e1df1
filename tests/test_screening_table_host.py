"""The screening table (build_table, no GPU): for values around every edge and all
over the range, a value outside its entry's band lies in the slot that the entry
gives, and a value inside the band of an edge's entry is next to that edge.
Buckets of an octave or more take one edge each and bands that fit the entry."""
import numpy as np
import pytest

from host_calls import run
from paper_1208_3658_gb300 import wtheta as W

SETS = [(1 / 60, 5.0, 16, W.BINS_LN), (1 / 60, 10.0, 24, W.BINS_LN), (0.5 / 60, 20.0, 256, W.BINS_LN),
        (0.0, 180.0, 36, W.BINS_LINEAR), (0.0, 180.0, 256, W.BINS_LINEAR), (179.0, 180.0, 9, W.BINS_LINEAR),
        (0.01, 100.0, 4, W.BINS_LN), (1e-7, 1e-4, 5, W.BINS_LN), (1e-5, 1.0, 12, W.BINS_LN),
        (0.0, 1.0, 1, W.BINS_LINEAR), (90.0, 180.0, 1, W.BINS_LINEAR)]

BODY = """
    std::vector<double> e;
    for (int i = 1; i < argc; ++i) e.push_back(atof(argv[i]));
    const int K = (int)e.size() - 1;
    static BinTable t;
    if (build_table(e.data(), K, &t)) return 1;
    auto bits_of = [](float f) { unsigned u; __builtin_memcpy(&u, &f, 4); return u; };
    auto value = [](unsigned u) { float f; __builtin_memcpy(&f, &u, 4); return f; };
    long long bad = 0, band = 0, n = 0;
    auto check = [&](unsigned bits) {
        if (bits > bits_of(4.1f)) return;
        const double s = value(bits);
        int slot = 0;
        while (slot <= K && t.c64[slot] <= s) ++slot;   // edges at or below s
        long long idx = (long long)(bits >> t.shift) - t.base;
        idx = idx < 0 ? 0 : idx >= t.n_lut ? t.n_lut - 1 : idx;
        const unsigned x = t.lut[idx][0], y = t.lut[idx][1], w = y >> kLutWidthShift;
        const int k = (int)(y & kLutSlot);
        ++n;
        if (bits < x) bad += slot != k;
        else if (bits - x > w) bad += slot != k + 1;
        else {
            ++band;
            if (y & kLutSeveral) bad += bits > t.h_top;
            else bad += slot != k && slot != k + 1;
        }
    };
    for (int k = 0; k <= K; ++k) {
        const unsigned b = bits_of((float)t.c64[k]);
        for (int d = -3000; d <= 3000; ++d) if ((long long)b + d >= 0) check(b + d);
        for (int sh = 12; sh < 24; ++sh) { check(b + (1u << sh)); if (b >> sh) check(b - (1u << sh)); }
    }
    for (unsigned b = 0; b < bits_of(4.1f); b += 997) check(b);
    printf("%lld %lld %lld %d %d %d\\n", bad, band, n, t.n_lut, t.shift, t.n_complex);
"""


@pytest.mark.parametrize("lo,hi,K,mode", SETS)
def test_entries_place_every_value(tmp_path, lo, hi, K, mode):
    e = W.wtheta_edges(lo, hi, K, mode)
    ((bad, band, n, n_lut, shift, n_complex),) = run(tmp_path, BODY, [repr(float(x)) for x in e])
    assert int(bad) == 0 and int(band) > 0 and int(n) > 10 ** 6
    assert 0 < int(n_lut) <= 1024
    assert int(shift) <= 22 or int(n_complex) == 0


def test_an_octave_per_bucket_where_one_edge_lies_in_each(tmp_path):
    """16 bins from 1 arcmin to 5 degrees lie about an octave apart."""
    e = W.wtheta_edges(1 / 60, 5.0, 16)
    ((_, _, _, n_lut, shift, _),) = run(tmp_path, BODY, [repr(float(x)) for x in e])
    assert (int(shift), int(n_lut)) == (23, 17)
