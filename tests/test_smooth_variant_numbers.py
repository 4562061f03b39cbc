"""The variant numbers of mgk_smooth_variant_* are part of the interface (a caller may store one):
shapes and sweeps of every number of the row-marching family, new ones behind the old."""

MARCH = {1: [(240, 0, 2), (240, 0, 1), (112, 0, 2), (240, 0, 2), (240, 0, 2), (52, 0, 2)],
         0: [(120, 0, 1), (112, 0, 2), (248, 0, 1), (120, 0, 1), (22, 0, 2)]}


def test_marching_variants_keep_their_numbers(libmg):
    for f32, want in MARCH.items():
        assert [(t[0], t[1], n) for _, t, n in libmg.smooth_variants(bool(f32), 4)] == want
    assert libmg.lib().mgk_march_sweeps() == 2 and libmg.lib().mgk_march_sweeps_f64() == 1
