"""The columns at which engine 50 adds the restriction's partial planes 1 and 3
(load_rhs in solve_stream.cu): exactly those whose number the period divides,
for every transform length and every period that a fine tile leaves (64 columns
wide, or 16, at l = 1 to 4).  One test of the thread's index t stands for its
sixteen columns where the period divides L/16; at 128 intervals it does not."""
import pytest


def columns(t, G):
    """Column of register r of thread t (r >= 8: the mirrored half)."""
    return [t + G * r if r < 8 else (16 - r) * G - t for r in range(16)]


@pytest.mark.parametrize("lg", range(8, 15))
@pytest.mark.parametrize("width", [64, 16])
@pytest.mark.parametrize("levels", [1, 2, 3, 4])
def test_planes_are_read_on_the_seams_only(lg, width, levels):
    G, N, px = 2**lg // 16, 2**lg // 2, width >> levels
    max_period = 32
    assert px <= max_period
    seen = set()
    for t in range(G // 2 + 1):
        cx = t & (px - 1) == 0
        for c in columns(t, G):
            if c in (0, N):
                continue
            added = cx and (G >= max_period or c & (px - 1) == 0)
            assert added == (c % px == 0), (t, c)
            if added:
                seen.add(c)
    assert seen == set(range(px, N, px))


def test_one_test_of_t_is_not_enough_at_128_intervals():
    G, px = 16, 32
    assert any(t & (px - 1) == 0 and c % px for t in range(G // 2 + 1) for c in columns(t, G))
