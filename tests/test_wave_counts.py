"""Waves of CTAs in the built-in launch choice: a longer work line never gets
fewer of them, and each step lies where the rule says.  The count itself is
read off the plan: its grid over the grid of the same shape with the
multiplier 1 from a tuning table, so the resident CTAs per SM of whatever
device is there (none on a host without one) cancel."""
import pytest

from paper_0902_4463_gb300 import build, g6gb

BIG = 1 << 20
DS = g6gb.G6X_PREC_DS


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    g6gb.g6x_clear_tuning()
    yield
    g6gb.g6x_clear_tuning()


def _waves(tmp_path, nj, ni):
    p = g6gb.g6x_plan_launch(DS, nj, ni)
    f = tmp_path / "one.txt"
    f.write_text(f"{DS} {ni.bit_length() - 1} {p['variant']} 1\n")
    try:
        g6gb.g6x_load_tuning(str(f))
        one = g6gb.g6x_plan_launch(DS, nj, ni)
    finally:
        g6gb.g6x_clear_tuning()
    assert one["variant"] == p["variant"] and p["grid"] % one["grid"] == 0
    return p["variant"], p["grid"] // one["grid"]


# N = 2^20: 4096 j-tiles, so i-tiles x 4096 units
@pytest.mark.parametrize("variant,itile,steps", [
    (9, 256, ((16, 1), (31, 1), (32, 2), (511, 2), (512, 4), (2047, 4), (2048, 8), (4096, 8))),
    (16, 128, ((2, 1), (3, 1), (4, 2), (15, 2), (16, 4))),
])
def test_steps_lie_at_their_lengths(tmp_path, variant, itile, steps):
    for tiles, want in steps:
        for ni in (tiles * itile, (tiles - 1) * itile + 1):
            if variant == 9 and ni <= 2048 or variant == 16 and not 128 < ni <= 2048:
                continue
            assert _waves(tmp_path, BIG, ni) == (variant, want), (tiles, ni)


@pytest.mark.parametrize("nj", [131072, 262144, 1000003, BIG])
def test_a_longer_line_never_gets_fewer_waves(tmp_path, nj):
    last = {}
    ni = 129
    while ni <= nj:
        v, w = _waves(tmp_path, nj, ni)
        assert w >= last.get(v, 1), (nj, ni, v, w, last)
        last[v] = w
        ni += max(1, ni // 9)
