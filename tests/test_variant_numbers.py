"""Variant numbers stand in saved tuning tables: a number keeps its shape.  The
small-block shapes are 28 to 37; later shapes come after them."""
import pytest

from paper_0902_4463_gb300 import build, g6gb


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def test_small_block_shapes_keep_their_numbers():
    want = [(16, 16, 1), (32, 8, 1), (64, 4, 1), (128, 2, 1), (256, 1, 1),
            (16, 16, 2), (32, 8, 2), (64, 4, 2), (128, 2, 2), (8, 32, 1)]
    for v, shape in enumerate(want, 28):
        info = g6gb.g6x_variant_info(v)
        assert info["ws"] == 1 and (info["ti"], info["tj"], info["ni_per"]) == shape, v
    assert not any(g6gb.g6x_variant_info(v)["ws"] for v in range(g6gb.g6x_variant_count())
                   if not 28 <= v <= 37)


@pytest.mark.parametrize("prec,bucket,variant", [(0, 4, 28), (0, 4, 33), (0, 5, 34), (0, 3, 37),
                                                 (1, 3, 39), (1, 4, 38), (1, 5, 7)])
def test_a_saved_table_names_the_same_shape(tmp_path, prec, bucket, variant):
    f = tmp_path / "table.txt"
    f.write_text(f"{prec} {bucket} {variant} 1\n")
    try:
        assert g6gb.g6x_load_tuning(str(f)) == 1
        assert g6gb.g6x_plan_launch(prec, 1 << 20, 1 << bucket)["variant"] == variant
    finally:
        g6gb.g6x_clear_tuning()
