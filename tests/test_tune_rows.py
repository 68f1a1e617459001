"""Rows of a guided-filter item in a tile-shape file: 16 to 128, the built-in bound
(host only: needs the compiled library, no GPU)."""
import pytest

import paper_1609_01839_gb300 as gfd


@pytest.mark.parametrize("rows", [16, 32, 64, 128])
def test_accepted(tmp_path, rows):
    path = tmp_path / "t.txt"
    path.write_text(f"class 512 512 col_threads 64 row_threads 64 gf_rows {rows}\n")
    assert gfd.tune_read(str(path)) == (4, {(512, 512): (64, 64, rows)})


@pytest.mark.parametrize("rows", [0, 8, 48, 256])
def test_rejected(tmp_path, rows):
    path = tmp_path / "t.txt"
    path.write_text(f"class 512 512 col_threads 64 row_threads 64 gf_rows {rows}\n")
    with pytest.raises(gfd.GfdError) as e:
        gfd.tune_read(str(path))
    assert e.value.code == -1
