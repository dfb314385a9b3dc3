"""Tiling records that no grid may use are refused on import, as they always were, and leave nothing
behind: a record that was kept would make the contexts of its grid fail (host only, no GPU)."""
import pytest

from paper_2602_07354_gb300 import binding as B


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2602_07354_gb300 import build

    build.build()


@pytest.mark.parametrize("k,line", list(enumerate([
    "1290 1290 1290 4 152 1 1 1",        # 2,146,689,000 tiles: above 2^30
    "1290 1290 1290 8 152 1 1 1",
    "60000 60000 60000 4 152 17 20 1",   # a wide FP32 tile, 6e11 of them
    "48 48 47 4 152 19 19 4",            # 400 columns: wider than any block
])))
def test_unusable_records_are_refused(k, line):
    with pytest.raises(B.ElasError):
        B.elas_tuning_import(f"47 46 {60 + k} 4 152 15 15 8\n{line}\n")
    text = B.elas_tuning_export()
    assert line not in text and f"47 46 {60 + k}" not in text


def test_wide_fp32_records_are_kept():
    line = "47 46 44 4 152 17 20 4"  # 378 columns: a block of an earlier build
    B.elas_tuning_import(line + "\n")
    assert line in B.elas_tuning_export().splitlines()
