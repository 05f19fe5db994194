"""The sort's count arrays are taken for zero only when the launch that clears them went out: between
the launch that counts and that one every early return leaves them marked as not clean."""
import pathlib

SORT = pathlib.Path(__file__).resolve().parents[1] / "paper_2606_01598_gb300" / "csrc" / "sort.cu"


def test_counts_are_marked_until_cleared():
    text = SORT.read_text()
    body = text[text.index("int launch_sort_t("):]
    body = body[:body.index("\n}\n")]
    dirty, clean = body.index("p->counts_clean = false"), body.index("p->counts_clean = true")
    assert dirty < body.index("pdl_launch(k_bin<BATCH>")
    assert body.index('check_launch(p, "k_scatter")') < clean
    assert body.count("p->counts_clean = ") == 2
