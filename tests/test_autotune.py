"""The autotuner's candidates (host only): none twice, in the fields that apply to
its shape, and each once."""
from paper_1411_0127_gb300 import autotune


def test_candidates_differ_in_fields_that_apply():
    cands = autotune.candidates()
    assert cands[0] == (0, 32, 1, 1)                  # the library's default
    applies = [c if 1 <= c[0] <= 3 else (c[0], c[3]) for c in cands]
    assert len(set(applies)) == len(cands)
    assert {c[0] for c in cands} == {0, 1, 2, 3, 4, 5} and {c[3] for c in cands} == {1, 2}
