"""The autotuner times the library's default among the other tiles, records it unless another tile is clearly
faster, and the committed records are of such runs."""
import json

import pytest

from paper_1903_12522_gb300 import autotune


@pytest.mark.parametrize("dim", [2, 3])
def test_the_default_is_a_candidate(dim):
    cands = autotune.candidates(dim)
    assert cands[0] == (0, 0, 0, 0) and len(set(cands)) == len(cands)
    assert set(autotune.candidates_3d() if dim == 3 else autotune.candidates_2d()) < set(cands)


def test_choice():
    d, a, b = autotune.DEFAULT, (0, 0, 0, 5), (16, 0, 0, 3)
    assert autotune.choose({d: 1.0, a: 0.99, b: 1.2}) == d
    assert autotune.choose({d: 1.0, a: 0.9, b: 0.95}) == a
    assert autotune.choose({d: 1.0, a: 1.1}) == d


def test_committed_records_are_of_all_candidates():
    for key, entry in json.load(open(autotune.CACHE)).items():
        if key.startswith("d"):
            cands = autotune.candidates(int(key[1]))
            assert entry["candidates"] == len(cands) and tuple(entry["tile"]) in cands, key
            assert entry["ms_per_adjoint_period"] <= entry["worst_ms"], key
