"""The autotuner's candidates: only what changes a launch is tried, and an entry without a register cap leaves the plan's."""
import re

import pytest

from paper_1701_06588_gb300 import _lib as L
from paper_1701_06588_gb300 import api, autotune


@pytest.mark.parametrize("ops,precision,caps", [
    (["coulomb"], "fp64", False), (["overlap", "coulomb", "erf", "gauss"], "fp64", False), (["gauss_coulomb"], "mixed", False),
    (["ra2n"], "fp64", False), (["coulomb"], "mixed", True), (["erfc"], "fp64", True), (["overlap", "erfc"], "fp64", True),
    (["coulomb"], "fp64_fused", False), (["coulomb"], "mixed_fused", True), (["overlap", "coulomb"], "fp64_fused", True),
    (["coulomb", "erfc"], "mixed_fused", True)])
def test_variants(ops, precision, caps):
    assert autotune.variants(ops, precision) == ((0, 1, 2) if caps else (None,))


def test_candidates_of_short_lists():
    shapes = autotune.candidates(L.SHG_SHORT_LIST_TILES, ["coulomb"])
    assert [c for c in shapes if c[0] == "persistent"] == [("persistent", 128, 0)]
    assert [c for c in shapes if c[0] == "per_class"] == [c for c in autotune.CANDIDATES if c[0] == "per_class"]
    assert autotune.candidates(L.SHG_SHORT_LIST_TILES + 1, ["coulomb"]) == autotune.CANDIDATES
    assert autotune.candidates(10, ["ra2n"]) == autotune.CANDIDATES


def test_entry_without_a_cap_keeps_the_plans(monkeypatch):
    class Plan:
        handle = 1

    calls = []
    monkeypatch.setattr(api, "Plan2c", lambda *a, **k: Plan())
    monkeypatch.setattr(L, "shg_plan_2c_set_launch", lambda *a: calls.append(a))
    monkeypatch.setattr(L, "shg_plan_2c_set_variant", lambda *a: calls.append(a))
    shape = {"schedule": "persistent", "threads_per_cta": 64, "ctas_per_sm": 2}
    autotune.tuned_plan(None, None, None, shape)
    autotune.tuned_plan(None, None, None, dict(shape, variant=None))
    assert calls == [(1, 64, 2)] * 2
    autotune.tuned_plan(None, None, None, dict(shape, variant=2))
    assert calls[2:] == [(1, 64, 2), (1, 2)]


def test_the_short_list_limit_is_the_headers():
    src = open(re.sub(r"paper_1701_06588_gb300.*", "include/shg.h", L.__file__)).read()
    assert int(re.search(r"#define SHG_SHORT_LIST_TILES (\d+)", src).group(1)) == L.SHG_SHORT_LIST_TILES
