"""The x drift with the fused density is told from the other drifts of the same
kernel by its name in an ncu launch list, however ncu prints truth values."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("args,want", [
    ("48, 1, 0, 0", False), ("48, 1, 0, 1", True), ("64, 1, 1, 1", True), ("64, 0, 1, 0", False),
    ("(int)48, (bool)1, (bool)0, (bool)1", True), ("(int)48, (bool)1, (bool)1, (bool)0", False),
    ("48, true, false, true", True), ("48, true, true, false", False)])
def test_density_flag_of_the_drift(args, want):
    for name in (f"k_drift_fast<{args}>(const float *, const LineCoef<float> *, DriftGeom, double *)",
                 f"void <unnamed>::k_drift_fast<{args}>(...)", f"k_drift_fast<{args}>"):
        assert bench._drift_with_density(name) is want


def test_an_unknown_form_is_refused():
    with pytest.raises(ValueError):
        bench._drift_with_density("k_drift_fast<48, 1, 0, RHO>(...)")
