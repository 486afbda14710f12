"""The calibration of the present kernels (theta_gb300_rev2*.json) against its table
and report, and the statement in the earlier parameter files (CPU only)."""
import json
import os

import numpy as np
import pytest

import oracle as O
from test_calibration_data import _mae_by_family, _theta

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_04178_gb300")


def load(name):
    with open(os.path.join(PKG, name)) as f:
        return json.load(f)


@pytest.fixture(params=[O.READING_LITERAL, O.READING_MEASURED], ids=["literal", "measured"])
def reading(request):
    prev = O.reading()
    O.set_reading(request.param)
    yield request.param
    O.set_reading(prev)


def test_parameters_fit_their_table(reading):
    suffix = "" if reading == O.READING_MEASURED else "_literal"
    meta = load("theta_gb300_rev2%s.json" % suffix)
    assert meta["reading"] == reading and meta["fitted_on"] == "sweep_gb300_rev2.json"
    th = np.array(meta["theta"], dtype=np.float64)
    assert th.size == O.N_PARAMS
    table = load("data/sweep_gb300_rev2.json")
    got = _mae_by_family(table, th)
    if reading == O.READING_MEASURED:
        report = load("data/calib_report_gb300_rev2.json")
        assert np.allclose(report["theta"], th, rtol=1e-12, atol=0)
        for fam, v in report["mae_all"].items():
            assert got[fam] == pytest.approx(v["mae_pct"], abs=0.05), fam
    # the earlier parameters miss this table by what their files say
    old = _mae_by_family(table, _theta(reading))["all"]
    assert "(mean error %.1f %%)" % old in load("theta_gb300%s.json" % suffix)["kernels"]
    assert got["all"] < 0.5 * old
