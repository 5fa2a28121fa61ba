"""The fixed-point tables after a change of ln A (csrc/mech_tables.cpp, host code): chem_set_lnA updates what depends
on ln A, with the same result as building every table, and without its cost (a calibration loop calls it in every
iteration).  The update converts R numbers where the build converts R and 40 K and bounds R sums of polynomials:
a tenth of the work for 53 species, asked for here with a factor of two in hand."""
import os
import subprocess

import pytest

from paper_2105_12070_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2105_12070_gb300", "csrc")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fx_tables") / "fx_tables_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "fx_tables_check.cpp"),
                    os.path.join(CSRC, "mech_tables.cpp")], check=True)
    return lambda path: subprocess.run([exe, path], check=True, capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("make", [synth.mechanism_small, synth.mechanism_53, synth.mechanism_100])
def test_update_gives_the_built_tables(check, make):
    out = check(make().write_temp())
    equal, lows, ratio = out[0:14:2], [float(x) for x in out[1:14:2]], float(out[14])
    assert equal == ["1"] * 7
    assert lows[0] == lows[1] == lows[6] > 0.0      # moderate changes keep the interval
    assert lows[2] == lows[3] == lows[4] == 0.0     # these leave none
    assert lows[5] == 512.0                         # and this one a narrower one
    assert ratio > 5.0
