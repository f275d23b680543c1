"""Checkpoint files of earlier builds, which hold the same particle state behind
shorter instance records (624 and 688 bytes): the eight particles of
test_degenerate.sparse_instance after four steps, saved by those builds."""
import os

import numpy as np
import pytest

from paper_2405_03980_gb300 import _binding as B
from test_degenerate import _max_rel, sparse_instance
from test_gpu_fp64 import _cuda, sim_of  # noqa: F401

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


@pytest.mark.parametrize("record", [624, 688])
@pytest.mark.parametrize("form,tol", [("fp64", 1e-12), ("mixed", 64 * 2.0**-24)])
def test_files_of_earlier_builds_resume(record, form, tol):
    """Three steps on from the file give the fields of seven steps in one run, to
    the rounding of the passes; a file of other constants, or one cut short, is
    refused and changes nothing."""
    path = os.path.join(GOLDEN, f"checkpoint_{record}_{form}.bin")
    c = sparse_instance()
    prec = B.SPH_FP64 if form == "fp64" else B.SPH_MIXED
    sim = sim_of(c, precision=prec, nbr_cap=64)
    before = sim.state_arrays()["pos"]
    ck = np.fromfile(path, dtype=np.uint8)
    bad = ck.copy()
    bad[80 + 13 * 8] ^= 1  # B of the first record (the header has 80 bytes)
    for broken in (bad, ck[:-8], ck[:40]):
        with pytest.raises(B.SphError):
            sim.load_checkpoint(broken)
    assert np.array_equal(sim.state_arrays()["pos"], before)
    sim.load_checkpoint(path)
    sim.step(3)
    one = sim_of(c, precision=prec, nbr_cap=64)
    one.step(7)
    st, ref = sim.state_arrays(), one.state_arrays()
    for k in ("pos", "vel", "spin", "rho", "P", "acc", "dspin"):
        assert _max_rel(st[k], ref[k]) <= tol, k
    assert sim.diagnostics()["step"] == 7
    sim.close()
    one.close()
