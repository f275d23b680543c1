"""Checkpoint files of earlier builds, which hold the same particle state behind
shorter instance records (624 and 688 bytes): the eight particles of
test_degenerate.sparse_instance after four steps, saved by those builds, and
files of several instances put together from present ones."""
import os

import numpy as np
import pytest

from paper_2405_03980_gb300 import _binding as B
from test_degenerate import _max_rel, single_instance, sparse_instance
from test_gpu_fp64 import _cuda, sim_of  # noqa: F401

pytestmark = pytest.mark.gpu
HEADER = 72
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
    bad[HEADER + 14 * 8] ^= 1  # B of the first record
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


@pytest.mark.parametrize("record", [624, 688])
@pytest.mark.parametrize("precision", [B.SPH_FP64, B.SPH_MIXED])
def test_batches_behind_shorter_records(record, precision):
    """The particle state stands behind all records, at a multiple of 256 bytes:
    a present file of three instances with its records cut down to the earlier
    ones (and their chunk counts changed, which no state depends on) resumes bit
    for bit."""
    batch = [sparse_instance(), single_instance(), sparse_instance()]
    a = sim_of(batch, precision=precision, nbr_cap=64)
    a.step(3)
    ck = a.save_checkpoint()
    a.step(2)
    state_bytes, inst_bytes = (int(x) for x in ck[32:48].view(np.uint64))
    size, up = inst_bytes // 3, lambda b: (b + 255) // 256 * 256
    recs = ck[HEADER:HEADER + inst_bytes].reshape(3, size).copy()
    recs[:, 424:440] = 7  # the first chunk and their number
    keep = [slice(0, 688)] if record == 688 else [slice(0, 280), slice(336, 440), slice(448, 688)]
    old = np.concatenate([recs[:, k] for k in keep], axis=1).ravel()
    assert old.size == 3 * record
    body = ck[HEADER + up(inst_bytes):HEADER + state_bytes]
    head = ck[:HEADER].copy()
    head[32:48] = np.array([up(old.size) + body.size, old.size], dtype=np.uint64).view(np.uint8)
    file = np.concatenate([head, old, np.zeros(up(old.size) - old.size, np.uint8), body])
    b = sim_of(batch, precision=precision, nbr_cap=64)
    b.load_checkpoint(file)
    b.step(2)
    x, y = a.state_arrays(), b.state_arrays()
    for k in x:
        assert np.array_equal(x[k], y[k]), k
    assert [b.diagnostics(k)["step"] for k in range(3)] == [5, 5, 5]
    a.close()
    b.close()
