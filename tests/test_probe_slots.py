"""The phase probes of the discharge kernels (built with -DMF_DIAG): a slot
holds either times or counts, and every copy of the counters has a reader."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1109_1146_gb300", "csrc")


def _read(path):
    with open(path) as f:
        return f.read()


@pytest.mark.parametrize("name", ["ard_bits2d.cuh", "ard_discharge3d.cu"])
def test_a_slot_holds_times_or_counts(name):
    src = _read(os.path.join(CSRC, name))
    laps, adds = (set(re.findall(rf"{m}\((\d+)", src)) for m in ("DIAG_LAP", "DIAG_ADD"))
    assert laps and adds and not laps & adds
    assert max(map(int, laps | adds)) < 16


def test_every_unit_with_counters_reads_them():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = _read(path)
        if '#include "ard_bits2d.cuh"' in src or "mf_diag3[" in src:
            assert re.search(r"cudaMemcpyFromSymbol\(out, mf::mf_diag", src), path
