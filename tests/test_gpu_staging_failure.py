"""A region whose planes do not arrive in shared memory: the discharge raises
error 2 and leaves the region as it was, active, with no flag of the sweep
before that the fusion would act on.

tests/c/staging_failure.cu builds the discharge kernels with a wait that
reports failure after the copies have landed, and checks the state after one
launch."""
import os
import subprocess

import pytest

from paper_1109_1146_gb300 import build

SRC = os.path.join(build.ROOT, "tests", "c", "staging_failure.cu")


def _compile(out, *defs):
    subprocess.run([build._nvcc()] + build.ARCH + ["-O1", "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I",
                                                   build.CSRC] + list(defs) + [SRC, os.path.join(build.CSRC, "devinfo.cu"),
                                                                               "-o", out],
                   check=True, capture_output=True)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("defs", [(), ("-DVOLUME",)], ids=["2d", "3d"])
def test_region_is_left_as_it_was(tmp_path, defs):
    r = subprocess.run([_compile(str(tmp_path / "staging_failure"), *defs)], capture_output=True, text=True, timeout=60)
    assert (r.returncode, r.stdout) == (0, "ok\n"), r.stdout + r.stderr
