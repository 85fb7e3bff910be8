"""The discharge kernels that the benchmark's roofline lines name, against the
launches in the sources."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1109_1146_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _launched():
    """(conn, tile, batch) -> the kernels launched for it, template arguments up to the threads per block"""
    out = {}
    for b, args in re.findall(r"launch2d(_batch)?<(\d+, \d+, \d+, \d+)>\(", _read("ard_discharge2d.cu")):
        conn, tx, ty, nt = args.split(", ")
        out.setdefault((int(conn), (int(tx), int(ty), 1), bool(b)), set()).add(
            f"ard_discharge2d{b}_kernel<{conn},{tx},{ty},{nt}>")
    for b, args in re.findall(r"launch3d(_batch)?<(\d+, \d+, \d+, \d+)>\(", _read("ard_discharge3d.cu")):
        ty, tz, nt, _ = args.split(", ")
        out.setdefault((6, (32, int(ty), int(tz)), bool(b)), set()).add(f"ard_discharge3d{b}_kernel<{ty},{tz},{nt}>")
    return out


def test_names_are_those_of_the_launched_kernels():
    launched = _launched()
    assert len(launched) == 2 * (2 * 4 + 5)  # single and batched: four 2D tiles at two connectivities, five 3D tiles
    for (conn, tile, batch), names in launched.items():
        assert names == {bench.kernel_name(conn, tile, batch)}
