"""The discharge kernels that the benchmark's roofline lines name, against the
launches in the sources."""
import os
import re

import pytest

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


@pytest.mark.parametrize("kernel,body", [("ard_discharge2d_kernel<8,32,32,256>", "discharge2d_region"),
                                         ("ard_discharge3d_batch_kernel<8,4,256>", "discharge3d_region")])
def test_the_hashed_file_holds_the_kernel_body(kernel, body):
    src = _read(bench.kernel_source(kernel))
    assert re.search(rf"__device__ __forceinline__ void {body}\([^;{{]*\{{", src)


def test_a_figure_recorded_against_another_file_is_not_reported(tmp_path, monkeypatch):
    # the file is unchanged since, but it does not hold the kernel's body
    import hashlib
    kernel, tile = bench.kernel_name(8, (32, 32, 1)), (32, 32, 1)

    def record(source):
        with open(os.path.join(CSRC, source), "rb") as f:
            sha = hashlib.sha256(f.read()).hexdigest()[:16]
        (tmp_path / "profiles" / "a.txt").write_text(
            f"bench: kernel={kernel}\nbench: source={source}\nbench: kernel_sha256_16={sha}\nbench: tile=32x32x1\n"
            "bench: dram_bytes_per_discharged_vertex=70.5\n")

    (tmp_path / "profiles").mkdir()
    os.symlink(os.path.join(ROOT, "paper_1109_1146_gb300"), tmp_path / "paper_1109_1146_gb300")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    record("ard_discharge2d.cu")
    assert bench.committed_traffic(kernel, tile) is None
    record("ard_bits2d.cuh")
    assert bench.committed_traffic(kernel, tile) == 70.5
