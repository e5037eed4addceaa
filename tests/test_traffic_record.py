"""The recorded DRAM traffic of the pass kernels is dropped when any file they are
compiled from changes."""
import json
import os

import bench


def test_every_source_file_counts(tmp_path, monkeypatch):
    names = {os.path.basename(p) for p in bench.KERNEL_SRC}
    csrc = os.path.dirname(bench.KERNEL_SRC[0])
    # pdot_kernels.cu and what it includes, without the resident kernel (no plan pass)
    included = {line.split('"')[1] for line in open(os.path.join(csrc, "pdot_kernels.cu")) if line.startswith('#include "')}
    assert names == {"pdot_kernels.cu"} | included - {"pdot_resident.cuh"}
    copies = []
    for p in bench.KERNEL_SRC:
        copies.append(str(tmp_path / os.path.basename(p)))
        with open(copies[-1], "wb") as fh:
            fh.write(open(p, "rb").read())
    monkeypatch.setattr(bench, "KERNEL_SRC", copies)
    rec = {"cost_dtype": "f32", "grid": 64, "kernel_variant": 2, "dram_bytes_per_launch_full_size": 5.0,
           "kernel_source_sha256": bench.kernel_source_sha256()}
    traffic = tmp_path / "traffic.json"
    traffic.write_text(json.dumps({"records": [rec]}))
    monkeypatch.setattr(bench, "TRAFFIC", str(traffic))
    assert bench.recorded_traffic("f32", 64, 2) == 5.0
    for p in copies:
        before = open(p, "rb").read()
        with open(p, "ab") as fh:
            fh.write(b"// changed\n")
        assert bench.recorded_traffic("f32", 64, 2) is None, p
        with open(p, "wb") as fh:
            fh.write(before)
    assert bench.recorded_traffic("f32", 64, 2) == 5.0
