"""bench.py's traffic figures: every kernel of a step has a key, in every size
class, and what the 3D report looks up is what a capture records."""
import os
import sys

import pytest

from conftest import ROOT

HDR = ('"ID","Process ID","Process Name","Host Name","Kernel Name","Context","Stream","Block Size",'
       '"Grid Size","Device","CC","Section Name","Metric Name","Metric Unit","Metric Value"')


def _record(tmp_path, names):
    sys.path.insert(0, ROOT)
    import bench
    rows = ["==PROF== Connected", HDR]
    for i, name in enumerate(names):
        for metric, v in (("dram__bytes_read.sum", 1000 * (i + 1)), ("dram__bytes_write.sum", 1)):
            rows.append(f'"{i}","1","python","h","{name}","1","7","(32, 1, 1)","(9, 1, 1)","0","10.3",'
                        f'"Command line profiler metrics","{metric}","byte","{v}"')
    p = tmp_path / "t.csv"
    p.write_text("\n".join(rows) + "\n")
    return bench, bench.record_traffic(str(p), str(tmp_path / "t.json"), 64, 32)


@pytest.mark.parametrize("name,key", [
    ("void k_sweep_x32h<0, 0>(StepArgs)", "k_sweep_x_fp32"),
    ("void k_sweep_x32<32, 0, 0>(StepArgs)", "k_sweep_x_fp32"),
    ("void k_sweep_yl64<0>(StepArgs)", "k_sweep_y_fp64"),
    ("void k_sweep_y64<8, 0>(StepArgs)", "k_sweep_y_fp64"),
    ("void k_sweep_x64<1, 0>(StepArgs)", "k_sweep_x_fp64")])
def test_every_2d_sweep_has_a_key(tmp_path, name, key):
    bench, out = _record(tmp_path, [name])
    assert out[f"{key}_64x64"]["dram_bytes_per_launch"] == 1001
    assert out[f"{key}_64x64"]["source_digest"] == bench.source_digest()


def test_the_3d_report_finds_what_a_capture_records(tmp_path):
    bench, out = _record(tmp_path, [
        "void pk::k3_sweep_xp<0, 0>(Args3)", "void pk::k3_sweep_vp<0, 0>(Args3)",
        "void k3_source<float>(Args3)", "void k3_sweep64<0>(Args3)", "void k3_source<double>(Args3)"])
    for precision, kernels in bench._KERNELS3.items():
        for k in kernels:
            assert f"{k.split()[0]}_{precision}_32" in out, (k, sorted(out))


def test_the_digest_covers_the_sources_of_the_sweeps():
    sys.path.insert(0, ROOT)
    import bench
    csrc = os.path.join(ROOT, "paper_1311_3004_gb300", "csrc")
    swept = {f for f in os.listdir(csrc) if f.endswith((".cuh", ".cu", ".inc", ".h"))}
    other = {"fvna_net.cu", "fvna_net.h", "fvna_noalloc.cu"}
    assert swept - other == set(bench._SWEEP_SOURCES) | set(bench._SWEEP3_SOURCES)
