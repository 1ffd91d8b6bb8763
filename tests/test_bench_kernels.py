"""Host checks of the kernels bench.py reports as launched, and of the keys it
finds their recorded traffic under."""

import json

import bench

from test_bench_names import small


def test_launched_kernels_are_the_librarys():
    ctu64 = small("rt256-fp64-ctu")
    # as the profiler lists them on the GPU
    assert bench.launched_kernels(ctu64, 0) == ["ctu3d_kernel<double, 0, 16, 8, 1>"]
    assert bench.launched_kernels(ctu64.replace(grav=(0.1, 0.0, -1.0)), 0) == ["ctu3d_kernel<double, 0, 16, 8, 0>"]
    assert bench.launched_kernels(small("rt512-fp32-ctu"), 0) == ["ctu3d_kernel<float, 1, 16, 16, 0>"]
    # FP64: variants v and v + 4 are one kernel
    assert bench.launched_kernels(small("rt256-fp64"), 6) == ["step3d_kernel<double, 0, 16, 16, 0, 0, 0, 1>"]
    assert bench.launched_kernels(small("rt512-fp32"), 7) == ["step3d_kernel<float, 1, 32, 16, 0, 0, 1, 0>"]


def test_traffic_is_recorded_and_found_by_the_launched_name(tmp_path, monkeypatch, capsys):
    name = bench.launched_kernels(small("rt256-fp64-ctu"), 0)[0]
    csv = tmp_path / "t.csv"
    csv.write_text('"ID","Kernel Name","Metric Name","Metric Value"\n' + "".join(
        f'"0","void {name}(StepArgs)","{m}","{v}"\n' for m, v in
        (("gpu__time_duration.sum", 5), ("dram__bytes_read.sum", 100), ("dram__bytes_write.sum", 20))))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_source_sha", lambda kernel="": "sha")
    (tmp_path / "profiles").mkdir()
    assert bench.record_traffic("rt256-fp64-ctu", str(csv)) == 0
    table = json.loads((tmp_path / "profiles" / "traffic.json").read_text())
    assert list(table["rt256-fp64-ctu"]) == bench.step_kernel_names(small("rt256-fp64-ctu"), 0)
    assert bench.measured_traffic("rt256-fp64-ctu", name) == 120.0
