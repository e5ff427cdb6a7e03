"""The tuner's table and its choice, on the CPU: entries belong to the kernels
they were timed on, and a step replaces another only by the stated margin."""
import argparse
import json

import pytest

torch = pytest.importorskip("torch")

from paper_2206_11524_gb300 import autotune, build


@pytest.fixture
def gpu_name(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda _: "GPU")


def test_an_entry_of_other_kernels_is_not_applied(tmp_path, monkeypatch, gpu_name):
    path = tmp_path / "t.json"
    # as written before entries named their kernels
    path.write_text(json.dumps({"GPU|500x1x1|f32": {"config": [1, 6, 7, 0, 0, 0], "timings_ms": {}}}))
    assert autotune.TuneTable(str(path)).get(500, 1, 1, "f32") is None
    autotune.TuneTable(str(path)).put(500, 1, 1, "f32", (-1, -1, -1, 0, 0, 0), {})
    assert autotune.TuneTable(str(path)).get(500, 1, 1, "f32") == (-1, -1, -1, 0, 0, 0)
    monkeypatch.setattr(autotune, "_kernels", lambda: "other")
    assert autotune.TuneTable(str(path)).get(500, 1, 1, "f32") is None


def test_the_hash_follows_the_code_and_not_its_comments(tmp_path, monkeypatch):
    for f in build.SOURCES + build.HEADERS:
        (tmp_path / f).write_text("int a;  // one\n")
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    first = build.kernel_hash()
    (tmp_path / build.HEADERS[0]).write_text("// more\n\nint a;\n")
    assert build.kernel_hash() == first
    (tmp_path / build.HEADERS[0]).write_text("int b;\n")
    assert build.kernel_hash() != first


def test_each_step_has_to_win_by_the_margin_once():
    wave, single = (0, (2, 4)), (8, (0, 0))
    choose = autotune._choose
    # 288^3: two passes 1718 us, the library's wavefront launch 1646, 4 % less
    assert choose(1718.0, [(wave, 1700.0)], 1646.0, 0.03) == "untuned"
    assert choose(100.0, [], 97.5, 0.03) == "two_pass"
    assert choose(100.0, [(wave, 97.5)], 96.5, 0.03) == "untuned"   # the wavefront fell short
    assert choose(100.0, [(wave, 90.0)], 88.0, 0.03) == wave        # 2 % on the best
    assert choose(100.0, [(wave, 90.0)], 87.0, 0.03) == "untuned"
    assert choose(100.0, [(wave, 90.0), (single, 89.0)], 95.0, 0.03) == single
    assert choose(100.0, [(wave, 98.0), (single, 99.0)], 99.0, 0.03) == "two_pass"


def test_bench_times_the_step_that_runs():
    """Where the tuner leaves the lattice alone the benchmark times lbm_step,
    not the halves of a two-pass step."""
    import bench

    def own(launch, **set_):
        args = {"single_pass": 0, "wavefront": "", "no_wavefront": False} | set_
        return bench._own_choice(launch, argparse.Namespace(**args))
    assert own([-1, -1, -1, 0, 0, 0]) and own(None)
    assert not own([1, 6, 7, 0, 0, 0]) and not own([1, 6, 7])
    assert not own([-1, -1, -1, 0, 0, 0], no_wavefront=True)
    assert not own([-1, -1, -1, 0, 0, 0], wavefront="2,4") and not own(None, single_pass=4)
