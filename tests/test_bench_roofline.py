"""bench.py's roofline model: the bytes, sweeps, sources and texts of the launch that runs the sweeps, for
every form that a handle reports.  A launch is charged one pass over the state, whatever the sweeps it
carries, so no form can exceed the bandwidth."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("fform,fused,kind,fp16,form,sweeps,nbytes,sources", [
    (0, 1, 2, False, "single", 1, 72, "single"),
    (1, 4, 1, False, "stages", 4, 72, "stages"),
    (2, 2, 1, False, "staged_rows", 2, 72, "two_sweep"),
    (3, 2, 1, False, "direct", 2, 72, "two_sweep"),
    (4, 4, 1, False, "quad", 4, 72, "four_sweep"),
    (5, 4, 2, False, "resident", None, 72, "resident"),
    (5, 1, 2, False, "resident", None, 72, "resident"),
    (0, 1, 3, True, "single", 1, 44, "single_fp16"),
    (4, 4, 3, True, "quad", 4, 44, "four_sweep_fp16"),
])
def test_launch_of_each_form(fform, fused, kind, fp16, form, sweeps, nbytes, sources):
    lc = bench.sweep_launch(fform, fused, kind, fp16)
    assert (lc["form"], lc["sweeps"], lc["bytes_per_node"], lc["sources"]) == (form, sweeps, nbytes, sources)
    assert lc["sources"] in bench.KERNEL_SOURCES
    assert lc["bound"] == ("hbm" if sweeps else "cluster barriers")
    assert ("FP16" in lc["text"]) == fp16
    if sweeps is None:
        assert "whole solve" in lc["text"] and "sweeps per launch" not in lc["text"]
    elif sweeps > 1:
        assert lc["text"].endswith(bench.FUSED_FORM_TEXT[fform]) and f"{sweeps} sweeps per launch" in lc["text"]
    else:
        assert lc["text"].endswith(bench.SWEEP_KERNEL_NAMES[kind])
    assert lc["bytes_model"].startswith(f"{nbytes} B per node and ")


def test_measured_launches_stay_below_the_bandwidth():
    """4096^2, four sweeps in 219 us, and FP16 at 2048^2, four in 78 us: 0.8 and 0.35 of 6790.7 GB/s."""
    quad, half = bench.sweep_launch(4, 4, 1, False), bench.sweep_launch(4, 4, 3, True)
    assert quad["bytes_per_node"] * 4096 ** 2 / 219e-6 / 6790.7e9 == pytest.approx(0.812, abs=0.001)
    assert half["bytes_per_node"] * 2048 ** 2 / 78e-6 / 6790.7e9 == pytest.approx(0.348, abs=0.001)


@pytest.mark.parametrize("n,every,sweeps", [(128, 8, 4), (1024, 16, 4), (512, 4, 2), (1024, 12, 2), (256, 4, 1),
                                            (512, 6, 1)])
def test_sweeps_of_a_batched_launch(n, every, sweeps):
    assert bench.batch_sweeps_per_launch(n, n, every) == sweeps


@pytest.mark.parametrize("form,needs", [
    ("single", {"kernels.cu", "sweep_rows.cu", "lbm2p_async.cuh", "residual.cuh"}),
    ("stages", {"kernels.cu", "residual.cuh", "step_node.cuh"}),
    ("two_sweep", {"sweep_rows.cu", "lbm2p_async.cuh"}),
    ("four_sweep", {"sweep_quad.cu", "sweep_quad.cuh", "lbm2p_async.cuh"}),
    ("resident", {"resident.cu", "residual.cuh", "lbm2p_async.cuh"}),
    ("single_fp16", {"fp16.cu", "lbm2p_async.cuh"}),
    ("four_sweep_fp16", {"fp16_quad.cu", "sweep_quad.cuh", "lbm2p_async.cuh"}),
])
def test_source_hash_covers_every_header_that_the_kernels_compile_from(form, needs, monkeypatch):
    """Every file is hashed: an edit of any of them changes the hash that keys a capture."""
    import builtins
    files = bench.kernel_source_files(form)
    assert needs | {"lbm2p_node.cuh", "lbm2p_device.cuh"} <= set(files) and len(files) == len(set(files))
    before = bench.kernel_source_hash(form)
    real = builtins.open
    for edited in files:
        class Edited:
            def __init__(self, f):
                self.f = f

            def __enter__(self):
                return self

            def __exit__(self, *exc):
                self.f.close()

            def read(self):
                return self.f.read() + b" "

        def fake(path, mode="r", *a, **k):
            f = real(path, mode, *a, **k)
            return Edited(f) if "b" in mode and str(path).endswith(os.sep + edited) else f

        monkeypatch.setattr(builtins, "open", fake)
        assert bench.kernel_source_hash(form) != before, edited
        monkeypatch.setattr(builtins, "open", real)
    assert bench.kernel_source_hash(form) == before
