"""The committed captures hold the figures that bench.py reads from them, and
bench.py's source hash covers every source of the kernels it reports on."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1903_06555_gb300", "csrc")


def test_capture_has_every_figure_that_is_read():
    text = open(os.path.join(bench.ROOT, "profiles", "vis_series_kernel_mwa-2048.md")).read()
    figures = dict(re.findall(r"^(\w+): ([0-9.a-f]+)$", text, re.M))
    for key in ("kernel_source_sha256", "lsu_wavefront_pct", "issue_active_pct", "fma_pipe_pct",
                "warp_inst_per_vis", "traffic_bytes_per_launch_degrid",
                "traffic_bytes_per_launch_grid", "traffic_bytes_per_launch_table_degrid",
                "traffic_bytes_per_launch_table_grid"):
        assert key in figures, key
        assert key == "kernel_source_sha256" or float(figures[key]) > 0


def test_source_hash_covers_the_kernels_and_their_launches(monkeypatch):
    """A change to any header that phi_ops.cu includes for the sampled
    quadrature, the transforms or their launches changes the hash."""
    seen = []
    real = open

    def spy(path, *a, **kw):
        seen.append(os.path.basename(str(path)))
        return real(path, *a, **kw)

    monkeypatch.setattr("builtins.open", spy)
    bench.kernel_source_hash()
    for name in ("phi_ops.cu", "phi_internal.cuh", "series_kernel.cuh", "series_launch.cuh",
                 "series_coef.cuh", "fft_kernel.cuh", "fft_launch.cuh", "czt_kernel.cuh",
                 "czt_launch.cuh"):
        assert name in seen, name
