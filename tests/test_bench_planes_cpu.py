"""bench.py's byte models count the w-planes of the grid that the transforms run on, and
the interpolation where that is not the image's own."""
import types

import pytest

import bench


def test_bytes_of_a_smaller_grid():
    wl = types.SimpleNamespace(M=1000, N=400)
    own = {"grid_side": 1024, "n_planes": 9, "kernel_width": 7}
    small = dict(own, transform_grid=512, transform_image=256)
    reach = {"rows": 96, "col_groups": 4}
    peaks = {"hbm_gbs": 1.0}
    prof = {k: (1, 1, 1.0) for k in ("grid", "fft_rows", "fft_cols", "degrid_fft")}

    def got(info, dom):
        return bench.roofline(prof, info, wl, [], 1, peaks, dom, reach)["achieved"] * 1e6     # bytes in 1 ms

    inter = 4.0 * (400 ** 2 + 256 ** 2 + 2 * 400 * 256)
    cells = 96 * 32.0 * 4
    for info, n, extra in ((own, 400, 0.0), (small, 256, inter)):
        assert got(info, "fft_rows") == pytest.approx(8.0 * 9 * (cells + n * 96))
        assert got(info, "fft_cols") == pytest.approx(8.0 * 9 * n * 96 + 20.0 * n * n + extra)
        assert got(info, "degrid_fft") == pytest.approx(4.0 * n * n + 8.0 * 9 * (cells + 2 * n * 96) + extra)
    r = bench.gridding_roofline(prof, small, wl, peaks)
    assert r["bytes_full_planes"] == 20.0 * 1000 + 8.0 * 9 * 512 ** 2 == r["bytes_per_launch"]
