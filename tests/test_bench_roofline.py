"""bench.py's roofline of an FFT pass: bytes that the pass must move against the
measured HBM bandwidth, in both precisions, so that no pass exceeds one (the
FP64 passes once were held against the FP64 FMA rate, a unit they do not use)."""
import os
import sys
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("kind", ["plane_fwd", "plane_merged", "plane_combine", "plane_hpsi",
                                  "pencil", "pencil_kinetic"])
@pytest.mark.parametrize("s,mixed", [(8, False), (4, True)])
def test_pass_roofline(kind, s, mixed):
    g = types.SimpleNamespace(nx=128, ny=128, nz=128, n_points=128 ** 3)
    m, peak = 128, 6776.3
    spectrum = m * 128 * 128 * 65 * 2 * s      # every pass reads or writes it once
    r = bench.pass_roofline(kind, g, m, s, 5.0, peak, mixed=mixed)
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["peak"] == peak
    assert r["algorithmic_bytes_per_launch"] >= spectrum
    assert r["achieved"] == pytest.approx(r["algorithmic_bytes_per_launch"] / 5e-3 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / peak)
    # a launch as long as its bytes take at the peak is at one, not above
    at_peak = r["algorithmic_bytes_per_launch"] / peak / 1e6
    assert bench.pass_roofline(kind, g, m, s, at_peak, peak, mixed)["frac"] == pytest.approx(1.0)
