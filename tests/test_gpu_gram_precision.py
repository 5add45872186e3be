"""Precision of the FP64 overlap (csrc/fx_gemm.cu) on its diagonal, the squared
norms, through the device-block orthonormalisation of rows that do not
overlap (each on points of its own, so L^{-1} is diagonal and |psi_i|^2 dV
is 1 up to the relative error of S_ii).

Bound, worst case, in units of u = 2^-53: the kernel's sum over a run 1,
its conversion to FP64 3, runs added within a chunk and chunks within a slot
of the reduction at most 8, slots and scale 3; then 1 / sqrt(S_ii) 1 + 2, and
the roundings of the scaled values, which average out: together 18 u.  The
roundings of a row are independent of the other rows' and of no preferred
sign, so the mean over 32 rows stays within three standard deviations,
3 * 18 u / sqrt(3 * 32).

A squared norm without the products of the elements' lower halves is too
small by up to 350 u for these rows, in every row."""
import numpy as np
import pytest
import torch

import paper_0809_3739_gb300 as P
from gpu_helpers import EPS64, report

pytestmark = pytest.mark.gpu

RUN = 512   # points that the kernel scales together


def rows(shape, m, per, rng):
    """m rows of `per` points each."""
    a = rng.standard_normal((m, per))
    p = np.arange(per)
    if shape == "one large value per run":
        a *= 1e-5
        a[:, 7::RUN] = 1.0 + rng.random((m, len(range(7, per, RUN))))
    elif shape == "one large value":
        a *= 1e-4
        a[:, per // 2] = 1.0
    elif shape == "decay in each run":
        a *= np.exp(-(p % RUN) / 30.0)
    elif shape == "smooth":
        a = np.exp(-((p - per / 2) / (per / 6.0)) ** 2) * (1.0 + 0.1 * rng.random((m, 1)))
    return a


@pytest.mark.parametrize("m", [1, 16, 32])
@pytest.mark.parametrize("shape", ["normal", "smooth", "decay in each run",
                                   "one large value per run", "one large value"])
def test_squared_norms(m, shape):
    per = 16 * RUN
    rng = np.random.default_rng(1000 * m + len(shape))
    phi = np.zeros((m, m * per))
    a = rows(shape, m, per, rng)
    for i in range(m):
        phi[i, i * per:(i + 1) * per] = a[i]
    dV = 0.25
    d = torch.from_numpy(phi).cuda()
    out = torch.empty_like(d)
    P.itp_orthonormalize_noalloc(d.data_ptr(), out.data_ptr(), m, m * per, dV)
    psi = out.cpu().numpy()
    norms = np.array([(psi[i, i * per:(i + 1) * per].astype(np.longdouble) ** 2).sum() * dV
                      for i in range(m)])
    err = (norms - 1).astype(float)
    tol, tol_mean = 18 * EPS64, 3 * 18 * EPS64 / np.sqrt(3 * 32)
    report(f"squared norms, {shape}, m={m}", np.max(np.abs(err)), tol)
    report(f"squared norms, {shape}, m={m}, mean", abs(err.mean()), tol_mean)
    assert np.max(np.abs(err)) < tol, err
    if m >= 32:
        assert abs(err.mean()) < tol_mean, err
