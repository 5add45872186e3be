"""The integer Gram and update kernels of the FP64 path (csrc/fx_gemm.cu)
through the device-block orthonormalisation, at the edges of their state
blocks and point tiles, against the FP64 oracle.  Bound: 1e-11 relative, the
FP64 orthonormalisation bound of the other tests."""
import numpy as np
import pytest
import torch

import paper_0809_3739_gb300 as P
from gpu_helpers import report
from itp_workloads import Grid, normal_states
from oracle import itp_oracle as O

pytestmark = pytest.mark.gpu


def orthonormalise(phi, dV=0.25):
    a = torch.from_numpy(phi).cuda()
    b = torch.empty_like(a)
    P.itp_orthonormalize_noalloc(a.data_ptr(), b.data_ptr(), phi.shape[0], phi.shape[1], dV)
    return b.cpu().numpy()


@pytest.mark.parametrize("m,n", [(1, 1), (1, 4097), (2, 31), (15, 1023), (16, 16), (17, 513),
                                 (32, 4096), (33, 511), (48, 8193), (49, 2000), (64, 64),
                                 (65, 5001), (97, 1025), (128, 333), (128, 20011)])
def test_block_edges(m, n):
    rng = np.random.default_rng(100 * m + n)
    phi = rng.standard_normal((m, n)) + 3 * np.eye(m, n)
    ref, _ = O.cholesky_orthonormalize(phi, 0.25)
    got = orthonormalise(phi)
    err = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
    report(f"integer Gram and update m={m} n={n}", err, 1e-11)
    assert err < 1e-11


@pytest.mark.parametrize("m", [5, 40, 100])
def test_rows_and_points_of_very_different_size(m):
    rng = np.random.default_rng(m)
    n = 6000
    phi = rng.standard_normal((m, n)) * np.exp(-np.linspace(0, 60, n))[rng.permutation(n)]
    size = 10.0 ** rng.uniform(-100, 100, (m, 1))
    ref, _ = O.cholesky_orthonormalize(phi, 0.25)   # L^{-1} D^{-1} D phi: the rows' sizes drop out
    got = orthonormalise(phi * size)
    err = np.max(np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1))
    report(f"rows over 200 orders of magnitude, m={m}", err, 1e-11)
    assert err < 1e-11


def test_more_than_one_block():
    # 200 states: the update of a handle walks 128-row blocks and adds
    g = Grid(16, 16, 16, 8.0, 8.0, 8.0)
    psi = normal_states(200, g.n_points, 11)
    V = np.zeros((16, 16, 16))
    phi = O.propagate(psi, V, g, 2, 0.05)
    ref, _ = O.cholesky_orthonormalize(phi, g.dV)
    with P.ItpGrid(16, 16, 16, 8.0, 8.0, 8.0, 200, 0, P.ITP_FP64) as h:
        h.set_potential(V)
        h.set_states(psi)
        h.propagate(2, 0.05)
        h.orthonormalize()
        got = h.get_states()
    err = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
    report("integer update, 200 states", err, 1e-11)
    assert err < 1e-11
