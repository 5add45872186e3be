"""The FP32-core Gram and update kernels of the mixed path (csrc/f32_gemm.cu,
up to 64 states) at the edges of their blocks and tiles, and the first count
beyond them, against the oracle.  Bounds: orthonormalised states 2e-4
relative, subspace energies 1e-5 relative, as in the other mixed tests."""
import numpy as np
import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import report, wells_problem
from itp_workloads import Grid, normal_states
from oracle import itp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,dims", [(1, (4, 2, 2)), (3, (6, 4, 2)), (15, (8, 6, 4)),
                                    (16, (16, 16, 8)), (17, (24, 18, 4)), (32, (32, 16, 6)),
                                    (33, (12, 12, 12)), (48, (16, 8, 24)), (63, (32, 32, 4)),
                                    (64, (32, 24, 8)), (65, (32, 24, 8)), (16, (128, 128, 64))])
def test_block_edges(m, dims):
    g = Grid(*dims, *(0.6 * n for n in dims))
    V = wells_problem(g)
    psi = normal_states(m, g.n_points, 31 + m)
    phi = O.propagate(psi, V, g, 2, 0.02)
    ref, _ = O.cholesky_orthonormalize(phi, g.dV)
    E_ref, _, _ = O.energies(ref, V, g, ritz=True)
    with P.ItpGrid(*dims, g.lx, g.ly, g.lz, m, 0, P.ITP_MIXED) as h:
        h.set_potential(V)
        h.set_states(psi)
        h.propagate(2, 0.02)
        h.orthonormalize()
        got = h.get_states()
        E = h.energies("values")
        Er = h.energies(True)          # rotation by the full matrix
    err = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
    errE = max(np.max(np.abs(e - E_ref)) for e in (E, Er)) / np.max(np.abs(E_ref))
    report(f"FP32 Gram and update m={m} {dims}", err, 2e-4)
    report(f"FP32 subspace energies m={m} {dims}", errE, 1e-5)
    assert err < 2e-4 and errE < 1e-5
