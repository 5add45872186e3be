"""The tensor-core contractions of the mixed path at state counts that run them
in use (more than 64: fewer go to the FP32 cores): the overlap's accuracy over
long sums, and the expiry of their bounded waits."""
import numpy as np
import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import seeded_states, wells_problem
from itp_workloads import Grid, cubic, normal_states
from oracle import itp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [65, 130])
def test_overlap_of_long_chunks(m):
    # 20 CTAs over 128^3 points: each sums 10^5 of them
    g = cubic(128, 32.0)
    with P.ItpGrid(128, 128, 128, 32.0, 32.0, 32.0, m, 0, P.ITP_MIXED) as h:
        t = h.get_tuning()
        h.set_tuning(t["pencil_w"], t["split"], t["row_tb"], 20)
        h.set_potential(np.zeros(g.n_points))
        h.set_states(normal_states(m, g.n_points, seed=99))
        h.propagate(2, 1e-3)
        h.orthonormalize()
        got = h.get_states()
    S = got @ got.T * g.dV
    assert np.max(np.abs(S - np.eye(m))) < 1e-5   # as at 8 states over 256^3


@pytest.mark.parametrize("which", ["overlap", "update", "subspace"])
def test_expired_wait_is_reported_and_the_handle_recovers(which):
    g = Grid(16, 16, 8, 8.0, 8.0, 6.0)
    V = wells_problem(g)
    m = 65
    psi = seeded_states(g, m)
    with P.ItpGrid(g.nx, g.ny, g.nz, g.lx, g.ly, g.lz, m, 0, P.ITP_MIXED) as h:
        h.set_potential(V)
        h.set_states(psi)
        h.propagate(4, 0.2)
        if which != "subspace":
            h.test_expire_waits(1 if which == "overlap" else 2)
            h.orthonormalize()
        else:
            h.orthonormalize()
            h.synchronize()
            h.test_expire_waits(1)
        with pytest.raises(P.ItpError) as ei:
            h.energies("values")
        assert ei.value.code == P.itp.ITP_ERR_TIMEOUT
        h.set_states(psi)
        ref = psi.copy()
        for _ in range(2):
            E = h.step_graph(4, 0.2)
            ref, E_ref = O.itp_step(ref, V, g, 4, 0.2)
            assert np.max(np.abs(E - E_ref)) < 1e-5 * np.max(np.abs(E_ref))
