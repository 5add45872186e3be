"""Steps that run the terms of the expansion together, one launch per pass
over all of them (small problems), against the same calls made one by one,
which run term by term: the same states and energies bit for bit, fewer
launches; and a step between host buffers, whose chunks hold fewer states."""
import numpy as np
import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import seeded_states, wells_problem
from itp_workloads import Grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [P.ITP_FP64, P.ITP_MIXED])
@pytest.mark.parametrize("order", [2, 4, 12])
@pytest.mark.parametrize("dims,m", [((24, 18, 12), 5), ((32, 32, 32), 1), ((16, 8, 128), 3),
                                    ((64, 48, 1), 7), ((256, 256, 1), 3), ((192, 256, 4), 2)])
def test_step_equals_its_parts(prec, order, dims, m):
    g = Grid(*dims, *(0.5 * n if n > 1 else 1.0 for n in dims))
    V = wells_problem(g)
    psi = seeded_states(g, m)
    tau = 0.1
    with P.ItpGrid(*dims, g.lx, g.ly, g.lz, m, 0, prec) as h:
        h.set_potential(V)
        if dims[2] == 128 and prec == P.ITP_MIXED:   # the column-per-thread pencil
            t = h.get_tuning()
            h.set_tuning(0, t["split"], t["row_tb"], t["gram_ctas"])
        h.set_states(psi)
        h.propagate(order, tau)
        n0 = h.kernel_launches
        h.propagate(order, tau)
        alone = h.kernel_launches - n0
        h.orthonormalize()
        E = h.energies("values")
        ref = h.get_states()
        h.set_states(psi)
        h.step_graph(order, tau)   # captures
        h.set_states(psi)
        n0 = h.kernel_launches
        Es = h.step_graph(order, tau)
        step = h.kernel_launches - n0
        assert np.array_equal(E, Es)
        assert np.array_equal(ref, h.get_states())
        out, Eh = h.step_host(order, tau, psi)
        assert np.array_equal(E, Eh) and np.array_equal(ref, out)
        if order == 12:   # 48 passes in 14 (mixed), 18 (FP64) launches
            assert step < alone
