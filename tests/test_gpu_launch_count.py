"""itp_kernel_launches above 128 states, where one update or overlap is several
kernels: the count of a per-problem batch graph (added up by the library's
calls) is the number of kernel nodes that the grouped graph of the same one
problem has."""
import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import seeded_states, wells_problem
from itp_workloads import Grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [P.ITP_FP64, P.ITP_MIXED])
@pytest.mark.parametrize("m", [20, 64, 128, 129, 256])
def test_launches_are_kernel_nodes(m, prec):
    g = Grid(16, 16, 8, 8.0, 8.0, 4.0)
    n = []
    for grouped in (True, False):
        with P.ItpBatch([(16, 16, 8)], [(8.0, 8.0, 4.0)], [m], precision=prec) as b:
            b.set_grouping(grouped)
            b[0].set_potential(wells_problem(g))
            b[0].set_states(seeded_states(g, m))
            b.step(4, 0.05)
            n.append(b.kernel_launches)
    assert n[0] == n[1]
