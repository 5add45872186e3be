"""The autotuner times the overlap with the CTA counts that a step would launch:
in FP64 with more than 32 states both candidates may lead to one count, which
is then timed once."""
import re

import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import seeded_states, wells_problem
from itp_workloads import Grid

pytestmark = pytest.mark.gpu


# 5184 points are too few for two CTAs per SM of the tensor-core form; at 96^3
# a chunk of 304 has more than four runs of 512 points
@pytest.mark.parametrize("dims,m,prec,counts", [
    ((24, 18, 12), 10, P.ITP_FP64, 2), ((24, 18, 12), 40, P.ITP_FP64, 1),
    ((96, 96, 96), 40, P.ITP_FP64, 2), ((24, 18, 12), 40, P.ITP_MIXED, 2)])
def test_overlap_candidates(dims, m, prec, counts):
    g = Grid(*dims, *(0.5 * n for n in dims))
    with P.ItpGrid(*dims, g.lx, g.ly, g.lz, m, 0, prec) as h:
        h.set_potential(wells_problem(g))
        h.set_states(seeded_states(g, m))
        report = h.autotune(4, 0.1)[1]
        timed = [int(c) for c in re.findall(r" (\d+)=", report.split("gram:")[1])]
        assert len(timed) == counts and len(set(timed)) == counts, report
        assert h.get_tuning()["gram_ctas"] in timed
