"""Grouped batches whose passes, with the terms of the expansion together,
have more rows (states x terms) than one launch takes (65535): up to 65535
states form a group, whatever the order, and the results are those of the
per-problem graph, bit for bit."""
import numpy as np
import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import wells_problem
from itp_workloads import Grid, normal_states

pytestmark = pytest.mark.gpu

G = Grid(16, 16, 4, 9.6, 9.6, 2.4)


def batch(total, prec):
    """Problems of up to 256 states, `total` in all."""
    counts = [256] * (total // 256) + ([total % 256] if total % 256 else [])
    b = P.ItpBatch([(G.nx, G.ny, G.nz)] * len(counts), [(G.lx, G.ly, G.lz)] * len(counts), counts,
                   precision=prec)
    V = wells_problem(G)
    for q in b.problems:
        q.set_potential(V)
    return b, counts


def load(b, counts, psi):
    for p, (q, n) in enumerate(zip(b.problems, counts)):
        q.set_states(np.roll(psi[:n], p, axis=1))


# at order 12 (six terms) 10922 states are 65532 rows, 10923 are 65538
@pytest.mark.parametrize("prec", [P.ITP_MIXED, P.ITP_FP64])
@pytest.mark.parametrize("total", [10922, 10923])
def test_more_rows_than_one_launch_takes(total, prec):
    psi = normal_states(256, G.n_points, 5)
    b, counts = batch(total, prec)
    with b:
        load(b, counts, psi)
        E = b.step(12, 0.05)
        assert b.groups == 1
        got = [b[p].get_states() for p in (0, len(counts) - 2, len(counts) - 1)]
        b.set_grouping(False)
        load(b, counts, psi)
        Eref = b.step(12, 0.05)
        for p, (e, r) in enumerate(zip(E, Eref)):
            assert np.array_equal(e, r), p
        for p, s in zip((0, len(counts) - 2, len(counts) - 1), got):
            assert np.array_equal(s, b[p].get_states()), p


def test_more_states_than_a_group_takes():
    psi = normal_states(256, G.n_points, 5)
    b, counts = batch(65536, P.ITP_MIXED)
    with b:
        load(b, counts, psi)
        with pytest.raises(P.ItpError) as e:
            b.step(2, 0.05)
        assert e.value.code == P.itp.ITP_ERR_ARG and "more than 65535 states" in str(e.value)
