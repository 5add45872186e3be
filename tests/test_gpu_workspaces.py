"""Device memory that a step takes beyond its handle's own (a workspace per term
of the expansion): given back where it cannot be had whole, left alone where
the card is nearly full, one bound for all problems of a batch; the results
do not depend on it."""
import numpy as np
import pytest
import torch

import paper_0809_3739_gb300 as P
from gpu_helpers import seeded_states, wells_problem
from itp_workloads import Grid

pytestmark = pytest.mark.gpu

MiB = 1 << 20
G = Grid(64, 64, 64, 32.0, 32.0, 32.0)
ORDER, TAU, M = 12, 0.1, 80


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def handle(prec, psi):
    h = P.ItpGrid(G.nx, G.ny, G.nz, G.lx, G.ly, G.lz, M, 0, prec)
    h.set_potential(wells_problem(G))
    h.set_states(psi)
    return h


# five more workspaces of 80 states: 5 x 173 MB (FP64), 5 x 87 MB (FP32); tables
# and graph take less than 100 MB
@pytest.mark.parametrize("prec,left", [(P.ITP_FP64, 600 * MiB), (P.ITP_MIXED, 300 * MiB)])
def test_a_nearly_full_card_keeps_its_memory(prec, left):
    psi = seeded_states(G, M)
    with handle(prec, psi) as h:
        E = h.step_graph(ORDER, TAU)
        ref = h.get_states()
    with handle(prec, psi) as h:
        torch.cuda.empty_cache()
        ballast = torch.empty(free() - left, dtype=torch.uint8, device="cuda")
        before = free()
        Es = h.step_graph(ORDER, TAU)
        taken = before - free()
        got = h.get_states()
        del ballast
        torch.cuda.empty_cache()
    print(f"taken {taken / MiB:.0f} MiB of {left / MiB:.0f}")
    assert taken < 100 * MiB
    # term by term, FP32 contributions are summed in FP64 instead of TwoSum
    tol = 0.0 if prec == P.ITP_FP64 else 1e-5
    assert np.max(np.abs(E - Es)) <= tol * np.max(np.abs(E))
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))


def test_a_batch_has_one_bound():
    # eight FP64 problems whose workspaces would be 1.7 GiB
    m = 20
    psi = seeded_states(G, m)
    V = wells_problem(G)
    with P.ItpBatch([(64, 64, 64)] * 8, [(G.lx, G.ly, G.lz)] * 8, [m] * 8,
                    precision=P.ITP_FP64) as b:
        for q in b.problems:
            q.set_potential(V)
            q.set_states(psi)
        before = free()
        E = b.step(ORDER, TAU)
        taken = before - free()
    print(f"taken {taken / MiB:.0f} MiB")
    assert taken < 1024 * MiB + 8 * 100 * MiB / 4   # the bound, and the problems' tables
    with P.ItpGrid(64, 64, 64, G.lx, G.ly, G.lz, m, 0, P.ITP_FP64) as h:
        h.set_potential(V)
        h.set_states(psi)
        Eh = h.step_graph(ORDER, TAU)
    for e in E:
        assert np.array_equal(e, Eh)
