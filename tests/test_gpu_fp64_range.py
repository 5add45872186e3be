"""FP64 propagation over the range of inputs that the fixed-point passes have
to keep the precision of a double for: smooth and rough states, single points,
plane waves, amplitudes far from one and deep or high potentials, against the
oracle, each state relative to its own largest value."""
import numpy as np
import pytest

import paper_0809_3739_gb300 as P
from gpu_helpers import propagate_tolerance, report, seeded_states, wells_problem
from itp_workloads import Grid
from oracle import itp_oracle as O

pytestmark = pytest.mark.gpu


def odd_states(g):
    x, y, z = (np.arange(n) for n in (g.nx, g.ny, g.nz))
    shape = (g.nz, g.ny, g.nx)
    point = np.zeros(shape)
    point[g.nz // 2, 1, 2] = 1.0
    wave = np.cos(2 * np.pi * (3 * x[None, None, :] / g.nx + y[None, :, None] / g.ny
                               + 0 * z[:, None, None]))
    decay = np.exp(-1.5 * (x[None, None, :] + y[None, :, None] + z[:, None, None]))
    noise = seeded_states(g, 4, seed=77).reshape(4, *shape)
    blocks = [point, wave + 0 * point, np.ones(shape), decay, noise[0], noise[1] * 1e-120,
              noise[2] * 1e120, noise[3] * decay]
    return np.stack(blocks).reshape(len(blocks), g.n_points)


@pytest.mark.parametrize("dims", [(32, 32, 32), (24, 18, 12), (128, 128, 4), (64, 64, 1),
                                  (256, 192, 1), (4, 6, 256)])
@pytest.mark.parametrize("offset", [0.0, -30.0, 200.0])
def test_each_state_keeps_double_precision(dims, offset):
    g = Grid(*dims, *(0.4 * n if n > 1 else 1.0 for n in dims))
    V = wells_problem(g) + offset
    psi = odd_states(g)
    order, tau = 6, 0.2
    ref = O.propagate(psi, V, g, order, tau)
    with P.ItpGrid(*dims, g.lx, g.ly, g.lz, len(psi), 0, P.ITP_FP64) as h:
        h.set_potential(V)
        h.set_states(psi)
        h.propagate(order, tau)
        phi = h.get_phi()
    tol = propagate_tolerance(order, g.n_points, "fp64")
    err = np.max(np.abs(phi - ref), axis=1) / np.max(np.abs(ref), axis=1)
    report(f"FP64 range {dims} V+{offset}", err.max(), tol)
    assert np.all(err < tol), err


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_state_is_reported(bad):
    g = Grid(24, 18, 12, 9.0, 7.0, 5.0)
    psi = seeded_states(g, 3, seed=5)
    psi[1, 100] = bad
    with P.ItpGrid(g.nx, g.ny, g.nz, g.lx, g.ly, g.lz, 3, 0, P.ITP_FP64) as h:
        h.set_potential(wells_problem(g))
        h.set_states(psi)
        h.propagate(4, 0.2)
        assert not np.isfinite(h.get_phi()[1]).any()
        h.orthonormalize()
        with pytest.raises(P.ItpError) as e:
            h.synchronize()
        assert e.value.code == 3
