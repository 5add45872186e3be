"""The workloads that the library's speed is measured on.

Each case is what a user's program does with the library, through the Python
binding of its public entry points: create a handle (or a batch) once, hand
over the potential, then per pass load states, iterate, and read the states
and energies.  The sizes are those of the repository's own workloads (the
oscillator on 32^3, the C60-like well on 64^3 to 256^3, the 9 x 9 quantum dots
on 256^2, batches of random-well problems on 32^3 to 96^3) and ragged
grids between them; both precisions are there, whole iterations, the
host-to-host step, the final FP64 evaluation and the orthonormalisation of a
caller's own device block.

A mixed-precision handle keeps its states as FP32 values; a pass over one
hands them on as an FP32 tensor, as a program that goes on with them in torch
does, and its energies, which the FP32 iteration knows to about 1e-7, as FP32.
"""
import math
import random

import numpy as np
import torch

import paper_0809_3739_gb300 as P

#: Axis lengths that the transforms take (products of two of 1, 2, 3, 4, 6,
#: 8, 12, 16), over the range of the listed three-dimensional cases.
EDGES = (18, 24, 32, 36, 48, 64, 72, 96, 128, 144)


def listed():
    return [
        # the textbook start: oscillator, ten states, fourth order, a few
        # steps at a time -- small launches, latency counts
        {"name": "osc32_fp64", "kind": "iterate", "fp64": True, "nx": 32, "ny": 32, "nz": 32,
         "h": 0.5, "well": "osc", "n": 10, "guard": 0, "order": 4, "tau": 0.1, "steps": 4},
        # one small random-well problem on its own, FP32 passes
        {"name": "wells32_mixed", "kind": "iterate", "fp64": False, "nx": 32, "ny": 32, "nz": 32,
         "h": 1.0, "well": "wells", "n": 20, "guard": 4, "order": 8, "tau": 0.25, "steps": 4},
        # a box of three different edges and an odd number of states
        {"name": "ragged_fp64", "kind": "iterate", "fp64": True, "nx": 72, "ny": 48, "nz": 36,
         "h": 0.4, "well": "wells", "n": 33, "guard": 4, "order": 6, "tau": 0.25, "steps": 2},
        # the planar quantum dots: no z transform, planes of 256 x 256
        {"name": "dots256_mixed", "kind": "iterate", "fp64": False, "nx": 256, "ny": 256, "nz": 1,
         "h": 0.125, "well": "dots", "n": 81, "guard": 8, "order": 12, "tau": 0.25, "steps": 4},
        # the C60-like well on its small grid, all FP64
        {"name": "c60_64_fp64", "kind": "iterate", "fp64": True, "nx": 64, "ny": 64, "nz": 64,
         "h": 0.5, "well": "c60", "n": 49, "guard": 8, "order": 12, "tau": 0.25, "steps": 2},
        # the headline: C60-like, 128^3, 120 + 8 states, twelfth order, FP32 passes
        {"name": "c60_128_mixed", "kind": "iterate", "fp64": False, "nx": 128, "ny": 128,
         "nz": 128, "h": 0.25, "well": "c60", "n": 120, "guard": 8, "order": 12, "tau": 0.25,
         "steps": 4},
        # the same grid and order in FP64, a smaller block of states
        {"name": "c60_128_fp64", "kind": "iterate", "fp64": True, "nx": 128, "ny": 128, "nz": 128,
         "h": 0.25, "well": "c60", "n": 40, "guard": 8, "order": 12, "tau": 0.25, "steps": 1},
        # the largest grid: planes that do not fit one SM
        {"name": "c60_256_mixed", "kind": "iterate", "fp64": False, "nx": 256, "ny": 256,
         "nz": 256, "h": 0.125, "well": "c60", "n": 12, "guard": 4, "order": 8, "tau": 0.25,
         "steps": 3},
        # many independent problems of uneven size, one graph launch per step
        {"name": "batch16_mixed", "kind": "batch", "problems": 16, "largest": 96, "box": 32.0,
         "most": 64, "order": 8, "tau": 0.25, "steps": 3},
        # one step from host buffers to host buffers (a driver that keeps
        # its states on the host), a ragged box
        {"name": "host_ragged_mixed", "kind": "host", "fp64": False, "nx": 96, "ny": 72, "nz": 48,
         "h": 0.3, "well": "wells", "n": 55, "guard": 6, "order": 8, "tau": 0.25},
        # the end of a mixed run: orthonormalise and evaluate the block in FP64
        {"name": "final_c60_64", "kind": "final", "nx": 64, "ny": 64, "nz": 64, "h": 0.5,
         "well": "c60", "n": 49, "guard": 79},
        # a caller's own device block, odd number of points, no allocation
        {"name": "ortho_block", "kind": "ortho", "m": 100, "points": 250047},
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Transform work of a drawn case: points x states x transform pairs."""
    k = c.get("order", 2) // 2
    return (c["nx"] * c["ny"] * c["nz"] * (c["n"] + c["guard"]) * (k * (k + 1) // 2 + 1)
            * c.get("steps", 1))


def draw(rng):
    kind = rng.choice(["iterate"] * 7 + ["host", "final", "ortho", "batch"])
    if kind == "ortho":
        m = _log_between(rng, 3, 128)
        return {"kind": kind, "m": m, "points": _log_between(rng, 3000, 40_000_000 // m)}
    if kind == "batch":
        return {"kind": kind, "problems": rng.randint(3, 14), "largest": rng.choice([48, 64, 96]),
                "box": rng.choice([24.0, 32.0]), "most": rng.randint(12, 64),
                "order": rng.choice([4, 6, 8]), "tau": rng.choice([0.1, 0.25]),
                "steps": rng.randint(1, 3)}
    while True:
        c = {"kind": kind}
        if kind != "final":
            c["fp64"] = rng.random() < 0.5
        if rng.random() < 0.15:   # planar
            c.update(nx=rng.choice([64, 96, 128, 192, 256]), ny=rng.choice([64, 96, 128, 192, 256]),
                     nz=1, h=rng.choice([0.125, 0.2]), well=rng.choice(["osc", "dots"]))
        else:
            e = rng.choice(EDGES) if rng.random() < 0.4 else None
            c.update(nx=e or rng.choice(EDGES), ny=e or rng.choice(EDGES),
                     nz=e or rng.choice(EDGES), h=rng.choice([0.25, 0.3, 0.4, 0.5]),
                     well=rng.choice(["osc", "c60", "wells"]))
        c["guard"] = rng.choice([0, 0, 2, 4, 7, 8])
        c["n"] = _log_between(rng, 4, 140)
        if kind != "final":
            c["order"] = rng.choice([2, 4, 6, 8, 10, 12])
            c["tau"] = rng.choice([0.1, 0.25, 0.5])
        if kind == "iterate":
            c["steps"] = rng.randint(1, 4)
        n_points, m = c["nx"] * c["ny"] * c["nz"], c["n"] + c["guard"]
        fp64 = c.get("fp64", True)
        if 40 * m > n_points or m * n_points > 60_000_000:
            continue
        if _cost(c) <= (1_500_000_000 if fp64 else 8_000_000_000):
            return c


# ---- inputs ------------------------------------------------------------------
def _axis(n, length):
    return -0.5 * length + (length / n) * torch.arange(n, dtype=torch.float64)


def _icosahedron(radius):
    """The 60 vertices of a truncated icosahedron."""
    phi = (1.0 + math.sqrt(5.0)) / 2.0
    pts = set()
    for b in ((0.0, 1.0, 3 * phi), (1.0, 2 + phi, 2 * phi), (phi, 2.0, phi ** 3)):
        for s in range(8):
            v = [b[i] * (1 if s >> i & 1 else -1) for i in range(3)]
            for r in range(3):
                pts.add(tuple(round(v[(i + r) % 3], 12) + 0.0 for i in range(3)))
    return [[x * radius / math.sqrt(sum(y * y for y in p)) for x in p] for p in sorted(pts)]


def _potential(shape, box, well, rnd):
    """V on the grid (nz, ny, nx), float64, on the host."""
    z, y, x = (_axis(n, length) for n, length in zip(shape, box))
    if shape[0] == 1:
        z = torch.zeros(1, dtype=torch.float64)
    if well == "osc":
        return 0.5 * (z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2)
    V = torch.zeros(shape, dtype=torch.float64)
    if well == "dots":   # 9 x 9 wells of the sech shape, 3 bohr apart
        for cy in range(-4, 5):
            for cx in range(-4, 5):
                r = torch.sqrt((y[:, None] - 3.0 * cy) ** 2 + (x[None, :] - 3.0 * cx) ** 2)
                V -= (2.0 / torch.cosh(r / 0.6))[None]
        return V
    if well == "c60":
        wells = [(c, 2.0, 0.8) for c in _icosahedron(6.7)]
    else:   # random Gaussian wells, depths 0.5 to 3 Ha, widths 0.5 to 1.2 bohr
        wells = [([rnd.uniform(-0.25, 0.25) * length for length in box[::-1]],
                  rnd.uniform(0.5, 3.0), rnd.uniform(0.5, 1.2)) for _ in range(rnd.randint(4, 40))]
    for (cx, cy, cz), depth, sigma in wells:
        ex, ey, ez = (torch.exp(-(a - c) ** 2 / (2 * sigma ** 2))
                      for a, c in ((x, cx), (y, cy), (z, cz)))
        V -= depth * (ez[:, None, None] * ey[None, :, None] * ex[None, None, :])
    return V


def _k2(shape, box, device):
    """|k|^2 of the half spectrum of a real (nz, ny, nx) grid."""
    k = [2 * math.pi * torch.fft.fftfreq(n, length / n, dtype=torch.float64, device=device)
         for n, length in zip(shape[:2], box[:2])]
    kx = 2 * math.pi * torch.fft.rfftfreq(shape[2], box[2] / shape[2], dtype=torch.float64,
                                          device=device)
    return k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + kx[None, None, :] ** 2


def _states(m, shape, box, seed):
    """m random states as an iteration meets them: smooth (normal noise
    without its shortest waves), of unit norm; float64 on the GPU, (m, N)."""
    gen = torch.Generator("cuda").manual_seed(seed)
    low = torch.exp(-0.125 * _k2(shape, box, "cuda"))
    dV = math.prod(length / n for n, length in zip(shape, box))
    out = torch.empty((m, math.prod(shape)), dtype=torch.float64, device="cuda")
    for j in range(m):
        a = torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)
        a = torch.fft.irfftn(torch.fft.rfftn(a) * low, s=shape)
        out[j] = (a / torch.sqrt((a * a).sum() * dV)).reshape(-1)
    return out


def _grid(case):
    """(shape, box) of a case, both (z, y, x); a planar box is 1 deep."""
    shape = (case["nz"], case["ny"], case["nx"])
    return shape, tuple(1.0 if n == 1 else case["h"] * n for n in shape)


def _problem(case, seed):
    shape, box = _grid(case)
    V = _potential(shape, box, case["well"], random.Random(seed))
    return shape, box, V, _states(case["n"] + case["guard"], shape, box, seed)


def _batch_sizes(case):
    """Edge and state count of each problem of a batch (the problem list of
    a case does not depend on the seed, its potentials and states do)."""
    rnd = random.Random(1000 * case["problems"] + case["largest"])
    edges = [e for e in (32, 48, 64, 96) if e <= case["largest"]]
    return [(rnd.choice(edges), rnd.randint(8, case["most"])) for _ in range(case["problems"])]


def _batch_problems(case, seed):
    for p, (edge, n) in enumerate(_batch_sizes(case)):
        shape, box = (edge,) * 3, (case["box"],) * 3
        V = _potential(shape, box, "wells", random.Random(seed * 1000 + p))
        yield shape, box, V, _states(n, shape, box, seed * 1000 + p)


# ---- the calls -----------------------------------------------------------------
def _handle(case, shape, box, V, fp64):
    h = P.ItpGrid(shape[2], shape[1], shape[0], box[2], box[1], box[0], case["n"], case["guard"],
                  P.ITP_FP64 if fp64 else P.ITP_MIXED)
    h.set_potential(V.numpy())
    return h


def _host_block(*shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ortho":
        gen = torch.Generator("cuda").manual_seed(seed)
        phi = torch.randn((case["m"], case["points"]), dtype=torch.float64, device="cuda",
                          generator=gen)
        state = {"phi": phi, "psi": torch.empty_like(phi)}
    elif kind == "batch":
        probs = list(_batch_problems(case, seed))
        batch = P.ItpBatch([s[::-1] for s, _, _, _ in probs], [b[::-1] for _, b, _, _ in probs],
                           [psi.shape[0] for _, _, _, psi in probs], precision=P.ITP_MIXED)
        for q, (_, _, V, _) in zip(batch.problems, probs):
            q.set_potential(V.numpy())
        out = [_host_block(*psi.shape) for _, _, _, psi in probs]
        state = {"batch": batch, "psi": [psi for _, _, _, psi in probs], "out": out}
    else:
        shape, box, V, psi = _problem(case, seed)
        state = {"h": _handle(case, shape, box, V, case.get("fp64", False)),
                 "out": _host_block(*psi.shape)}
        if kind == "host":
            state["psi"] = _host_block(*psi.shape)
            state["psi"].copy_(psi)
        else:
            state["psi"] = psi
    torch.cuda.synchronize()
    return {"case": case, **state}


def _fp32(host):
    """The FP32 states of a mixed handle, on the GPU, from the host block
    that they were read into."""
    return host.cuda(non_blocking=True).float()


def _read(h, out):
    P.itp.itp_get_states(h.h, out.numpy())
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ortho":
        P.itp_orthonormalize_noalloc(state["phi"].data_ptr(), state["psi"].data_ptr(), case["m"],
                                     case["points"], 0.01,
                                     torch.cuda.current_stream().cuda_stream)
        return state["psi"]
    if kind == "batch":
        batch = state["batch"]
        for q, psi in zip(batch.problems, state["psi"]):
            P.itp.itp_set_states_device(q.h, psi.data_ptr())
        for _ in range(case["steps"]):
            E = batch.step(case["order"], case["tau"])
        return {"E": np.concatenate(E).astype(np.float32),
                "psi": [_fp32(_read(q, out)) for q, out in zip(batch.problems, state["out"])]}
    h = state["h"]
    if kind == "host":
        out, E = h.step_host(case["order"], case["tau"], state["psi"].numpy(),
                             state["out"].numpy())
        out = state["out"]
    elif kind == "final":
        P.itp.itp_set_states_device(h.h, state["psi"].data_ptr())
        E = h.energies("values", fp64=True)
        return {"E": E, "psi": _read(h, state["out"])}
    else:
        P.itp.itp_set_states_device(h.h, state["psi"].data_ptr())
        for _ in range(case["steps"]):
            E = h.step_graph(case["order"], case["tau"])
        out = _read(h, state["out"])
    if case["fp64"]:
        return {"E": E, "psi": out}
    return {"E": E.astype(np.float32), "psi": _fp32(out)}


# ---- what a pass cannot do without -----------------------------------------------
def _iteration(points, m, order, steps):
    """FFT pairs of the propagation, overlap, update, H psi and subspace matrix."""
    k = order // 2
    fft = 2 * 2.5 * points * math.log2(points)
    step = (m * (k * (k + 1) // 2 + 1) * fft + m * (m + 1) * points + m * (m + 1) * points
            + m * (m + 1) * points)
    return {"bytes": 8.0 * points * (2 * m + 1), "flops": float(steps * step)}


def work(case):
    kind = case["kind"]
    if kind == "ortho":
        m, n = case["m"], case["points"]
        return {"bytes": 16.0 * m * n, "flops": 2.0 * m * (m + 1) * n}
    if kind == "batch":
        parts = [_iteration(e ** 3, n, case["order"], case["steps"]) for e, n in _batch_sizes(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    points, m = case["nx"] * case["ny"] * case["nz"], case["n"] + case["guard"]
    if kind == "final":
        return _iteration(points, m, 0, 1)
    return _iteration(points, m, case["order"], case.get("steps", 1))


# ---- the same in 64 bits -----------------------------------------------------------
def _by_state(psi, shape, f):
    """f on blocks of states in grid form."""
    out = torch.empty_like(psi)
    block = max(1, 40_000_000 // psi.shape[1])
    for j in range(0, psi.shape[0], block):
        out[j:j + block] = f(psi[j:j + block].reshape(-1, *shape)).reshape(-1, psi.shape[1])
    return out


def _exact_propagate(psi, V, k2, shape, order, tau):
    k = order // 2

    def block(a):
        total = torch.zeros_like(a)
        for i in range(1, k + 1):
            c = math.prod(i * i / (i * i - j * j) for j in range(1, k + 1) if j != i)
            half, kin = torch.exp(-0.5 * tau / i * V), torch.exp(-0.5 * tau / i * k2)
            u = a
            for _ in range(i):
                u = half * torch.fft.irfftn(torch.fft.rfftn(half * u, dim=(1, 2, 3)) * kin,
                                            s=shape, dim=(1, 2, 3))
            total += c * u
        return total

    return _by_state(psi, shape, block)


def _exact_orthonormal(phi, dV):
    L = torch.linalg.cholesky(phi @ phi.T * dV)
    return torch.linalg.solve_triangular(L, phi, upper=False)


def _exact_ritz(psi, V, k2, shape, dV):
    hpsi = _by_state(psi, shape, lambda a: V * a + torch.fft.irfftn(
        torch.fft.rfftn(a, dim=(1, 2, 3)) * (0.5 * k2), s=shape, dim=(1, 2, 3)))
    H = psi @ hpsi.T * dV
    return torch.linalg.eigvalsh(0.5 * (H + H.T)).cpu()


def _exact_iterate(shape, box, V, psi, order, tau, steps, fp64):
    V, k2 = V.cuda(), _k2(shape, box, "cuda")
    dV = math.prod(length / n for n, length in zip(shape, box))
    if not fp64:
        psi = psi.float().double()   # what a mixed handle takes in
    for _ in range(steps):
        if order:
            psi = _exact_propagate(psi, V, k2, shape, order, tau)
        psi = _exact_orthonormal(psi, dV)
    return _exact_ritz(psi, V, k2, shape, dV), psi


def exact(case, seed):
    kind = case["kind"]
    if kind == "ortho":
        gen = torch.Generator("cuda").manual_seed(seed)
        phi = torch.randn((case["m"], case["points"]), dtype=torch.float64, device="cuda",
                          generator=gen)
        return _exact_orthonormal(phi, 0.01)
    if kind == "batch":
        done = [_exact_iterate(*p, case["order"], case["tau"], case["steps"], False)
                for p in _batch_problems(case, seed)]
        return {"E": torch.cat([E for E, _ in done]), "psi": [psi for _, psi in done]}
    E, psi = _exact_iterate(*_problem(case, seed), case.get("order", 0), case.get("tau", 0.0),
                            case.get("steps", 1), case.get("fp64", False))
    return {"E": E, "psi": psi}
