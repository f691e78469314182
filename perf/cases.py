"""Performance cases of the EBIT phase-change framework: what its users run, over the real range.

A pass is one call a simulation program makes, through paper_2402_13677_gb300/ebit.py and the C ABI
behind it:

  * "step": ebit_step(n) of one instance, then the whole new state read back into the caller's
    device buffers (a snapshot, as a program that couples or stores the fields takes it);
  * "host_step": the same with the state coming from and going to page-locked host buffers each
    step, as bench.py's end-to-end figure has it;
  * "batch": ebit_step(n) of many instances of uneven size in one context, and their state;
  * "solve": the library's solver on a caller's five-point system, device arrays
    (ebit_solve_system_noalloc) or host arrays (ebit_solve_system).

Grids, properties and time steps are those of paper_2402_13677_gb300/workloads.py (bench.py runs
them at the same sizes) or lie between them; every step solves to the 1e-8 relative residual that
bench.py and config_from_problem use.  The multigrid schedule is the library's default one.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w

FIELDS = {"T_l": E.F_T_L, "T_v": E.F_T_V, "u_l": E.F_U_L, "u_v": E.F_U_V, "ufx_l": E.F_UFX_L, "ufx_v": E.F_UFX_V,
          "ufy_l": E.F_UFY_L, "ufy_v": E.F_UFY_V, "p": E.F_P, "gc": E.F_GC, "mdot": E.F_MDOT, "vcol": E.F_VCOL,
          "hx_pos": E.F_HX_POS, "vy_pos": E.F_VY_POS}
INTERFACE = ("vcol", "hx_pos", "vy_pos")
RTOL = 1e-8          # of the steps: bench.py's, and the default of config_from_problem
FMIN = w.FMIN


def listed():
    return [
        # the smallest simulation: a front on 64 x 64 cells in FP64, where launches and latency count
        {"name": "stefan_64_fp64", "kind": "step", "problem": "stefan", "nx": 64, "ny": 64, "precision": "fp64",
         "steps": 10},
        # the benchmark's headline: the bubble on 512 x 512, FP32 solves inside FP64 refinement
        {"name": "bubble_512_mixed", "kind": "step", "problem": "bubble", "nx": 512, "ny": 512, "precision": "mixed",
         "steps": 4},
        # the same in the parity precision
        {"name": "bubble_512_fp64", "kind": "step", "problem": "bubble", "nx": 512, "ny": 512, "precision": "fp64",
         "steps": 2},
        # the one-fluid variant on a smaller grid of ragged tiles
        {"name": "bubble_336_one_fluid", "kind": "step", "problem": "bubble_one_fluid", "nx": 336, "ny": 336,
         "precision": "mixed", "steps": 4},
        # an axisymmetric bubble with surface tension
        {"name": "axi_bubble_160_mixed", "kind": "step", "problem": "axi_bubble", "nx": 160, "ny": 160,
         "precision": "mixed", "steps": 6},
        # film boiling at the ordinary size, ...
        {"name": "film_1024x2048_mixed", "kind": "step", "problem": "film", "nx": 1024, "ny": 2048,
         "precision": "mixed", "steps": 2},
        # ... in FP64 with surface tension on an odd size, ...
        {"name": "film_416x736_sigma_fp64", "kind": "step", "problem": "film_sigma", "nx": 416, "ny": 736,
         "precision": "fp64", "steps": 2},
        # ... and at the largest
        {"name": "film_4096_mixed", "kind": "step", "problem": "film_wide", "nx": 4096, "ny": 4096,
         "precision": "mixed", "steps": 1},
        # a program that keeps its state on the host between steps
        {"name": "host_bubble_512_mixed", "kind": "host_step", "problem": "bubble", "nx": 512, "ny": 512,
         "precision": "mixed", "steps": 1},
        # many independent instances of uneven size
        {"name": "batch_384_mixed", "kind": "batch", "count": 384, "precision": "mixed", "steps": 6},
        # the solver alone on small device arrays (a service loop that may not allocate), ...
        {"name": "solve_120x104_fp64", "kind": "solve", "system": "helmholtz", "nx": 120, "ny": 104, "nr": 2,
         "precision": "fp64", "rtol": 1e-12, "device": True},
        # ... and on a host program's larger system
        {"name": "solve_512x256_mixed", "kind": "solve", "system": "poisson", "nx": 512, "ny": 256, "nr": 1,
         "precision": "mixed", "rtol": 1e-10, "device": False},
    ]


def _side(rng, lo, hi, k):
    """A multiple of 2^k between lo and hi, spread over their logarithm."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2 ** k)) * 2 ** k
    return min(max(n, -(-lo // 2 ** k) * 2 ** k), hi // 2 ** k * 2 ** k)


def _levels(cells):
    """Halvings that bring a grid of that many cells to the solver's coarsest level (1024 cells)."""
    k = 0
    while cells > 1024:
        cells /= 4
        k += 1
    return k


def draw(rng):
    prec = rng.choice(["mixed", "mixed", "fp64"])
    kind = rng.choice(["step", "step", "step", "host_step", "batch", "solve"])
    if kind == "batch":
        return {"kind": "batch", "count": int(math.exp(rng.uniform(math.log(8), math.log(512)))), "precision": prec,
                "steps": rng.randint(3, 6)}
    if kind == "solve":
        device = rng.random() < 0.5
        if device and rng.random() < 0.3:      # one level, odd sides
            nx, ny = rng.randint(5, 31), rng.randint(5, 31)
        else:
            top = 128 if device else 1024
            side = _side(rng, 32, top, 0)
            k = _levels(4.0 * side * side)
            nx, ny = _side(rng, max(32, side // 2), min(top, 2 * side), k), _side(rng, max(32, side // 2), side, k)
        return {"kind": "solve", "system": rng.choice(["poisson", "helmholtz"]), "nx": nx, "ny": ny,
                "nr": rng.choice([1, 2]), "precision": prec, "rtol": 1e-10 if prec == "mixed" else 1e-12,
                "device": device}
    problem = rng.choice(["stefan", "bubble", "bubble_one_fluid", "axi_bubble", "film", "film_sigma", "film_wide"])
    if problem.startswith("film"):
        side = math.exp(rng.uniform(math.log(96), math.log(2900 if kind == "step" and prec == "mixed" else 900)))
        k = _levels(2.5 * side * side)
        nx, ny = _side(rng, int(side) // 2 + 2 ** k, int(side) + 2 ** k, k), _side(rng, int(side), int(1.4 * side), k)
    else:
        side = math.exp(rng.uniform(math.log(40), math.log(520)))
        k = _levels(side * side)
        nx = ny = int(side) // 2 ** k * 2 ** k
    cells = nx * ny
    return {"kind": kind, "problem": problem, "nx": nx, "ny": ny, "precision": prec,
            "steps": 1 if kind == "host_step" or cells > 4 << 20 else (2 if cells > 1 << 19 else 4)}


# ---------------------------------------------------------------------------------------------
# initial states on the device
# ---------------------------------------------------------------------------------------------
def _full(shape, value=0.0, dtype=torch.float64):
    return torch.full(shape, value, dtype=dtype, device="cuda")


def _at_rest(pb, st):
    nx, ny = pb.nx, pb.ny
    st.update(u_l=_full((ny, nx, 2)), u_v=_full((ny, nx, 2)), ufx_l=_full((ny, nx + 1)), ufx_v=_full((ny, nx + 1)),
              ufy_l=_full((ny + 1, nx)), ufy_v=_full((ny + 1, nx)), p=_full((ny, nx)))
    return pb, st


def _centres(pb):
    x = pb.x0 + pb.h * (torch.arange(pb.nx, dtype=torch.float64, device="cuda") + 0.5)
    y = pb.y0 + pb.h * (torch.arange(pb.ny, dtype=torch.float64, device="cuda") + 0.5)
    return x[None, :], y[:, None]


def _interface(phi, pb):
    """Vertex colours (1 where phi > 0) and the roots of phi on the cut edges (bisection)."""
    nx, ny, h = pb.nx, pb.ny, pb.h
    xs = pb.x0 + h * torch.arange(nx + 1, dtype=torch.float64, device="cuda")
    ys = pb.y0 + h * torch.arange(ny + 1, dtype=torch.float64, device="cuda")
    vcol = (phi(xs[None, :], ys[:, None]) > 0).to(torch.uint8).expand(ny + 1, nx + 1).contiguous()
    out = [vcol]
    for axis in (0, 1):
        a, b = (vcol[:, :-1], vcol[:, 1:]) if axis == 0 else (vcol[:-1, :], vcol[1:, :])
        j, i = torch.nonzero(a != b, as_tuple=True)
        up = a[j, i] == 0                       # phi rises along the edge
        lo, hi = torch.zeros_like(xs[i]), torch.ones_like(xs[i])
        for _ in range(52):
            m = 0.5 * (lo + hi)
            f = phi(xs[i] + h * m, ys[j]) if axis == 0 else phi(xs[i], ys[j] + h * m)
            left = (f > 0) == up                # the root lies below m
            lo, hi = torch.where(left, lo, m), torch.where(left, m, hi)
        pos = _full((ny + 1, nx) if axis == 0 else (ny, nx + 1))
        pos[j, i] = (0.5 * (lo + hi)).clamp(FMIN, 1.0 - FMIN)
        out.append(pos)
    return dict(zip(INTERFACE, out))


def _stefan(n_x, n_y, rng, rho_l=10.0, St=0.1, dt=1e-4, X0=None):
    """The planar front of workloads.stefan: vapour on a hot wall, erf profile, liquid leaving."""
    h = 1.0 / n_x
    X0 = 0.1 * (1.0 + 0.05 * rng.uniform(-1, 1)) if X0 is None else X0
    beta = w.stefan_beta(St)
    t0 = (X0 / (2.0 * beta)) ** 2
    if dt is None:
        dt = 0.2 * h / (beta / math.sqrt(t0))
    pb = w.Problem("stefan", n_x, n_y, h, dt=dt, rho_l=rho_l, h_lg=1.0 / St,
                   bc=(w.WALL, w.OUTFLOW, w.SYMMETRY, w.SYMMETRY), T_bc=(1.0, None, None, None), t0=t0)
    st = _interface(lambda x, y: x - X0 + 0.0 * y, pb)
    x, _ = _centres(pb)
    T_v = 1.0 - torch.erf(x / (2.0 * math.sqrt(t0))) / math.erf(beta)
    st.update(T_v=T_v.expand(n_y, n_x).contiguous(), T_l=_full((n_y, n_x)))
    _at_rest(pb, st)
    U = beta / math.sqrt(t0) * (1.0 - 1.0 / rho_l)
    st["u_l"][..., 0] = U
    st["ufx_l"][:, 1:] = U
    return pb, st


def _bubble_layer(n, rng, rho=20.0, St=0.2, R0=0.15, axi=False, sigma=0.0, cfl=0.2):
    """The bubble of workloads.bubble_layer: fluid at rest, a linear thermal layer of two cells;
    axisymmetric: a sphere on the axis with surface tension."""
    h, R0 = 1.0 / n, R0 * (1.0 + 0.05 * rng.uniform(-1, 1))
    delta = 2.0 * h
    S, O = w.SYMMETRY, w.OUTFLOW
    pb = w.Problem("bubble_layer", n, n, h, dt=cfl * h * delta / St, rho_l=rho, h_lg=1.0 / St, sigma=sigma, axi=axi,
                   bc=(S, O, S, O) if axi else (O, O, O, O))
    c = 0.0 if axi else 0.5
    st = _interface(lambda x, y: torch.sqrt((x - c) ** 2 + (y - c) ** 2) - R0, pb)
    x, y = _centres(pb)
    r = torch.sqrt((x - c) ** 2 + (y - c) ** 2)
    st.update(T_l=((r - R0) / delta).clamp(0.0, 1.0), T_v=_full((n, n)))
    return _at_rest(pb, st)


def _film(nx, ny, rng, wide, sigma):
    """The films of workloads.film: c3_film's properties, or c5_film's with `wide`."""
    props = dict(rho_l=50.0, mu_l=1e-2, mu_v=1e-3, lam_l=1e-2, lam_v=1e-3, h_lg=10.0) if wide else \
        dict(rho_l=5.0, mu_l=5e-3, mu_v=1e-3, lam_l=1e-2, lam_v=1e-3, h_lg=1.0 / 0.064)
    Lx = 8.0 * nx / 4096 if wide else 1.0
    modes = 32 * nx // 4096 + 1 if wide else rng.randint(1, 4)
    h = Lx / nx
    mean = max(0.05, 4.0 * h)
    if sigma:
        sigma = (props["rho_l"] - 1.0) / (12.0 * math.pi ** 2)   # Taylor wavelength = domain width
    pb = w.Problem("film", nx, ny, h, dt=0.25 * h, rho_v=1.0, gy=-1.0, sigma=sigma,
                   bc=(w.SYMMETRY, w.SYMMETRY, w.WALL, w.OUTFLOW), T_bc=(None, None, 1.0, None), **props)
    ks = [2.0 * math.pi * (k + 1) / Lx for k in range(modes)]
    a = [0.1 * mean / modes * rng.choice([-1.0, 1.0]) * rng.uniform(0.9, 1.1) for _ in ks]

    def eta(x):
        return mean + sum(q * torch.cos(k * x) for q, k in zip(a, ks))

    st = _interface(lambda x, y: y - eta(x), pb)
    x, y = _centres(pb)
    st.update(T_v=1.0 - y / eta(x), T_l=_full((ny, nx)))
    return _at_rest(pb, st)


def _problem(case, seed):
    """(Problem, its fields as device tensors) of a step case."""
    import random
    rng = random.Random(1000003 * seed + 17)
    kind, nx, ny = case["problem"], case["nx"], case["ny"]
    if kind == "stefan":
        return _stefan(nx, ny, rng)
    if kind == "axi_bubble":
        return _bubble_layer(nx, rng, R0=0.3, axi=True, sigma=0.05, cfl=0.02)
    if kind.startswith("film"):
        return _film(nx, ny, rng, kind == "film_wide", 1.0 if kind == "film_sigma" else 0.0)
    # the planar bubble with its similarity profile and seeded noise, the time step of the 512^2 grid
    # scaled to the cell size
    pb = w.bubble(nx, R0=max(0.05, 8.0 / nx) * (1.0 + 0.05 * rng.uniform(-1, 1)), dt=1.96e-6 * (512.0 / nx) ** 2,
                  seed=1 + seed)
    if kind == "bubble_one_fluid":
        pb = w.one_fluid(pb)
    st = {k: torch.from_numpy(np.ascontiguousarray(getattr(pb, k))).cuda()
          for k in ("T_l", "T_v", "u_l", "u_v", "ufx_l", "ufx_v", "ufy_l", "ufy_v", "p", "vcol", "hx_pos", "vy_pos")}
    return pb, st


def _precision(case):
    return E.EBIT_FP64 if case["precision"] == "fp64" else E.EBIT_MIXED


# ---------------------------------------------------------------------------------------------
# a program's state
# ---------------------------------------------------------------------------------------------
class Sim:
    """A context with its instances and the caller's buffers; destroyed with the program's object."""

    def __init__(self, case, problems):
        self.case, self.ctx = case, None
        self.alloc, self.stream = E.TorchAllocator(), torch.cuda.Stream()
        self.lib = E.load()
        self.ctx = E.ebit_init([E.config_from_problem(pb, _precision(case), RTOL, 400) for pb, _ in problems],
                               self.stream.cuda_stream, self.alloc)
        torch.cuda.synchronize()
        for b, (pb, st) in enumerate(problems):
            liq, vap = E.props_from_problem(pb)
            E.ebit_set_phase_props(self.ctx, b, liq, vap, pb.T_sat, pb.h_lg, pb.sigma, pb.gx, pb.gy)
            E.check(self.ctx, self.lib.ebit_set_interface(self.ctx, b, *[st[k].data_ptr() for k in INTERFACE], 1))
            names = [k for k in FIELDS if k in st and k not in INTERFACE]
            E.ebit_set_fields(self.ctx, b, [FIELDS[k] for k in names], [st[k].data_ptr() for k in names], True)
            E.ebit_set_time(self.ctx, b, pb.t0)
        E.ebit_run_stage(self.ctx, E.STAGE_PREPARE)
        # one buffer per field over all instances
        n = len(problems)
        shape = {k: [E.ebit_field_shape(self.ctx, b, f) for b in range(n)] for k, f in FIELDS.items()}
        host = case["kind"] == "host_step"
        self.out, ptrs = {}, [[] for _ in range(n)]
        for k in FIELDS:
            sizes = [c * e for c, e in shape[k]]
            buf = torch.empty(sum(sizes), dtype=torch.uint8, pin_memory=True) if host else \
                torch.empty(sum(sizes), dtype=torch.uint8, device="cuda")
            at = 0
            for b, s in enumerate(sizes):
                ptrs[b].append(buf.data_ptr() + at)
                at += s
            self.out[k] = buf if k == "vcol" else buf.view(torch.float64)
        self.ids = (ctypes.c_int * len(FIELDS))(*FIELDS.values())
        self.ptrs = [(ctypes.c_void_p * len(FIELDS))(*p) for p in ptrs]
        self.state_ids = (ctypes.c_int * (len(FIELDS) - 3))(*[f for k, f in FIELDS.items() if k not in INTERFACE])
        self.state_ptrs = (ctypes.c_void_p * (len(FIELDS) - 3))(
            *[p for k, p in zip(FIELDS, ptrs[0]) if k not in INTERFACE])
        self.read()

    def read(self):
        dev = 0 if self.case["kind"] == "host_step" else 1
        for b, p in enumerate(self.ptrs):
            E.check(self.ctx, self.lib.ebit_get_fields(self.ctx, b, len(p), self.ids, p, dev))
        return self.out

    def __del__(self):
        if self.ctx is not None:
            E.ebit_destroy(self.ctx)


def _batch_problems(case, seed):
    """Instances of workloads.c4_instance's ranges: sides 32..256, fronts and bubbles, uneven properties."""
    import random
    grids, rng = random.Random(case["count"]), random.Random(7919 * seed + 3)
    out = []
    for _ in range(case["count"]):
        n, front = grids.choice(w.C4_SIDES), grids.random() < 0.5    # the case's, not the seed's
        St, rho = rng.uniform(0.05, 0.5), rng.uniform(2.0, 100.0)
        if front:
            out.append(_stefan(n, n, rng, rho_l=rho, St=St, dt=None))
        else:
            out.append(_bubble_layer(n, rng, rho=rho, St=St))
    return out


class System:
    """A five-point system of a caller's program with its known solution."""

    def __init__(self, case, seed):
        nx, ny, nr = case["nx"], case["ny"], case["nr"]
        g = torch.Generator(device="cuda").manual_seed(int(seed))

        def uniform(*shape):
            return torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda")

        self.case = case
        x = torch.linspace(0.0, 1.0, nx, dtype=torch.float64, device="cuda")[None, :]
        y = torch.linspace(0.0, 1.0, ny, dtype=torch.float64, device="cuda")[:, None]
        self.wl, self.wb = _full((ny, nx)), _full((ny, nx))
        c = uniform(3)
        inside = (x - 0.3 - 0.4 * c[0]) ** 2 + (y - 0.3 - 0.4 * c[1]) ** 2 < (0.1 + 0.15 * c[2]) ** 2
        coef = torch.where(inside, 1.0, 20.0) * (1.0 + 0.01 * uniform(ny, nx))
        if case["system"] == "poisson":     # a pressure system: weights 1 / rho, Dirichlet on the top side
            self.wl[:, 1:] = 2.0 / (coef[:, 1:] + coef[:, :-1])
            self.wb[1:, :] = 2.0 / (coef[1:, :] + coef[:-1, :])
            self.D = _full((ny, nx))
            self.D[-1, :] = 2.0 / coef[-1, :]
        else:                               # a diffusion system: mean conductances, rho c / dt on the diagonal
            self.wl[:, 1:] = 0.5 * (coef[:, 1:] + coef[:, :-1])
            self.wb[1:, :] = 0.5 * (coef[1:, :] + coef[:-1, :])
            self.D = 0.5 + 0.1 * uniform(ny, nx)
        self.solution = torch.sin(5.0 * x + 3.0 * y)[..., None] + 0.1 * uniform(ny, nx, nr)
        s = self.solution
        b = self.D[..., None] * s
        fl, fb = self.wl[:, 1:, None] * (s[:, 1:] - s[:, :-1]), self.wb[1:, :, None] * (s[1:] - s[:-1])
        b[:, 1:] += fl
        b[:, :-1] -= fl
        b[1:] += fb
        b[:-1] -= fb
        self.b = b
        self.ctx = None
        self.x = torch.empty_like(s)
        self.stream = torch.cuda.Stream()
        if not case["device"]:
            self.host = [t.reshape(-1).cpu().numpy() for t in (self.D, self.wl, self.wb, self.b)]
            self.alloc = E.TorchAllocator()
            pb = w.Problem("system", nx, ny, 1.0 / nx)
            self.ctx = E.ebit_init([E.config_from_problem(pb, _precision(case))], self.stream.cuda_stream, self.alloc)

    def __del__(self):
        if self.ctx is not None:
            E.ebit_destroy(self.ctx)


# ---------------------------------------------------------------------------------------------
# the cases' interface
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    if case["kind"] == "solve":
        return System(case, seed)
    problems = _batch_problems(case, seed) if case["kind"] == "batch" else [_problem(case, seed)]
    return Sim(case, problems)


def run(state):
    case = state.case
    if case["kind"] == "solve":
        if not case["device"]:
            D, wl, wb, b = state.host
            x, _, _ = E.ebit_solve_system(state.ctx, 0, D, wl, wb, b, nr=case["nr"], precision=_precision(case),
                                          rtol=case["rtol"], max_iter=500)
            return x
        with torch.cuda.stream(state.stream):
            state.x.zero_()
        s, _, _ = E.ebit_solve_system_noalloc(case["nx"], case["ny"], state.D, state.wl, state.wb, state.b, state.x,
                                              nr=case["nr"], precision=_precision(case), rtol=case["rtol"],
                                              max_iter=500, stream=state.stream.cuda_stream)
        if s != E.EBIT_OK:
            raise RuntimeError(E.STATUS_NAMES.get(s, s))
        return state.x.view(-1)
    if case["kind"] == "host_step":
        o = state.out
        E.check(state.ctx, state.lib.ebit_set_interface(state.ctx, 0, *[o[k].data_ptr() for k in INTERFACE], 0))
        E.check(state.ctx, state.lib.ebit_set_fields(state.ctx, 0, len(state.state_ids), state.state_ids,
                                                     state.state_ptrs, 0))
        E.ebit_run_stage(state.ctx, E.STAGE_RECONSTRUCT)
    E.ebit_step(state.ctx, case["steps"], allow_noconv=True)
    return state.read()


def _mean_cells():
    return sum(n * n for n in w.C4_SIDES) / len(w.C4_SIDES)


def work(case):
    """Bytes: a step reads the state once and writes it once, 16 words and a colour byte per cell each
    way; a solve reads D, wl, wb, b and writes x.  Operations: the least the method has per cell, the
    explicit stencils of a step (about 600) and one preconditioned iteration (about 150) per
    unknown of its implicit systems (temperature, four velocity components, pressure)."""
    if case["kind"] == "solve":
        cells, nr = case["nx"] * case["ny"], case["nr"]
        return {"bytes": 8.0 * cells * (3 + 2 * nr), "flops": 150.0 * cells * nr}
    cells = case["count"] * _mean_cells() if case["kind"] == "batch" else case["nx"] * case["ny"]
    return {"bytes": 2.0 * 129.0 * cells * case["steps"], "flops": 1500.0 * cells * case["steps"]}


def exact(case, seed):
    """The solution a system's right-hand side was made from (in 64 bits); a step has no closed value."""
    if case["kind"] != "solve":
        return None
    return System({**case, "device": True}, seed).solution.reshape(-1)
