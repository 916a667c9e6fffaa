"""Measured workloads of the coupled cathode step.

Each case is one thing a program does with this package: advance a lattice
and read it, watch every step's current, sweep operating points, or take the
gradient of the current.  A pass starts from wherever the last pass on the
same domain ended, as a time-marching program's does.

`exact` restates the method in torch at 64 bits, vectorised over the lattice:
stream with the boundary links, velocity and pressure (Eq. 8, 11 of arXiv
2103.01444), MRT collisions (Eq. 1, 3-7 and 10), catalyst sources
(Eq. 12-17).  Gradients come from torch's own differentiation of it.

Numbers that a domain computes in 32 bits come back as float32, those of
16-bit storage as 16-bit floats of the same type, those of FP64 storage as
float64.
"""
import math

import numpy as np
import torch

from paper_2103_01444_gb300.lbm import Batch, Domain, cathode_objective

# ------------------------------------------------------------------- cases
# kind "run":     from a state `warm` steps old: step(n), then the fields and (cathodes) current_density()
#      "observe": step_observe(n), residual(), then the fields; the first snapshot of the
#                 residual is `warm` steps old
#      "sweep":   Batch.step(n) over `count` cathodes of uneven size, then each one's read-outs
#      "grad":    grad(nsteps=n) into device tensors, from a state `warm` steps old
#      "design":  cathode_objective: forward and backward of torch.autograd
# material: "layers" (channel over a uniform GDL, thin catalyst film),
#      "blocks" (porosity and permeability drawn per block, catalyst rows),
#      "grains" (4 x 4 solid grains in the GDL, thin film), "cavity"
# steps are those of one pass.


def _case(name, kind, nx, ny, steps, precision="fp32", material="blocks", **more):
    d = dict(name=name, kind=kind, nx=nx, ny=ny, steps=steps, precision=precision,
             material=material, rounding="nearest", tune=False, count=1, warm=0)
    d.update(more)
    return d


def listed():
    return [
        # the shortest useful call: a controller moves a small cell ten steps and
        # looks at its current; all launches and host latency
        _case("poll_200x40_fp32", "run", 200, 40, 10, material="layers"),
        # the 200 x 40 cathode of the parity runs, marched a thousand steps at a time
        _case("march_200x40_fp32", "run", 200, 40, 1000, material="layers"),
        # steady-state studies run in FP64 storage; an odd lattice, every width ragged
        _case("steady_509x127_fp64", "observe", 509, 127, 100, precision="fp64", warm=40),
        # a polarisation transient watched step by step on the adjoint's lattice
        # (its two states fit in the L2 cache)
        _case("observe_1024x256_fp32", "observe", 1024, 256, 128, tune=True, warm=40),
        # the production lattice with the whole hot path: update, every step's
        # current to the host, the residual
        _case("observe_4096x1024_fp32", "observe", 4096, 1024, 64, tune=True, warm=40),
        # the same lattice in 16-bit storage
        _case("run_4096x1024_bf16", "run", 4096, 1024, 64, precision="bf16", tune=True),
        # pore-scale GDL at full size: FP16 with stochastic rounding is the 16-bit
        # storage that holds its fields over a long run
        _case("grains_8192x2048_fp16sr", "run", 8192, 2048, 32, precision="fp16",
              material="grains", rounding="stochastic", tune=True),
        # natural convection in a closed box (Sec. 3), not a power of two, once it has begun to turn
        _case("cavity_1000x1000_fp32", "run", 1000, 1000, 100, material="cavity", warm=1500),
        # the paper's operating-point sweeps: 64 uneven cathodes
        _case("sweep_64_cases_fp32", "sweep", 2048, 512, 64, count=64, tune=True),
        # and many small ones, each far too small to fill the GPU
        _case("sweep_96_small_fp32", "sweep", 512, 128, 128, count=96, tune=True),
        # gradient of the mean current to the material of a 1024 x 256 cathode
        _case("grad_1024x256_fp32", "grad", 1024, 256, 256, warm=400),
        # one iteration of a design loop on a small cathode through torch.autograd; in FP64
        # storage, which the gradients to porosity and permeability need
        _case("design_250x64_fp64", "design", 250, 64, 150, precision="fp64"),
    ]


def _between(rng, lo, hi):
    """A whole number, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "observe", "sweep", "grad", "design"])
    if kind == "sweep":
        nx, ny, count = _between(rng, 200, 2048), _between(rng, 64, 512), _between(rng, 8, 64)
        return dict(_case("", kind, nx, ny, rng.randrange(20, 97), count=count,
                          tune=rng.random() < 0.5), **{"name": "sweep %d %dx%d" % (count, nx, ny)})
    if kind in ("grad", "design"):
        nx, ny = _between(rng, 96, 1024), _between(rng, 32, 256)
        precision = "fp64" if kind == "design" else rng.choice(["fp32", "fp32", "fp64"])
        if precision == "fp64":
            nx, ny = nx // 2, max(24, ny // 2)
        return _case("%s %dx%d %s" % (kind, nx, ny, precision), kind, nx, ny, rng.randrange(40, 257), precision=precision,
                     material=rng.choice(["blocks", "layers"]), warm=300 if kind == "grad" else 0)
    nx = _between(rng, 100, 6000)
    ny = max(24, min(2048, int(nx * rng.uniform(0.15, 0.5))))
    material = rng.choice(["layers", "blocks", "blocks", "grains"] + (["cavity"] if kind == "run" else []))
    precision = rng.choice(["fp32", "fp32", "bf16", "fp16", "fp64"])
    if nx * ny > 1 << 21 and precision == "fp64":
        precision = "fp32"
    if material == "cavity":   # young, it is at rest: its velocity would be rounding alone
        nx, ny = min(nx, 1200), min(ny, 600)
    rounding = rng.choice(["nearest", "stochastic"]) if precision in ("bf16", "fp16") and material != "cavity" else "nearest"
    steps = max(5, min(_between(rng, 5, 400), int(2.5e8 / (nx * ny))))
    return _case("%s %dx%d %s" % (kind, nx, ny, precision), kind, nx, ny, steps, precision=precision,
                 material=material, rounding=rounding, tune=rng.random() < 0.5,
                 warm=40 if kind == "observe" else 1500 if material == "cavity" else 0)


# ------------------------------------------------------------------ inputs
# Constants of the paper (Nomenclature, Eq. 13-19) and the lattice scales of
# this package's cathodes: nu = D_O2 = 0.05, Pr 0.7, D_H2O = 1.3 D_O2,
# (rho c_p)_s / (rho c_p)_f = 1500, k_s / k_f = 1.5 / 0.026.
_DEV = "cuda"


def _cathode(nx, ny, material, seed):
    """(params, fields, geometry) of one cathode in lattice units."""
    gen = torch.Generator().manual_seed(seed * 1000003 + nx * 4099 + ny)
    u = lambda lo, hi, *s: lo + (hi - lo) * torch.rand(*s, generator=gen, dtype=torch.float64)  # noqa: E731
    ny_cl = max(1, round(0.05 * ny)) if material == "blocks" else 0
    ny_gdl = round(0.55 * ny) if material == "blocks" else (ny // 2 if material == "layers" else ny - round(0.4 * ny))
    rows = ny - ny_cl - ny_gdl
    dx = 254.4e-4 / ny_gdl
    dt = 0.05 * dx * dx / 5.2197e-2
    phi, K = torch.ones(ny, nx, dtype=torch.float64), torch.full((ny, nx), math.inf, dtype=torch.float64)
    gdl = slice(ny_cl, ny_cl + ny_gdl)
    solid = None
    if material == "blocks":
        b = 32 if nx * ny >= 1 << 18 else 8
        grid = (-(-ny // b), -(-nx // b))
        spread = lambda t: t.repeat_interleave(b, 0).repeat_interleave(b, 1)[:ny, :nx]  # noqa: E731
        phi[gdl] = spread(u(0.4, 0.8, *grid))[gdl]
        K[gdl] = spread(10.0 ** u(-12.0, -10.0, *grid))[gdl] * 1e4 / dx ** 2
        phi[:ny_cl], K[:ny_cl] = 0.4, 1e-8 / dx ** 2
    elif material == "layers":
        phi[gdl] = float(u(0.5, 0.7, 1))
        K[gdl] = float(u(0.5e-3, 2e-3, 1)) * ny_gdl ** 2
    else:
        t = torch.rand(ny_gdl // 4, nx // 4, generator=gen) < 0.3
        solid = torch.zeros(ny, nx, dtype=torch.uint8)
        s = t.to(torch.uint8).repeat_interleave(4, 0).repeat_interleave(4, 1)
        solid[:s.shape[0], :s.shape[1]] = s
        solid[:, :4] = 0
        solid[:, nx - 4:] = 0
    phi, K = phi.to(_DEV), K.to(_DEV)
    kr, cr, a_gas = 1.5 / 0.026, 1500.0, 0.05 / 0.7
    fields = dict(phi=phi, K=K, alpha_T=a_gas * (phi + kr * (1 - phi)) / (phi + cr * (1 - phi)),
                  D_O2=0.05 * phi ** 1.5, D_H2O=0.065 * phi ** 1.5, rho_cp_ratio=phi + cr * (1 - phi))
    # Re as high as the workload's 50, lower where a short channel would need a fast inlet
    Re = min(float(u(20.0, 50.0, 1)), 0.06 * rows / 0.05)
    c_tot = 17.808e-6 / 0.21
    T_in = float(u(338.0, 353.0, 1))
    params = dict(nu=0.05, u_in_avg=Re * 0.05 / rows, body_force_x=0.0, V_op=float(u(0.4, 0.7, 1)), T_in=T_in,
                  C_O2_in=0.21, C_H2O_in=0.0, T_top=T_in, C_O2_top=0.21, C_H2O_top=0.0, aj0_ref=1e-4,
                  T_ref_kin=353.15, E_act=16456.0, alpha_c=1.0, F=96487.0, R=8.314, dU0dT=0.0025, U0_0=0.2329,
                  x_ref=0.21, dx_cm=dx, dt_s=dt, delta_cl_cm=10e-4, c_tot=c_tot, rho_cp_f=29.3 * c_tot,
                  forchheimer=1, top_dirichlet=0, interface_mode=1, inlet_mode=0, dp_in=0.0, alpha_a=0.0,
                  scalar_advection=1)
    geometry = dict(nx=nx, ny=ny, ny_cl=ny_cl, ny_gdl=ny_gdl, reaction_mode=1 if ny_cl else 0, periodic_x=0,
                    solid=None if solid is None else solid.numpy())
    return params, fields, geometry


def _cavity(nx, ny, seed):
    """Natural convection between a hot left and a cold right wall over a hot floor."""
    gen = torch.Generator().manual_seed(seed * 1000003 + nx * 4099 + ny)
    Ra = 10.0 ** (5.0 + float(torch.rand(1, generator=gen, dtype=torch.float64)))
    Pr, L, hot, cold = 0.71, float(nx), 348.0, 338.0
    alpha = min(0.1, 0.05 * L / math.sqrt(Ra * Pr))
    nu, mean = Pr * alpha, 0.5 * (hot + cold)
    full = lambda v: torch.full((ny, nx), float(v), dtype=torch.float64, device=_DEV)  # noqa: E731
    fields = dict(phi=full(1.0), K=full(math.inf), alpha_T=full(alpha), D_O2=full(alpha), D_H2O=full(alpha),
                  rho_cp_ratio=full(1.0))
    params = dict(nu=nu, u_in_avg=0.0, body_force_x=0.0, V_op=0.0, T_in=mean, C_O2_in=0.21, C_H2O_in=0.0,
                  T_top=mean, C_O2_top=0.21, C_H2O_top=0.0, aj0_ref=0.0, T_ref_kin=343.0, E_act=0.0, alpha_c=0.0,
                  F=0.25, R=8.314, dU0dT=0.0, U0_0=0.0, x_ref=1.0, dx_cm=1.0, dt_s=1.0, delta_cl_cm=1.0, c_tot=1.0,
                  rho_cp_f=1.0, forchheimer=1, top_dirichlet=0, interface_mode=1, inlet_mode=0, dp_in=0.0,
                  alpha_a=0.0, buoy_gx=0.0, buoy_gy=Ra * nu * alpha / ((hot - cold) * L ** 3), T_buoy=mean,
                  wall_dirichlet=(1 << 0) | (1 << 3) | (1 << 6),
                  C_wall=[[hot, 0.21, 0.0], [cold, 0.21, 0.0], [hot, 0.21, 0.0]], scalar_advection=1)
    geometry = dict(nx=nx, ny=ny, ny_cl=0, ny_gdl=0, reaction_mode=0, periodic_x=0, closed_x=1, solid=None)
    return params, fields, geometry


def _problem(case, seed):
    if case["material"] == "cavity":
        return _cavity(case["nx"], case["ny"], seed)
    return _cathode(case["nx"], case["ny"], case["material"], seed)


def _sweep_sizes(case):
    """The lattices of a sweep: nx down to a quarter and ny down to a quarter of the largest; fixed by the case."""
    gen = torch.Generator().manual_seed(case["nx"] * 8191 + case["ny"] * 31 + case["count"])
    f = torch.rand(case["count"], 2, generator=gen, dtype=torch.float64)
    return [(max(48, int(case["nx"] * (0.25 + 0.75 * float(a)))), max(24, int(case["ny"] * (0.25 + 0.75 * float(b)))))
            for a, b in f]


def _problems(case, seed):
    if case["kind"] != "sweep":
        return [_problem(case, seed)]
    return [_cathode(nx, ny, case["material"], seed + 7919 * k) for k, (nx, ny) in enumerate(_sweep_sizes(case))]


# ----------------------------------------------------------------- program
_KEEP = 3   # cathodes of a sweep whose read-outs come back one by one; those of the others are put end to end


class _Reader:
    """One domain with the device buffers its program reads the fields into."""

    def __init__(self, case, problem, stream, out=None):
        params, fields, geometry = problem
        self.stream = stream
        self.domain = Domain(precision=case["precision"], rounding=case["rounding"], stream=stream.cuda_stream, **geometry)
        self.domain.set_params(params)
        self.domain.set_fields(**fields)
        self.domain.reset()
        self.raw = torch.empty(6, geometry["ny"], geometry["nx"], dtype=torch.float64, device=_DEV)
        self.np_type = np.float64 if case["precision"] == "fp64" else np.float32
        dtype = {"fp64": torch.float64, "fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[case["precision"]]
        self.out = torch.empty_like(self.raw, dtype=dtype) if out is None else out.view(self.raw.shape)
        self.cathode = "closed_x" not in geometry

    def fields(self):
        self.domain.fields(out=self.raw)
        with torch.cuda.stream(self.stream):
            self.out.copy_(self.raw)
        o = self.out
        return {"u": o[:2], "p": o[2], "T": o[3], "C_O2": o[4], "C_H2O": o[5]}

    def current(self):
        i_avg, heat, profile = self.domain.current_density()
        return {"i_avg": self.np_type(i_avg), "heat": self.np_type(heat), "profile": profile}


def prepare(case, seed):
    stream = torch.cuda.Stream()
    problems = _problems(case, seed)
    torch.cuda.synchronize()
    if case["kind"] in ("run", "observe", "sweep"):
        state = dict(case=case, stream=stream)
        if case["kind"] == "sweep":
            sizes = [p[2]["nx"] * p[2]["ny"] for p in problems]
            ends = np.concatenate([[0], np.cumsum(sizes[_KEEP:])])
            state["flat"] = torch.empty(6, int(ends[-1]), dtype=torch.float32, device=_DEV)
            outs = [None] * _KEEP + [state["flat"][:, a:b] for a, b in zip(ends[:-1], ends[1:])]
            readers = [_Reader(case, p, stream, o) for p, o in zip(problems, outs)]
            state["batch"] = Batch([r.domain for r in readers])
            if case["tune"]:
                state["batch"].tune(3)
        else:
            readers = [_Reader(case, problems[0], stream)]
            if case["tune"]:
                readers[0].domain.tune(10)
            readers[0].domain.step(case["warm"])
        state["readers"] = readers
        if case["kind"] == "observe":
            readers[0].domain.residual()
            state["i"], state["heat"] = np.zeros(case["steps"]), np.zeros(case["steps"])
        return state
    params, fields, geometry = problems[0]
    domain = Domain(precision=case["precision"], stream=stream.cuda_stream, **geometry)
    domain.set_params(params)
    domain.set_fields(**fields)
    domain.reset()
    state = dict(case=case, stream=stream, domain=domain, params=params, fields=fields)
    if case["kind"] == "grad":
        domain.step(case["warm"])
        state["out"] = {k: torch.empty_like(fields["phi"]) for k in ("phi", "K", "D_O2")}
    else:
        state["function"] = cathode_objective()
    return state


def run(state):
    case, stream = state["case"], state["stream"]
    stream.wait_stream(torch.cuda.current_stream())
    kind, n = case["kind"], case["steps"]
    if kind == "sweep":
        state["batch"].step(n)
        got = [dict(r.current(), **r.fields()) for r in state["readers"]]
        rest, flat = got[_KEEP:], state["flat"]
        out = {"first": got[:_KEEP],
               "rest": {"u": flat[:2], "p": flat[2], "T": flat[3], "C_O2": flat[4], "C_H2O": flat[5],
                        **{k: np.array([r[k] for r in rest]) for k in ("i_avg", "heat")},
                        "profile": np.concatenate([r["profile"] for r in rest])}}
    elif kind == "run":
        r = state["readers"][0]
        r.domain.step(n)
        out = r.fields()
        if r.cathode:
            out.update(r.current())
    elif kind == "observe":
        r = state["readers"][0]
        i, heat = r.domain.step_observe(n, state["i"], state["heat"])
        out = dict(r.fields(), i=i.astype(r.np_type), heat=heat.astype(r.np_type),
                   residual=r.np_type(r.domain.residual()))
    elif kind == "grad":
        J, g = state["domain"].grad(objective=0, nsteps=n, out=state["out"])
        np_type, dtype = (np.float64, torch.float64) if case["precision"] == "fp64" else (np.float32, torch.float32)
        out = {"J": np_type(J), "u_in": np_type(g["u_in"])}
        out.update({k: g[k].to(dtype, copy=True) for k in ("phi", "K", "D_O2")})   # grad() waited for its stream
    else:
        f = state["fields"]
        leaves = [f[k].clone().requires_grad_(True) for k in ("phi", "K", "D_O2")]
        u_in = torch.tensor(state["params"]["u_in_avg"], dtype=torch.float64, device=_DEV, requires_grad=True)
        torch.cuda.current_stream().synchronize()   # the library reads the material on its own stream
        J = state["function"].apply(*leaves, u_in, state["domain"], f, state["params"], 0, n, 0)
        J.backward()
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        out = {"J": J.detach().to(dtype), "u_in": u_in.grad.to(dtype)}
        out.update({k: t.grad.to(dtype) for k, t in zip(("phi", "K", "D_O2"), leaves)})
    torch.cuda.current_stream().wait_stream(stream)
    return out


# -------------------------------------------------------------------- work
def work(case):
    """Populations, mask and material index read once, populations and read-outs written once; about 420 operations
    for a cell and step, three times that where the step is also transposed."""
    es = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}[case["precision"]]
    rs = max(es, 4)
    sizes = _sweep_sizes(case) if case["kind"] == "sweep" else [(case["nx"], case["ny"])]
    cells = sum(nx * ny for nx, ny in sizes)
    if case["kind"] in ("grad", "design"):
        return {"bytes": cells * (24 * es + 3 + 3 * 8 + 3 * rs), "flops": 1260 * cells * case["steps"]}
    return {"bytes": cells * (48 * es + 3 + 6 * 8 + 6 * (8 + es)), "flops": 420 * cells * case["steps"]}


# ------------------------------------------------------------------- exact
_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_M = ((1, 1, 1, 1, 1, 1, 1, 1, 1), (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1),
      (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, -2, 0, 2, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1),
      (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))
_N = ((1, 1, 1, 1, 1), (0, 1, 0, -1, 0), (0, 0, 1, 0, -1), (-4, 1, 1, 1, 1), (0, 1, -1, 1, -1))


class _Lattice:
    """The method at 64 bits on one lattice; `leaves` replaces phi, K, D_O2 and u_in_avg."""

    def __init__(self, params, fields, geometry, leaves=None):
        p, g = params, geometry
        self.p, self.nx, self.ny = p, g["nx"], g["ny"]
        self.ny_cl, self.y0, self.mode = g["ny_cl"], g["ny_cl"] + g["ny_gdl"], g["reaction_mode"]
        self.closed = bool(g.get("closed_x", 0))
        d = leaves or {}
        dev = fields["phi"].device
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
        self.M, self.N = t(_M), t(_N)
        self.Mi, self.Ni = torch.linalg.inv(self.M), torch.linalg.inv(self.N)
        self.phi = d.get("phi", fields["phi"])
        K = d.get("K", fields["K"])
        clear = torch.isinf(fields["K"])
        Ks = torch.where(clear, torch.ones_like(K), K)
        zero = torch.zeros_like(self.phi)
        self.darcy = torch.where(clear, zero, self.phi * p["nu"] / Ks)
        self.forch = torch.where(clear, zero, 0.143 * self.phi ** -0.5 / torch.sqrt(Ks)) if p["forchheimer"] else zero
        self.l0, self.l1 = 0.5 + 0.25 * self.darcy, 0.5 * self.forch
        self.u_in = d.get("u_in", t(p["u_in_avg"]))
        solid = torch.zeros(self.ny, self.nx, dtype=torch.bool, device=dev)
        if g["solid"] is not None:
            solid = torch.from_numpy(g["solid"]).to(dev).bool()
        self.live = (~solid).double()
        alpha = (fields["alpha_T"], d.get("D_O2", fields["D_O2"]), fields["D_H2O"])
        self.b, self.q1 = [], []
        for a in alpha:   # Fickian interfaces: one b per scalar, each cell's diffusivity in the flux rate
            top = float(a.detach()[~solid].max())
            b = 20 * math.sqrt(3.0) * top - 4
            self.b.append(b)
            self.q1.append(1 / (a / ((4 + b) / 10) + 0.5))
        self.q3 = 6 / (3 + 2 * math.sqrt(3.0))
        tau = 3 * p["nu"] + 0.5
        sq = 8 * (2 - 1 / tau) / (8 - 1 / tau)
        self.S = t([1 / tau, 1 / tau, 1 / tau, 0.0, sq, 0.0, sq, 1 / tau, 1 / tau])[:, None, None]
        self.pw = [float(v) for v in self.Mi @ t([0.0, 6.0, -9.0, 0, 0, 0, 0, 0, 0])]
        self.sigma = fields["rho_cp_ratio"]
        self.Cin = (p["T_in"], p["C_O2_in"], p["C_H2O_in"])
        y = torch.arange(self.ny, device=dev)[:, None].expand(self.ny, self.nx)
        x = torch.arange(self.nx, device=dev)[None, :].expand(self.ny, self.nx)
        self.y = y[:, 0].double()
        self.inlet = (self.y >= self.y0) & (not self.closed)      # open rows of the inlet column
        self.bounce = []
        for i in range(9):
            sx, sy = x - _EX[i], y - _EY[i]
            wall = (sy < 0) | (sy >= self.ny) | (sx < 0) | ((sx >= self.nx) & self.closed)
            inside = (sx >= 0) & (sx < self.nx) & (sy >= 0) & (sy < self.ny)
            src = torch.roll(solid, (_EY[i], _EX[i]), (0, 1))
            self.bounce.append(wall | (inside & src))

    def start(self):
        f = torch.tensor(_W, dtype=torch.float64, device=self.phi.device)[:, None, None] * self.live
        g = [torch.stack([torch.full_like(self.phi.detach(), (1 - b) / 5 * c)] +
                         [torch.full_like(self.phi.detach(), (4 + b) / 20 * c)] * 4) * self.live
             for b, c in zip(self.b, self.Cin)]
        return f, g

    def _parabola(self, h):
        s = (h - self.y0 + 0.5) / (self.ny - self.y0)
        return torch.where((s > 0) & (s < 1), 6 * self.u_in * s * (1 - s), torch.zeros_like(s))

    def _column(self, v, x, col):
        """v with column x replaced by col."""
        c = col[:, None]
        return torch.cat([c, v[:, 1:]], 1) if x == 0 else torch.cat([v[:, :-1], c], 1)

    def _rates(self, T):
        p = self.p
        eta = p["V_op"] - (p["dU0dT"] * T + p["U0_0"])
        return (p["aj0_ref"] * torch.exp(-p["E_act"] * (1 / T - 1 / p["T_ref_kin"])) / p["x_ref"] *
                torch.exp(-p["alpha_c"] * p["F"] / (p["R"] * T) * eta))

    def stream(self, f, g):
        """Post-stream values, the volumetric sink and the O2 consumed per column (lattice units)."""
        p = self.p
        # flow
        cols = None
        if not self.closed:
            e = f[:, :, -1]
            jx = sum(_EX[k] * e[k] for k in range(9) if _EX[k])
            jy = sum(_EY[k] * e[k] for k in range(9) if _EY[k])
            ph = 0.6 * e[1:].sum(0) - 0.4 * (jx * jx + jy * jy) / self.phi[:, -1]
            cols = [e[k] + self.pw[k] * (1 / 3 - ph) for k in range(9)]
        fo = []
        for i in range(9):
            own = f[_OP[i]]
            v = torch.where(self.bounce[i], own, torch.roll(f[i], (_EY[i], _EX[i]), (0, 1))) if i else f[0]
            inner = (self.y - _EY[i] >= 0) & (self.y - _EY[i] <= self.ny - 1)
            if not self.closed and _EX[i] == 1:
                push = 6 * _W[i] * self._parabola(self.y - 0.5 * _EY[i])
                v = self._column(v, 0, own[:, 0] + torch.where(self.inlet & inner, push, torch.zeros_like(push)))
            if not self.closed and _EX[i] == -1:
                v = self._column(v, -1, torch.where(inner, torch.roll(cols[i], _EY[i], 0), own[:, -1]))
            fo.append(v * self.live)
        fo = torch.stack(fo)
        # scalars
        go = []
        wd, Cw = p.get("wall_dirichlet", 0), p.get("C_wall")
        for s in range(3):
            w1, gs, out = (4 + self.b[s]) / 20, g[s], []
            for i in range(5):
                own = gs[_OP[i]]
                v = torch.where(self.bounce[i], own, torch.roll(gs[i], (_EY[i], _EX[i]), (0, 1))) if i else gs[0]
                if i == 2 and (wd >> (6 + s)) & 1:
                    v = torch.cat([(-own[:1] + 2 * w1 * Cw[2][s]), v[1:]], 0)
                if i == 1:
                    o = own[:, 0]
                    held = (self.inlet, self.Cin[s]) if not self.closed else (torch.ones_like(self.inlet), Cw[0][s])
                    if not self.closed or (wd >> s) & 1:
                        v = self._column(v, 0, torch.where(held[0], -o + 2 * w1 * held[1], o))
                if i == 3 and self.closed and (wd >> (3 + s)) & 1:
                    v = self._column(v, -1, -own[:, -1] + 2 * w1 * Cw[1][s])
                if i == 3 and not self.closed:
                    v = self._column(v, -1, gs[3][:, -1])
                out.append(v * self.live)
            go.append(out)
        hpo = 4 * p["F"] * p["c_tot"] * (p["V_op"] - p["U0_0"]) / p["rho_cp_f"]   # Eq. 15 with Eq. 16
        sink = None
        if self.mode == 0:
            k = self._rates(g[0][:, 0].sum(0)) * p["delta_cl_cm"] / (4 * p["F"] * p["c_tot"]) * p["dt_s"] / p["dx_cm"]
            kap = k / (2 * (4 + self.b[1]) / 20)
            down = go[1][2][0]
            J = (down - down * (1 - kap) / (1 + kap)) * self.live[0]
            row = lambda v, add: torch.cat([(v[0] + add)[None], v[1:]], 0)  # noqa: E731
            go[1][2] = row(go[1][2], -J)
            go[2][2] = row(go[2][2], 2 * J)
            go[0][2] = row(go[0][2], hpo / self.sigma[0] * J)
        else:
            n = self.ny_cl
            k = self._rates(g[0][:, :n].sum(0)) / (4 * p["F"] * p["c_tot"]) * p["dt_s"]
            sink = -k * g[1][:, :n].sum(0) / (1 + k)
            J = -sink.sum(0)
        return fo, [torch.stack(v) for v in go], sink, J, hpo

    def _force(self, T):
        p = self.p
        gx = p["body_force_x"] + p.get("buoy_gx", 0.0) * (T - p.get("T_buoy", 0.0))
        return gx, p.get("buoy_gy", 0.0) * (T - p.get("T_buoy", 0.0))

    def macros(self, f, g):
        C = [v.sum(0) for v in g]
        gx, gy = self._force(C[0])
        vx = sum(_EX[k] * f[k] for k in range(9) if _EX[k]) + 0.5 * self.phi * gx
        vy = sum(_EY[k] * f[k] for k in range(9) if _EY[k]) + 0.5 * self.phi * gy
        v2 = vx * vx + vy * vy
        vn = torch.where(v2 > 0, torch.sqrt(torch.where(v2 > 0, v2, torch.ones_like(v2))), torch.zeros_like(v2))
        den = self.l0 + torch.sqrt(self.l0 * self.l0 + self.l1 * vn)
        ux, uy = vx / den, vy / den
        pr = 0.6 / self.phi * f[1:].sum(0) - 0.4 * (ux * ux + uy * uy) / self.phi ** 2
        return ux, uy, vn / den, pr, C, gx, gy

    def step(self, f, g):
        """(f, g) one step on, the step's J per column and hpo."""
        fs, gs, sink, J, hpo = self.stream(f, g)
        ux, uy, un, pr, C, gx, gy = self.macros(fs, gs)
        phi = self.phi
        Fx = -self.darcy * ux - self.forch * un * ux + phi * gx
        Fy = -self.darcy * uy - self.forch * un * uy + phi * gy
        u2, uF, one = ux * ux + uy * uy, ux * Fx + uy * Fy, torch.ones_like(ux)
        meq = torch.stack([one, -4 + 6 * phi * pr + 3 * u2 / phi, 4 - 9 * phi * pr - 3 * u2 / phi, ux, -ux, uy, -uy,
                           (ux * ux - uy * uy) / phi, ux * uy / phi])
        G = torch.stack([0 * one, 6 * uF / phi, -6 * uF / phi, Fx, -Fx, Fy, -Fy, 2 * (ux * Fx - uy * Fy) / phi,
                         (ux * Fy + uy * Fx) / phi])
        m = torch.tensordot(self.M, fs, 1)
        f = torch.tensordot(self.Mi, m - self.S * (m - meq) + (1 - 0.5 * self.S) * G, 1) * self.live
        out = []
        for s in range(3):
            Ca, b = C[s] - self.Cin[s], self.b[s]
            n = torch.tensordot(self.N, gs[s], 1)
            n = torch.stack([n[0], n[1] - self.q1[s] * (n[1] - ux * Ca), n[2] - self.q1[s] * (n[2] - uy * Ca),
                             n[3] - self.q3 * (n[3] - b * C[s]), n[4] - self.q3 * n[4]])
            v = torch.tensordot(self.Ni, n, 1)
            if sink is not None:
                k = self.ny_cl
                src = (-sink * hpo / self.sigma[:k], sink, -2 * sink)[s]
                w = torch.tensor([(1 - b) / 5] + [(4 + b) / 20] * 4, dtype=torch.float64, device=v.device)
                v = torch.cat([v[:, :k] + w[:, None, None] * src, v[:, k:]], 1)
            out.append(v * self.live)
        return f, out, J, hpo

    def current(self, J, hpo):
        """Mean current (A/cm^2), mean heat (W/cm^2) and the local current of a step's J."""
        p = self.p
        i = J * (4 * p["F"] * p["c_tot"] * p["dx_cm"] / p["dt_s"])
        heat = (J * hpo).sum() * (p["rho_cp_f"] * p["dx_cm"] / p["dt_s"]) / self.nx
        return i.sum() / self.nx, heat, i

    def fields(self, f, g):
        """Fields of the step that (f, g) is about to take."""
        fs, gs = self.stream(f, g)[:2]
        ux, uy, _, pr, C, _, _ = self.macros(fs, gs)
        on = self.live
        return {"u": torch.stack([ux, uy]) * on, "p": pr * on, "T": C[0] * on, "C_O2": C[1] * on, "C_H2O": C[2] * on}

    def moments(self, f, g):
        X = [sum(_EX[k] * f[k] for k in range(9) if _EX[k]), sum(_EY[k] * f[k] for k in range(9) if _EY[k]),
             (g[0].sum(0) - self.Cin[0]) * self.live, g[1].sum(0), g[2].sum(0)]
        return torch.stack(X)


def _marched(lat, warm, steps):
    """The state before the last of `steps` steps, the state after it, every step's (i, heat), the last profile, and the
    moments of the state `warm` steps old from which they start."""
    f, g = lat.start()
    for _ in range(warm):
        f, g = lat.step(f, g)[:2]
    first = lat.moments(f, g)
    i, heat = [], []
    for k in range(steps):
        before = (f, g)
        f, g, J, hpo = lat.step(f, g)
        a, q, profile = lat.current(J, hpo)
        i.append(a)
        heat.append(q)
    return before, (f, g), torch.stack(i), torch.stack(heat), profile, first


def _residual(a, b):
    r = 0.0
    for x, y in zip(a, b):
        num, den = float((x - y).square().sum()), float(x.square().sum())
        r = max(r, math.sqrt(num / den) if den > 0 else 0.0)
    return r


def _exact_grad(lat_of, params, fields, geometry, warm, n):
    leaves = {k: fields[k].clone().requires_grad_(True) for k in ("phi", "K", "D_O2")}
    leaves["u_in"] = torch.tensor(params["u_in_avg"], dtype=torch.float64, device=_DEV, requires_grad=True)
    with torch.no_grad():
        lat = lat_of(params, fields, geometry)
        state = lat.start()
        for _ in range(warm):
            state = lat.step(*state)[:2]
    # the mean current of step n, its graph rebuilt in stretches of steps
    chunk, marks = 8, [state]
    with torch.no_grad():
        for k in range(n - 1):
            state = lat.step(*state)[:2]
            if (k + 1) % chunk == 0:
                marks.append(state)
    names = list(leaves)
    total = {k: torch.zeros_like(v) for k, v in leaves.items()}
    lam, J_value, at = None, None, n - 1
    for c in range(len(marks) - 1, -1, -1):
        lo = c * chunk
        if at < lo or (at == lo and c < len(marks) - 1):
            continue
        f, g = marks[c]
        f = f.clone().requires_grad_(True)
        g = [v.clone().requires_grad_(True) for v in g]
        lat = lat_of(params, fields, geometry, leaves)
        state = (f, g)
        for _ in range(at - lo):
            state = lat.step(*state)[:2]
        if lam is None:
            J, hpo = lat.stream(*state)[3:]
            goal = lat.current(J, hpo)[0]
            J_value = goal.detach()
        else:
            goal = (state[0] * lam[0]).sum() + sum((a * b).sum() for a, b in zip(state[1], lam[1]))
        got = torch.autograd.grad(goal, [f, *g] + [leaves[k] for k in names], allow_unused=True)
        got = [torch.zeros_like(v) if t is None else t for t, v in zip(got, [f, *g] + [leaves[k] for k in names])]
        lam, at = (got[0], got[1:4]), lo
        for k, t in zip(names, got[4:]):
            total[k] += t
    return dict({k: total[k] for k in names}, J=J_value)


def exact(case, seed):
    # a step takes a few ms of launches, or some sixty passes over a 24-value FP64 state
    steps = case["warm"] + case["steps"]
    if case["kind"] in ("grad", "design"):
        if (steps + 3 * case["steps"]) * max(8e-3, case["nx"] * case["ny"] * 1.2e-8) > 18:
            return None
        params, fields, geometry = _problem(case, seed)
        return _exact_grad(_Lattice, params, fields, geometry, case["warm"], case["steps"])
    sizes = _sweep_sizes(case)[:_KEEP] if case["kind"] == "sweep" else [(case["nx"], case["ny"])]
    if sum(steps * max(5e-3, nx * ny * 6e-9) for nx, ny in sizes) > 18:
        return None
    out = []
    with torch.no_grad():
        for k, (nx, ny) in enumerate(sizes):
            lat = _Lattice(*(_cathode(nx, ny, case["material"], seed + 7919 * k) if case["kind"] == "sweep"
                             else _problem(case, seed)))
            before, after, i, heat, profile, first = _marched(lat, case["warm"], case["steps"])
            r = lat.fields(*before)
            if case["precision"] == "fp16":
                r["C_H2O"] = None   # the water of so few steps is below FP16's spacing
            if case["kind"] == "observe":
                r.update(i=i, heat=heat, residual=_residual(lat.moments(*after), first))
            elif case["material"] != "cavity":
                r.update(i_avg=i[-1], heat=heat[-1], profile=profile)
            out.append(r)
    return {"first": out, "rest": None} if case["kind"] == "sweep" else out[0]
