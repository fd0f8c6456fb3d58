"""Work that programs built on this solver have it do, as cases to time and compare.

Each case goes through the public entry points of paper_2406_19920_gb300 with
device-resident fields, as a flow solver calls them:

  poisson    one pressure solve (ibm_poisson_solve), wall-bounded or triply
             periodic, FP32 with refinement or FP64
  helmholtz  one implicit viscous solve with wall data
             (ibm_helmholtz_solve_bc) or without (ibm_helmholtz_solve)
  step       one whole time step: the three RK stages, with markers
             (ibm_substep, or ibm_substep_inout)
  markers    one interpolation and one spreading (ibm_interp, ibm_spread)
  batch      Poisson solves of many uneven grids in one call
             (ibm_batch_poisson)

Sizes are those of the repository's tests and benchmark or lie between them:
the transform lengths are 2^a 3^b in [8, 512], the wall axis takes any length
in [8, 512].  exact() states every result in plain FP64 torch.
"""

import ctypes
import math

import torch

import paper_2406_19920_gb300 as ibm

LENGTHS = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512)
CELL_NEUMANN, CELL_DIRICHLET, FACE_DIRICHLET = 0, 1, 2
STATIC, TRANSLATE, HEAVE = 0, 1, 2

ALPHA = (4 / 15, 1 / 15, 1 / 6)
GAMMA = (8 / 15, 5 / 12, 3 / 4)
ZETA = (0.0, -17 / 60, -5 / 12)


def listed():
    return [
        # a small pressure solve, as a batch instance or a served request is: launches and latency
        {"name": "poisson_f32_48x33x24", "kind": "poisson", "nx": 48, "ny": 33, "nz": 24, "dtype": "f32", "refine": 1},
        # the ordinary simulation grid of the tests and the benchmark
        {"name": "poisson_f32_128", "kind": "poisson", "nx": 128, "ny": 128, "nz": 128, "dtype": "f32", "refine": 1},
        # the benchmark's headline solve
        {"name": "poisson_f32_256", "kind": "poisson", "nx": 256, "ny": 256, "nz": 256, "dtype": "f32", "refine": 1},
        # a large grid with radix-3 lengths and a wall axis that is no power of two
        {"name": "poisson_f32_384x200x192", "kind": "poisson", "nx": 384, "ny": 200, "nz": 192, "dtype": "f32",
         "refine": 1},
        # double precision, on the grid of the reference's smaller sphere run
        {"name": "poisson_f64_256x128x128", "kind": "poisson", "nx": 256, "ny": 128, "nz": 128, "dtype": "f64",
         "refine": 0},
        # the triply periodic branch, on the grid of the reference's larger sphere run
        {"name": "poisson_3p_f32_512x256x256", "kind": "poisson", "nx": 512, "ny": 256, "nz": 256, "dtype": "f32",
         "refine": 1, "periodic": True},
        # one implicit viscous solve of the wall-normal velocity with wall data, odd wall axis
        {"name": "helmholtz_f32_192x129x96", "kind": "helmholtz", "nx": 192, "ny": 129, "nz": 96, "dtype": "f32",
         "refine": 1, "field": FACE_DIRICHLET, "walls": True},
        # a time step of the ordinary simulation: 128^3 with a translating sphere of 20,000 markers
        {"name": "step_f32_128_sphere20k", "kind": "step", "nx": 128, "ny": 128, "nz": 128, "dtype": "f32",
         "refine": 1, "markers": 20000, "motion": TRANSLATE},
        # a time step of the large simulation: a heaving plate of 100,000 markers
        {"name": "step_f32_384x256x256_plate100k", "kind": "step", "nx": 384, "ny": 256, "nz": 256, "dtype": "f32",
         "refine": 1, "markers": 100000, "motion": HEAVE},
        # a double-precision time step between inflow and outflow walls, odd wall axis
        {"name": "step_f64_inout_96x65x64", "kind": "step", "nx": 96, "ny": 65, "nz": 64, "dtype": "f64", "refine": 0,
         "markers": 4000, "motion": STATIC, "inout": True},
        # the Lagrangian operations alone, on a dense marker set
        {"name": "markers_f32_128_100k", "kind": "markers", "nx": 128, "ny": 128, "nz": 128, "dtype": "f32",
         "markers": 100000},
        # a parameter sweep: many uneven grids solved in one call
        {"name": "batch_f32_16", "kind": "batch", "dtype": "f32", "refine": 1,
         "cubes": "32,64,96,48,128,32,64,48,96,32,48,64,128,32,64,96"},
    ]


def draw(rng):
    def length(lo, hi):
        return rng.choice([n for n in LENGTHS if lo <= n <= hi])

    def wall(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(lo, hi, most, periodic=False):
        while True:
            nx, nz = length(lo, hi), length(lo, hi)
            ny = length(lo, hi) if periodic else wall(lo, hi)
            if nx * ny * nz <= most:
                return {"nx": nx, "ny": ny, "nz": nz}

    kind = rng.choice(["poisson", "poisson", "poisson", "helmholtz", "helmholtz", "step", "step", "markers", "batch"])
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    c = {"kind": kind, "dtype": dtype}
    if kind in ("poisson", "helmholtz"):
        periodic = rng.random() < 0.25
        c.update(grid(8, 512, 1 << 24 if dtype == "f64" else 1 << 25, periodic))
        c["refine"] = 0 if dtype == "f64" else rng.choice([0, 1, 1, 1, 2])
        if periodic:
            c["periodic"] = True
        if kind == "helmholtz" and not periodic:
            c["field"] = rng.choice([CELL_NEUMANN, CELL_DIRICHLET, FACE_DIRICHLET])
            c["walls"] = rng.random() < 0.5
    elif kind == "step":
        c.update(grid(32, 384, 1 << 21 if dtype == "f64" else 25 << 20))
        c["refine"] = 0 if dtype == "f64" else 1
        c["markers"] = int(round(10 ** rng.uniform(2.5, 5)))
        c["motion"] = rng.choice([STATIC, TRANSLATE, HEAVE])
        if rng.random() < 0.3:
            c["inout"] = True
    elif kind == "markers":
        c.update(grid(32, 256, 1 << 23))
        c["markers"] = int(round(10 ** rng.uniform(2.5, 5.3)))
        c["peskin"] = rng.random() < 0.3
        c["gather"] = rng.random() < 0.2
    else:
        c["refine"] = 0 if dtype == "f64" else 1
        c["cubes"] = ",".join(str(length(16, 96)) for _ in range(rng.randint(2, 16)))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _real(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _spacings(case):
    if case.get("motion") == HEAVE:  # the plate's box: uniform spacing
        return (2 * math.pi / case["nx"],) * 3
    return (2 * math.pi / case["nx"], 2.0 / case["ny"], 2 * math.pi / case["nz"])


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _noise(shape, kmax, slope, gen):
    """Periodic noise with spectral amplitude |k|^slope up to index wavenumber kmax."""
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device=_device(), dtype=torch.float64))
    ky, kz = (torch.fft.fftfreq(n, 1.0 / n, device=_device(), dtype=torch.float64) for n in shape[:2])
    kx = torch.fft.rfftfreq(shape[2], 1.0 / shape[2], device=_device(), dtype=torch.float64)
    k = torch.sqrt(ky[:, None, None] ** 2 + kz[None, :, None] ** 2 + kx[None, None, :] ** 2)
    f *= torch.where((k > 0) & (k <= kmax), k.clamp(min=1.0) ** slope, torch.zeros_like(k))
    f = torch.fft.irfftn(f, s=shape)
    return f / torch.sqrt(torch.mean(f * f)).clamp(min=1e-300)


def _rhs(nx, ny, nz, gen):
    """A right-hand side with a smooth part and broadband noise; its mean is not quite zero."""
    shape = (ny, nz, nx)
    f = _noise(shape, 32.0, 0.0, gen)
    return f + 1e-3 * torch.randn(shape, generator=gen, device=_device(), dtype=torch.float64)


def _velocity(case, gen):
    """A random discretely divergence-free velocity with v = 0 on the walls: the curl of an edge-centred potential."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    hx, hy, hz = _spacings(case)
    kmax = min(nx, ny, nz) / 4
    j = torch.arange(ny + 1, device=_device(), dtype=torch.float64)
    env_e = (torch.sin(math.pi * j / ny) ** 2)[:, None, None]
    env_c = (torch.sin(math.pi * (j[:ny] + 0.5) / ny) ** 2)[:, None, None]
    ax, az = (_noise((ny + 1, nz, nx), kmax, -17 / 6, gen) * env_e for _ in range(2))
    ay = _noise((ny, nz, nx), kmax, -17 / 6, gen) * env_c
    ax[0] = ax[ny] = az[0] = az[ny] = 0.0
    u = (az[1:] - az[:-1]) / hy - (ay.roll(-1, 1) - ay) / hz
    v = (ax[:ny].roll(-1, 1) - ax[:ny]) / hz - (az[:ny].roll(-1, 2) - az[:ny]) / hx
    w = (ay.roll(-1, 2) - ay) / hx - (ax[1:] - ax[:-1]) / hy
    v[0] = 0.0
    s = torch.sqrt(torch.mean(u * u + v * v + w * w) / 3)
    return [f / s for f in (u, v, w)]


def _markers(case, gen):
    """(X0 [n][3], dV [n]): a Fibonacci sphere, or for the heaving motion a plate normal to y."""
    n, h = case["markers"], _spacings(case)
    ly = case["ny"] * h[1]
    shift = 0.02 * torch.rand(3, generator=gen, device=_device(), dtype=torch.float64)
    i = torch.arange(n, device=_device(), dtype=torch.float64)
    if case.get("motion") == HEAVE:
        span = min(2.0, 2.5 * h[2] * case["nz"] / 4)
        chord = 1.0
        ns = max(1, int(round(math.sqrt(n * span / chord))))
        nc = -(-n // ns)
        x = math.pi - 0.5 * chord + (torch.div(i, ns, rounding_mode="floor") + 0.5) / nc * chord
        z = 0.5 * h[2] * case["nz"] - 0.5 * span + (i % ns + 0.5) / ns * span
        X = torch.stack([x, torch.full_like(x, 0.5 * ly), z], 1)
        dV = torch.full_like(x, chord * span / n * h[1])
    else:
        r = 0.25
        q = 1 - 2 * (i + 0.5) / n
        rad, th = torch.sqrt(1 - q * q), math.pi * (3 - math.sqrt(5.0)) * i
        X = torch.stack([math.pi + r * rad * torch.cos(th), 0.5 * ly + r * q, math.pi + r * rad * torch.sin(th)], 1)
        dV = torch.full_like(q, 4 * math.pi * r * r / n * min(h))
    return X + shift - 0.01, dV


def _motion(case):
    """(params, velocity scale): the marker motion's four parameters."""
    if case["motion"] == TRANSLATE:
        return (0.1, 0.0, 0.0, 0.0)
    if case["motion"] == HEAVE:  # within the box, whatever its height
        ly = case["ny"] * _spacings(case)[1]
        return (min(0.5, 0.2 * ly), 1.0, 0.0, 0.0)
    return (0.0, 0.0, 0.0, 0.0)


DT, NU = 5e-4, 1e-2  # time step and viscosity of the step cases
HELMHOLTZ_C = 5e-5   # beta dt / Re of a viscous solve


def _inputs(case, seed):
    """The case's inputs, rounded to its precision: a dict of device tensors."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        got = {"rhs%d" % i: _rhs(n, n, n, gen) for i, n in enumerate(_cubes(case))}
    elif kind in ("poisson", "helmholtz"):
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        got = {"rhs": _rhs(nx, ny, nz, gen)}
        if case.get("walls"):
            got["lo"], got["hi"] = (_noise((1, nz, nx), min(nx, nz) / 4, -1.0, gen)[0] for _ in range(2))
    else:
        u, v, w = _velocity(case, gen)
        X0, dV = _markers(case, gen)
        got = {"u": u, "v": v, "w": w, "X0": X0, "dV": dV}
        if kind == "step":
            shape = tuple(u.shape)
            got["p"] = 0.1 * _noise(shape, min(shape) / 4, -1.0, gen)
            if case.get("inout"):
                # a through-flow at the inflow speed with an outlet close to it
                plane = (1,) + shape[1:]
                got["v"] = v + 0.5
                for k, mean in (("u_out", 0.0), ("v_out", 0.5), ("w_out", 0.0)):
                    got[k] = mean + 0.05 * _noise(plane, min(plane[1:]) / 4, -1.0, gen)[0]
        else:
            got["F"] = torch.randn((case["markers"], 3), generator=gen, device=_device(), dtype=torch.float64)
    return {k: t.to(_real(case)).contiguous() for k, t in got.items()}


def _cubes(case):
    return [int(n) for n in case["cubes"].split(",")]


# ---------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------

class _Handle:
    """Owns a plan or a batch."""

    def __init__(self, value, destroy):
        self.value, self.destroy = value, destroy

    def __del__(self):
        self.destroy(self.value)


def _plan(case):
    prec = ibm.IBM_FP64 if case["dtype"] == "f64" else ibm.IBM_FP32_REFINED
    bc = ibm.IBM_BC_TRIPLY_PERIODIC if case.get("periodic") else ibm.IBM_BC_PXZ_WALL_Y
    return _Handle(ibm.ibm_plan_create(case["nx"], case["ny"], case["nz"], _spacings(case), prec,
                                       case.get("refine", 0), bc), ibm.ibm_plan_destroy)


def prepare(case, seed):
    s = {"case": case, "in": _inputs(case, seed)}
    kind, x = case["kind"], s["in"]
    if kind == "batch":
        cubes = _cubes(case)
        prec = ibm.IBM_FP64 if case["dtype"] == "f64" else ibm.IBM_FP32_REFINED
        s["batch"] = _Handle(ibm.ibm_batch_create([(n, n, n) for n in cubes],
                                                  [(2 * math.pi / n, 2.0 / n, 2 * math.pi / n) for n in cubes], prec,
                                                  case["refine"]), ibm.ibm_batch_destroy)
        s["rhs"] = [x["rhs%d" % i] for i in range(len(cubes))]
        s["out"] = [torch.empty_like(t) for t in s["rhs"]]
        return s
    s["plan"] = _plan(case)
    if kind in ("poisson", "helmholtz"):
        s["out"] = torch.empty_like(x["rhs"])
    elif kind == "markers":
        if case.get("peskin"):
            ibm.ibm_plan_set_delta(s["plan"].value, ibm.IBM_DELTA_PESKIN4)
        if case.get("gather"):
            ibm.ibm_plan_set_spread(s["plan"].value, ibm.IBM_SPREAD_GATHER)
        s["U"] = torch.empty_like(x["X0"])
        s["f"] = [torch.empty_like(x[k]) for k in ("u", "v", "w")]
    else:
        s["N"] = [torch.zeros_like(x["u"]) for _ in range(3)]
        s["X"], s["Ud"], s["F"] = (torch.empty_like(x["X0"]) for _ in range(3))
        s["state"] = ibm.ibm_state(*[t.data_ptr() for t in (x["u"], x["v"], x["w"], x["p"], *s["N"])], 0.0)
        s["mk"] = ibm.ibm_markers(case["markers"], x["X0"].data_ptr(), x["dV"].data_ptr(), s["X"].data_ptr(),
                                  s["Ud"].data_ptr(), s["F"].data_ptr(), case["motion"],
                                  (ctypes.c_double * 4)(*_motion(case)))
        if case.get("inout"):
            s["io"] = ibm.ibm_inout(0.5, 0.5, *[x[k].data_ptr() for k in ("u_out", "v_out", "w_out")])
    return s


def run(s):
    case, x = s["case"], s["in"]
    kind = case["kind"]
    if kind == "batch":
        ibm.ibm_batch_poisson(s["batch"].value, s["rhs"], s["out"])
        return s["out"]
    plan = s["plan"].value
    if kind == "poisson":
        ibm.ibm_poisson_solve(plan, x["rhs"], s["out"])
        return s["out"]
    if kind == "helmholtz":
        field = ibm.IBM_FIELD_PERIODIC if case.get("periodic") else case["field"]
        if case.get("walls"):
            ibm.ibm_helmholtz_solve_bc(plan, HELMHOLTZ_C, field, x["rhs"], s["out"], x["lo"], x["hi"])
        else:
            ibm.ibm_helmholtz_solve(plan, HELMHOLTZ_C, field, x["rhs"], s["out"])
        return s["out"]
    if kind == "markers":
        ibm.ibm_interp(plan, case["markers"], x["X0"], x["u"], x["v"], x["w"], s["U"])
        for f in s["f"]:
            f.zero_()
        ibm.ibm_spread(plan, case["markers"], x["X0"], x["F"], x["dV"], *s["f"])
        return {"U": s["U"], "f": s["f"]}
    for stage in (1, 2, 3):
        if case.get("inout"):
            ibm.ibm_substep_inout(plan, s["state"], s["io"], stage, DT, NU, s["mk"])
        else:
            ibm.ibm_substep(plan, s["state"], stage, DT, NU, s["mk"])
    out = {"u": x["u"], "v": x["v"], "w": x["w"], "p": x["p"], "N": s["N"], "X": s["X"], "Ud": s["Ud"], "F": s["F"]}
    if case.get("inout"):
        out["outlet"] = [x[k] for k in ("u_out", "v_out", "w_out")]
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    size = 8 if case["dtype"] == "f64" else 4
    kind = case["kind"]

    def solve_flops(nx, ny, nz, periodic=False):
        axes = math.log2(nx * nz) + (math.log2(ny) if periodic else 0)
        return nx * ny * nz * (2 * 2.5 * axes + 10)

    if kind == "batch":
        cubes = _cubes(case)
        return {"bytes": sum(2 * size * n ** 3 for n in cubes),
                "flops": sum((1 + case["refine"]) * solve_flops(n, n, n) for n in cubes)}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    pts, nm = nx * ny * nz, case.get("markers", 0)
    support = 64 if case.get("peskin") else 27
    if kind in ("poisson", "helmholtz"):
        return {"bytes": 2 * size * pts, "flops": (1 + case["refine"]) * solve_flops(nx, ny, nz, case.get("periodic"))}
    if kind == "markers":
        # reads of the touched grid points are bounded by the fields and by the stencils
        touched = min(3 * pts, 3 * support * nm)
        return {"bytes": size * (touched + 3 * pts + touched + 13 * nm), "flops": 3 * nm * support * 4}
    # each stage reads and writes the velocity, the pressure and the advection terms
    return {"bytes": 3 * 14 * size * pts,
            "flops": 3 * ((4 + case["refine"]) * solve_flops(nx, ny, nz) + 150 * pts + 3 * nm * support * 4)}


def tolerance(case):
    """About four times the errors seen against exact() (and, where atomics order the sums, between two runs)."""
    if case["dtype"] == "f64":
        return {"rel": 4e-12, "max": 4e-10}  # solves 3e-14, steps 1.4e-13 (p), more on thin grids
    if case["kind"] == "markers":
        return {"rel": 1e-6, "max": 1.2e-4}  # 2.4e-7; two runs of the atomic sums differ by 3e-5 at a point
    if case["kind"] == "step":
        # u 7e-8, p and the advection term 1.2e-6 (a difference of FP32 fluxes over h: more on smooth fields)
        return {"rel": 1e-5, "max": 5e-4}
    if case["refine"] == 0:
        return {"rel": 4e-6, "max": 4e-5}  # FP32 transforms and sweeps alone: 1e-6
    return {"rel": 4e-7, "max": 4e-6}  # refined: 3e-8 to 5e-8


# ---------------------------------------------------------------------------
# the same results in plain FP64
# ---------------------------------------------------------------------------

def _eigenvalues(n, h):
    k = torch.arange(n, device=_device(), dtype=torch.float64)
    return 2 / (h * h) * (1 - torch.cos(2 * math.pi * k / n))


def _wall_basis(ny, hy, field):
    """Orthonormal eigenvectors (columns) and eigenvalues of -d2/dy2 with the field's homogeneous wall rows."""
    if field == FACE_DIRICHLET:
        j, k = (torch.arange(1, ny, device=_device(), dtype=torch.float64) for _ in range(2))
        Q, angle = torch.sin(math.pi * j[:, None] * k[None, :] / ny), math.pi * k / ny
    else:
        j, k = (torch.arange(ny, device=_device(), dtype=torch.float64) for _ in range(2))
        if field == CELL_DIRICHLET:
            Q, angle = torch.sin(math.pi * (j[:, None] + 0.5) * (k[None, :] + 1) / ny), math.pi * (k + 1) / ny
        else:
            Q, angle = torch.cos(math.pi * (j[:, None] + 0.5) * k[None, :] / ny), math.pi * k / ny
    return Q / torch.linalg.norm(Q, dim=0), 2 / (hy * hy) * (1 - torch.cos(angle))


def _solve(b, h, sigma, tau, field, periodic=False):
    """x of sigma x + tau L x = b; the constant mode is set to 0 where the operator is singular."""
    ny, nz, nx = b.shape
    first = 1 if field == FACE_DIRICHLET and not periodic else 0
    f = torch.fft.rfft2(b[first:], dim=(1, 2))
    lam = _eigenvalues(nz, h[2])[:, None] + _eigenvalues(nx, h[0])[None, : nx // 2 + 1]
    if periodic:
        f = torch.fft.fft(f, dim=0)
        ly = _eigenvalues(ny, h[1])
    else:
        Q, ly = _wall_basis(ny, h[1], field)
        f = torch.view_as_complex((Q.T @ torch.view_as_real(f).reshape(len(Q), -1)).reshape(*f.shape, 2))
    for j in range(len(ly)):  # plane by plane: no array of eigenvalues
        d = sigma - tau * (lam + ly[j])
        if sigma == 0 and j == 0:
            d[0, 0] = 1.0
            f[0, 0, 0] = 0.0
        f[j] /= d
    if periodic:
        f = torch.fft.ifft(f, dim=0)
    else:
        f = torch.view_as_complex((Q @ torch.view_as_real(f.contiguous()).reshape(len(Q), -1)).reshape(*f.shape, 2))
    x = torch.zeros_like(b)
    x[first:] = torch.fft.irfft2(f, s=(nz, nx), dim=(1, 2))
    return x


def _laplacian(f, h, field, lo=0.0, hi=0.0):
    """L f with the field's ghost values from the wall data lo, hi (values at the walls; Neumann: slopes)."""
    ny = f.shape[0]
    r = (f.roll(-1, 2) - 2 * f + f.roll(1, 2)) / h[0] ** 2 + (f.roll(-1, 1) - 2 * f + f.roll(1, 1)) / h[2] ** 2
    up, dn = f.roll(-1, 0), f.roll(1, 0)
    if field == CELL_NEUMANN:
        dn[0], up[ny - 1] = f[0] - h[1] * lo, f[ny - 1] + h[1] * hi
    elif field == CELL_DIRICHLET:
        dn[0], up[ny - 1] = 2 * lo - f[0], 2 * hi - f[ny - 1]
    else:
        dn[1], up[ny - 1] = lo, hi
    r += (up - 2 * f + dn) / h[1] ** 2
    if field == FACE_DIRICHLET:
        r[0] = 0.0
    return r


def _helmholtz(b, h, c, field, lo=0.0, hi=0.0):
    """x of (I - c L) x = b with wall data: the data's share of L x goes to the right-hand side."""
    share = _laplacian(torch.zeros_like(b), h, field, lo, hi)
    x = _solve(b + c * share, h, 1.0, -c, field)
    if field == FACE_DIRICHLET:
        x[0] = lo
    return x


def _delta(r, peskin):
    a = r.abs()
    if peskin:
        near = (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp(min=0))) / 8
        far = (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp(min=0))) / 8
        return torch.where(a <= 1, near, torch.where(a <= 2, far, torch.zeros_like(a)))
    near = (1 + torch.sqrt((1 - 3 * a * a).clamp(min=0))) / 3
    far = (5 - 3 * a - torch.sqrt((1 - 3 * (1 - a) ** 2).clamp(min=0))) / 6
    return torch.where(a <= 0.5, near, torch.where(a <= 1.5, far, torch.zeros_like(a)))


def _stencil(X, case, comp, peskin):
    """For each marker the flat indexes and weights of component comp's stencil."""
    h, n = _spacings(case), (case["nx"], case["ny"], case["nz"])
    size = 4 if peskin else 3
    at, wt = [], []
    for ax in range(3):
        s = X[:, ax] / h[ax] - (0.0 if ax == comp else 0.5)
        base = torch.floor(s) - 1 if peskin else torch.floor(s + 0.5) - 1
        q = base[:, None] + torch.arange(size, device=X.device, dtype=torch.float64)
        wt.append(_delta(s[:, None] - q, peskin))
        at.append(q.long().clamp(0, n[1] - 1) if ax == 1 else q.long() % n[ax])
    idx = (at[1][:, :, None, None] * n[2] + at[2][:, None, :, None]) * n[0] + at[0][:, None, None, :]
    w = wt[1][:, :, None, None] * wt[2][:, None, :, None] * wt[0][:, None, None, :]
    return idx.reshape(len(X), -1), w.reshape(len(X), -1)


def _interp(X, fields, case, peskin=False):
    out = []
    for comp in range(3):
        idx, w = _stencil(X, case, comp, peskin)
        out.append((fields[comp].reshape(-1)[idx] * w).sum(1))
    return torch.stack(out, 1)


def _spread(X, F, dV, case, peskin=False):
    h = _spacings(case)
    out = []
    for comp in range(3):
        idx, w = _stencil(X, case, comp, peskin)
        f = torch.zeros(case["nx"] * case["ny"] * case["nz"], device=X.device, dtype=torch.float64)
        f.index_add_(0, idx.reshape(-1), (w * (F[:, comp] * dV / (h[0] * h[1] * h[2]))[:, None]).reshape(-1))
        out.append(f.reshape(case["ny"], case["nz"], case["nx"]))
    return out


def _advection(u, v, w, h, v_lo, top):
    """div(u u) on the staggered grid; top: (u, v, w) at the upper wall (planes or 0), below: v = v_lo, u = w = 0."""
    ny = u.shape[0]
    vn = v.roll(-1, 0)  # v on the upper face of each cell
    vn[ny - 1] = top[1]

    def at_faces(f, value_top):  # tangential component on the y faces j = 0 .. ny
        g = torch.zeros((ny + 1,) + tuple(f.shape[1:]), device=f.device, dtype=f.dtype)
        g[1:ny] = 0.5 * (f[:-1] + f[1:])
        g[ny] = value_top
        return g

    vf = torch.cat([v, vn[ny - 1:]])  # v on the y faces 0 .. ny
    # u: x-faces
    uc = 0.5 * (u + u.roll(-1, 2))
    nu = (uc ** 2 - uc.roll(1, 2) ** 2) / h[0]
    q = at_faces(u, top[0]) * 0.5 * (vf + vf.roll(1, 2))
    nu = nu + (q[1:] - q[:-1]) / h[1]
    q = 0.5 * (u + u.roll(1, 1)) * 0.5 * (w + w.roll(1, 2))
    nu = nu + (q.roll(-1, 1) - q) / h[2]
    # w: z-faces
    wc = 0.5 * (w + w.roll(-1, 1))
    nw = (wc ** 2 - wc.roll(1, 1) ** 2) / h[2]
    q = at_faces(w, top[2]) * 0.5 * (vf + vf.roll(1, 1))
    nw = nw + (q[1:] - q[:-1]) / h[1]
    q = 0.5 * (w + w.roll(1, 2)) * 0.5 * (u + u.roll(1, 1))
    nw = nw + (q.roll(-1, 2) - q) / h[0]
    # v: y-faces 1 .. ny-1
    vc = 0.5 * (v + vn)
    nv = torch.zeros_like(v)
    nv[1:] = (vc[1:] ** 2 - vc[:-1] ** 2) / h[1]
    q = 0.5 * (v[1:] + v[1:].roll(1, 2)) * 0.5 * (u[1:] + u[:-1])
    nv[1:] += (q.roll(-1, 2) - q) / h[0]
    q = 0.5 * (v[1:] + v[1:].roll(1, 1)) * 0.5 * (w[1:] + w[:-1])
    nv[1:] += (q.roll(-1, 1) - q) / h[2]
    return [nu, nv, nw]


def _gradient(p, h):
    gy = (p - p.roll(1, 0)) / h[1]
    gy[0] = 0.0
    return [(p - p.roll(1, 2)) / h[0], gy, (p - p.roll(1, 1)) / h[2]]


def _place(case, X0, t):
    """Marker positions and velocities at time t."""
    a, period = _motion(case)[:2]
    d, vel = torch.zeros(3, dtype=torch.float64), torch.zeros(3, dtype=torch.float64)
    if case["motion"] == TRANSLATE:
        vel = torch.tensor(_motion(case)[:3], dtype=torch.float64)
        d = vel * t
    elif case["motion"] == HEAVE:
        d[1] = a * math.sin(2 * math.pi * t / period)
        vel[1] = a * 2 * math.pi / period * math.cos(2 * math.pi * t / period)
    return X0 + d.to(X0), vel.to(X0).expand_as(X0).contiguous()


def _exact_step(case, x):
    h, dt, nu = _spacings(case), DT, NU
    bcs = (CELL_DIRICHLET, FACE_DIRICHLET, CELL_DIRICHLET)
    vel, p, N, t = [x["u"], x["v"], x["w"]], x["p"], [torch.zeros_like(x["u"]) for _ in range(3)], 0.0
    io = case.get("inout")
    v_in, c_out = (0.5, 0.5) if io else (0.0, 0.0)
    out = [x[k] for k in ("u_out", "v_out", "w_out")] if io else [0.0, 0.0, 0.0]
    for n in range(3):
        a = b = ALPHA[n]
        ab = a + b
        if io:
            near = (0.5 * h[1], h[1], 0.5 * h[1])
            out = [out[c] - ab * dt * c_out / near[c] * (out[c] - vel[c][-1]) for c in range(3)]
            out[1] = out[1] + (v_in - out[1].mean())
            vel[1] = vel[1].clone()
            vel[1][0] = v_in
        lo = (0.0, v_in, 0.0)
        lap = [_laplacian(vel[c], h, bcs[c], lo[c], out[c]) for c in range(3)]
        adv, G = _advection(*vel, h, v_in, out), _gradient(p, h)
        est = [vel[c] + dt * (ab * nu * lap[c] - ab * G[c] - GAMMA[n] * adv[c] - ZETA[n] * N[c]) for c in range(3)]
        est[1][0] = v_in
        X, Ud = _place(case, x["X0"], t)
        F = (Ud - _interp(X, est, case)) / dt
        f = _spread(X, F, x["dV"], case)
        c_visc = b * dt * nu
        star = [_helmholtz(est[c] - c_visc * lap[c] + dt * f[c], h, c_visc, bcs[c], lo[c], out[c]) for c in range(3)]
        del est, f, lap, G
        us, vs, ws = star
        vn = vs.roll(-1, 0)
        vn[-1] = out[1]
        div = (us.roll(-1, 2) - us) / h[0] + (vn - vs) / h[1] + (ws.roll(-1, 1) - ws) / h[2]
        phi = _solve(div / (ab * dt), h, 0.0, 1.0, CELL_NEUMANN)
        G = _gradient(phi, h)
        vel = [star[c] - ab * dt * G[c] for c in range(3)]
        vel[1][0] = v_in
        p = p + phi - c_visc * _laplacian(phi, h, CELL_NEUMANN)
        N, t = adv, t + ab * dt
    got = {"u": vel[0], "v": vel[1], "w": vel[2], "p": p, "N": N, "X": X, "Ud": Ud, "F": F}
    if io:
        got["outlet"] = out
    return got


def exact(case, seed):
    x = {k: t.double() for k, t in _inputs(case, seed).items()}
    kind = case["kind"]
    if kind == "batch":
        return [_solve(x["rhs%d" % i], (2 * math.pi / n, 2.0 / n, 2 * math.pi / n), 0.0, 1.0, CELL_NEUMANN)
                for i, n in enumerate(_cubes(case))]
    h = _spacings(case)
    if kind == "poisson":
        return _solve(x["rhs"], h, 0.0, 1.0, CELL_NEUMANN, case.get("periodic", False))
    if kind == "helmholtz":
        if case.get("periodic"):
            return _solve(x["rhs"], h, 1.0, -HELMHOLTZ_C, CELL_NEUMANN, True)
        return _helmholtz(x["rhs"], h, HELMHOLTZ_C, case["field"], x.get("lo", 0.0), x.get("hi", 0.0))
    if kind == "markers":
        peskin = bool(case.get("peskin"))
        return {"U": _interp(x["X0"], [x["u"], x["v"], x["w"]], case, peskin),
                "f": _spread(x["X0"], x["F"], x["dV"], case, peskin)}
    return _exact_step(case, x)
