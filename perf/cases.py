"""The work that users of this framework have it do, as cases to be timed and compared.

A case is a dict of plain values; its "kind" says which entry points one pass takes:

  eval      OrbitalSplines.eval_vgl into the caller's buffers (every basis, storage type, real
            and Bloch orbitals): the inner call of a quantum Monte Carlo step
  autograd  evaluate() and the gradients of its three outputs with respect to the positions and
            the coefficient tables: one step of an orbital optimisation
  backward  OrbitalSplines.backward for a whole walker population: forces and the coefficient
            gradient, into the caller's buffers
  slater    slater_kinetic: log-determinants, local kinetic energy and drift of every walker
  batch     eval_batched: several cells with different grids and orbital counts in one call

Orbitals are seeded synthetic planewave sets (spherical cutoff, Gaussian envelope, Hermitian for
real orbitals), positions are uniform in the cell, upstream weights N(0, 1).  exact() restates
every path in 64-bit torch: tables from a plain FFT, the stencil sums written out, determinants
from torch.linalg.
"""
import functools
import math

import numpy as np
import torch

from paper_1309_6250_gb300.api import OrbitalSplines, eval_batched, slater_kinetic
from paper_1309_6250_gb300.autograd import evaluate


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# --------------------------------------------------------------------------------- the cases

def _orbital_case(kind, name=None, **kw):
    c = dict(kind=kind, method="smooth", storage="f32", lap_table=True, grad_tables=False, degree=3, bloch=False,
             skew=0.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one walker of the 8-atom silicon cell moves all its electrons: the smallest call
        _orbital_case("eval", "one_walker_si8", nx=48, ny=48, nz=48, orb=16, a=10.26, ecut=15.0, decay=4.0, pos=32),
        # the double-precision interpolating spline with the Laplacian from second derivatives
        _orbital_case("eval", "interp_f64_16", nx=16, ny=16, nz=16, orb=8, a=10.26, ecut=15.0, decay=4.0, pos=1000,
                      method="interp", storage="f64", lap_table=False),
        # 1,024 walkers of the 8-atom silicon cell: an ordinary step, tables inside L2
        _orbital_case("eval", "step_si8", nx=48, ny=48, nz=48, orb=16, a=10.26, ecut=15.0, decay=4.0, pos=32768),
        # 2,048 walkers of the 64-atom MgO cell: the benchmark's step, the largest case
        _orbital_case("eval", "step_mgo64", nx=96, ny=96, nz=96, orb=128, a=15.9, ecut=40.0, decay=8.0, pos=524288),
        # 16-bit tables at odd sizes: skewed cell, unequal grid, orbital and position counts that fill nothing
        _orbital_case("eval", "ragged_bf16", nx=80, ny=72, nz=90, orb=109, a=15.3, ecut=15.0, decay=4.0, pos=200003,
                      storage="bf16", skew=0.12),
        # double-float tables (near double precision without the FP64 pipe), 64-atom silicon cell
        _orbital_case("eval", "step_si64_df64", nx=72, ny=72, nz=72, orb=128, a=20.52, ecut=15.0, decay=4.0, pos=65536,
                      storage="df64"),
        # the paper's most accurate form: separate tables of the gradient and the Laplacian (five tables)
        _orbital_case("eval", "five_tables", nx=64, ny=64, nz=64, orb=96, a=15.3, ecut=15.0, decay=4.0, pos=98304,
                      grad_tables=True),
        # complex orbitals at a zone-boundary k point
        _orbital_case("eval", "bloch_mgo64", nx=96, ny=96, nz=96, orb=64, a=15.9, ecut=40.0, decay=8.0, pos=131072,
                      bloch=True),
        # orbital optimisation through torch.autograd: forward and both adjoints
        _orbital_case("autograd", "autograd_si64", nx=72, ny=72, nz=72, orb=128, a=20.52, ecut=15.0, decay=4.0, pos=4096),
        # both adjoints for a walker population
        _orbital_case("backward", "backward_mgo64", nx=96, ny=96, nz=96, orb=128, a=15.9, ecut=40.0, decay=8.0,
                      pos=262144),
        # Slater determinants of the MgO step: 2,048 walkers x (128 up + 128 down)
        dict(name="slater_mgo64", kind="slater", walkers=2048, n_up=128, n_dn=128, orb=128, bloch=False, a=15.9),
        # three uneven cells (aluminium, silicon, MgO like) in one call: orbitals x grid x positions each
        dict(name="batch_three_cells", kind="batch", cells="48x64x49152,128x80x262144,32x64x131072", storage="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.15:
        bloch = rng.random() < 0.5
        up = _log_int(rng, 4, 96 if bloch else 144)
        dn = max(1, up - rng.randint(0, 3))
        cost = (up ** 3 + dn ** 3) * (4 if bloch else 1)
        walkers = _log_int(rng, 16, max(32, min(4096, 2048 * 2 * 128 ** 3 // cost)))
        return dict(kind="slater", walkers=walkers, n_up=up, n_dn=dn, orb=max(up, dn) + rng.randint(0, 4), bloch=bloch,
                    a=rng.choice([10.26, 15.9, 20.52]))
    if u < 0.23:
        cells = []
        for _ in range(rng.randint(2, 4)):
            cells.append("%dx%dx%d" % (rng.randint(8, 128), rng.choice([32, 45, 48, 64, 72, 80]), _log_int(rng, 64, 131072)))
        return dict(kind="batch", cells=",".join(cells), storage=rng.choice(["f32", "f32", "bf16"]))
    kind = "eval" if u < 0.85 else rng.choice(["autograd", "backward"])
    bloch = rng.random() < 0.2
    orb = _log_int(rng, 6, 80 if bloch else 160)
    nx = _log_int(rng, 16, 96)
    ny, nz = (min(96, max(12, nx + rng.randint(-6, 6))) for _ in range(2))
    storage = rng.choice(["f32"] * 5 + ["bf16"] * 3 + ["df64", "f64"])
    form = rng.choice(["lap"] * 6 + ["hessian"] * 3 + ["grad", "lagrange", "pp", "degree"])
    if storage == "df64" and form not in ("lap", "hessian", "grad"):
        form = "lap"
    if kind != "eval" and (storage == "df64" or form in ("grad", "lagrange", "pp", "degree")):
        storage, form = "f32", "lap"
    funs = orb * (2 if bloch else 1)
    evals = {"f32": 67e6, "bf16": 67e6, "df64": 8e6, "f64": 4e6}[storage] / (1 if kind == "eval" else 3)
    if form in ("grad", "lagrange", "degree"):
        evals /= 5
    hi = max(64, min(524288 if kind == "eval" else 262144, int(evals / funs)))
    c = _orbital_case(kind, nx=nx, ny=ny, nz=nz, orb=orb, bloch=bloch, storage=storage, decay=4.0,
                      a=rng.choice([10.26, 15.3, 15.9, 20.52]), skew=rng.choice([0.0, 0.0, 0.1]), pos=_log_int(rng, 16, hi))
    # the planewaves fill half of the grid's band on small grids and a third of it on large ones
    c["ecut"] = round(0.5 * ((0.7 if nx <= 64 else 0.5) * math.pi * min(nx, ny, nz) / c["a"]) ** 2 * 0.5, 3)
    c["method"] = rng.choice(["smooth", "interp"])
    if form == "hessian":
        c["lap_table"] = False
    elif form == "grad":
        c["grad_tables"] = True
    elif form in ("lagrange", "pp"):
        c["method"] = form
    elif form == "degree":
        c["degree"] = rng.choice([1, 5])
    return c


# ------------------------------------------------------------------------------- the inputs

def _lattice(a, skew):
    """Columns are the lattice vectors; skew tilts the second and third of them."""
    m = np.eye(3) * a
    m[0, 1] = skew * a
    m[1, 2] = -0.5 * skew * a
    return m


_KPOINT = (0.5, 0.5, 0.5)


@functools.lru_cache(maxsize=16)
def _planewaves(a, skew, ecut, bloch):
    """Miller indices with |k + G|^2 / 2 <= ecut and |k + G|^2.  Real orbitals: a half space, its
    mirror image in the same order, G = 0 last."""
    lat = _lattice(a, skew)
    b = 2.0 * math.pi * np.linalg.inv(lat).T
    k = np.asarray(_KPOINT if bloch else (0.0, 0.0, 0.0))
    m = [int(math.sqrt(2.0 * ecut) * np.linalg.norm(lat[:, i]) / (2.0 * math.pi)) + 2 for i in range(3)]
    n = np.stack(np.meshgrid(*[np.arange(-x, x + 1) for x in m], indexing="ij"), axis=-1).reshape(-1, 3)
    g2 = (((n + k) @ b.T) ** 2).sum(1)
    n, g2 = n[0.5 * g2 <= ecut], g2[0.5 * g2 <= ecut]
    if not bloch:
        half = (n[:, 0] > 0) | ((n[:, 0] == 0) & (n[:, 1] > 0)) | ((n[:, 0] == 0) & (n[:, 1] == 0) & (n[:, 2] > 0))
        n, g2 = np.concatenate([n[half], -n[half], np.zeros((1, 3), n.dtype)]), np.concatenate([g2[half], g2[half], [0.0]])
    return np.ascontiguousarray(n.astype(np.int32)), g2


def _coefficients(a, skew, ecut, decay, bloch, orb, seed):
    n, g2 = _planewaves(a, skew, ecut, bloch)
    rng = np.random.default_rng(seed)
    env = np.exp(-g2 / decay) / math.sqrt(2.0)
    if bloch:
        return n, (rng.standard_normal((orb, len(n), 2)).view(np.complex128)[..., 0]) * env
    h = (len(n) - 1) // 2
    c = np.empty((orb, len(n)), np.complex128)
    c[:, :h] = rng.standard_normal((orb, h, 2)).view(np.complex128)[..., 0] * env[:h]
    np.conjugate(c[:, :h], out=c[:, h:2 * h])
    c[:, -1] = rng.standard_normal(orb)
    return n, c


def _positions(lat, n, seed):
    s = np.random.default_rng(seed).random((n, 3))
    return torch.from_numpy(np.ascontiguousarray(s @ lat.T)).to(_dev())


def _upstream(case, seed):
    g = torch.Generator(device=_dev()).manual_seed(seed)
    real = torch.float64 if case["storage"] in ("f64", "df64") else torch.float32
    dt = {torch.float32: torch.complex64, torch.float64: torch.complex128}[real] if case["bloch"] else real
    p, o = case["pos"], case["orb"]
    return tuple(torch.randn(s, generator=g, dtype=dt, device=_dev()) for s in ((p, o), (p, 3, o), (p, o)))


def _orbital_inputs(case, seed):
    lat = _lattice(case["a"], case["skew"])
    n, c = _coefficients(case["a"], case["skew"], case["ecut"], case["decay"], case["bloch"], case["orb"], [seed, 1])
    return lat, n, c, _positions(lat, case["pos"], [seed, 2])


def _cells(case):
    """The cells of a batch: (orbitals, grid, positions, lattice constant, cutoff)."""
    out = []
    for t in case["cells"].split(","):
        orb, grid, pos = (int(x) for x in t.split("x"))
        out.append((orb, grid, pos, grid / 4.0, 15.0))
    return out


_SLATER_ECUT = 4.0


def _slater_inputs(case, seed):
    """Planewave orbitals of a walker population and their derivatives, in 32 bits (sums of
    planewaves written out): val [P, O], grad [P, 3, O], lap [P, O]."""
    lat = _lattice(case["a"], 0.0)
    ecut = max(_SLATER_ECUT, 0.5 * (2.0 * math.pi / case["a"]) ** 2 * (1.2 * case["orb"]) ** (2.0 / 3.0))
    n, c = _coefficients(case["a"], 0.0, ecut, 8.0, case["bloch"], case["orb"], [seed, 3])
    pos = _positions(lat, case["walkers"] * (case["n_up"] + case["n_dn"]), [seed, 4])
    k = np.asarray(_KPOINT if case["bloch"] else (0.0, 0.0, 0.0))
    if not case["bloch"]:   # c_G e^{iGr} + conj: twice the real part over a half space
        h = (len(n) - 1) // 2
        keep = np.r_[0:h, len(n) - 1]
        n, c = n[keep], c[:, keep] * np.r_[np.full(h, 2.0), 1.0]
    g = 2.0 * math.pi * (n + k) @ np.linalg.inv(lat)
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(_dev())  # noqa: E731
    re, im, gd, sd = d(c.real.T), d(c.imag.T), d(g), d((n + k) @ np.linalg.inv(lat))
    g2 = (gd * gd).sum(1, keepdim=True)
    P, O = len(pos), case["orb"]
    dt = torch.complex64 if case["bloch"] else torch.float32
    val, grad, lap = (torch.empty(s, dtype=dt, device=_dev()) for s in ((P, O), (P, 3, O), (P, O)))

    def sums(cos, sin, a, b):   # sum_G (a + i b) e^{i(k+G).r}
        r = cos @ a.float() - sin @ b.float()
        return torch.complex(r, sin @ a.float() + cos @ b.float()) if case["bloch"] else r

    for p0 in range(0, P, 65536):
        t = pos[p0:p0 + 65536] @ sd.T
        t = (2.0 * math.pi * (t - torch.round(t))).float()
        cos, sin = torch.cos(t), torch.sin(t)
        val[p0:p0 + 65536] = sums(cos, sin, re, im)
        lap[p0:p0 + 65536] = sums(cos, sin, -g2 * re, -g2 * im)
        for x in range(3):      # i G (a + i b) = -G b + i G a
            grad[p0:p0 + 65536, x] = sums(cos, sin, -gd[:, x:x + 1] * im, gd[:, x:x + 1] * re)
    return val, grad, lap


# ------------------------------------------------------------------------------ one pass

def _splines(case, lat, n, c):
    return OrbitalSplines(lat, (case["nx"], case["ny"], case["nz"]), n, c, method=case["method"], storage=case["storage"],
                          separate_lap=case["lap_table"], separate_grad=case["grad_tables"], degree=case["degree"],
                          kpoint=_KPOINT if case["bloch"] else None)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "slater":
        s["in"] = _slater_inputs(case, seed)
        return s
    if case["kind"] == "batch":
        s["splines"], s["pos"], s["out"] = [], [], []
        for i, (orb, grid, pos, a, ecut) in enumerate(_cells(case)):
            n, c = _coefficients(a, 0.0, ecut, 4.0, False, orb, [seed, 5, i])
            s["splines"].append(OrbitalSplines(_lattice(a, 0.0), (grid,) * 3, n, c, storage=case["storage"]))
            s["pos"].append(_positions(_lattice(a, 0.0), pos, [seed, 6, i]))
            s["out"].append(s["splines"][-1].alloc_outputs(pos))
        return s
    lat, n, c, s["pos"] = _orbital_inputs(case, seed)
    spl = s["spl"] = _splines(case, lat, n, c)
    if case["kind"] == "eval":
        s["out"] = spl.alloc_outputs(case["pos"])
        return s
    s["up"] = _upstream(case, seed)
    if case["kind"] == "autograd":
        s["pos"].requires_grad_(True)
        s["tables"] = [t for t in spl.coefficient_parameters() if t is not None]
    else:
        kw = dict(dtype=spl.out_dtype, device=_dev())
        s["dcoef"] = [torch.zeros(spl.coef_shape(), **kw) for _ in range(2 if case["lap_table"] else 1)]
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "eval":
        return state["spl"].eval_vgl(state["pos"], out=state["out"])
    if case["kind"] == "autograd":
        out = evaluate(state["spl"], state["pos"], *state["tables"])
        return list(out) + list(torch.autograd.grad(out, [state["pos"]] + state["tables"], grad_outputs=state["up"]))
    if case["kind"] == "backward":
        for t in state["dcoef"]:
            t.zero_()
        dpos = state["spl"].backward(state["pos"], *state["up"], *state["dcoef"])
        return [dpos] + state["dcoef"]
    if case["kind"] == "slater":
        return slater_kinetic(*state["in"], case["walkers"], case["n_up"] + case["n_dn"], case["n_up"])
    return eval_batched(state["splines"], state["pos"], outs=state["out"])


# ------------------------------------------------------------------------ what a pass needs

def _spline_work(case, adjoint):
    f = case["orb"] * (2 if case["bloch"] else 1)
    size = {"f64": 8, "df64": 8, "f32": 4, "bf16": 2}[case["storage"]]
    out = 8 if size == 8 else 4
    tables = 5 if case["grad_tables"] or case["method"] == "lagrange" else 8 if case["method"] == "pp" \
        else 2 if case["lap_table"] else 1
    points = 8 if case["method"] == "pp" else (case["degree"] + 1) ** 3
    grid = case["nx"] * case["ny"] * case["nz"]
    rows = grid * (1.0 - (1.0 - min(1.0, points / grid)) ** case["pos"])   # grid points that any stencil touches
    table = rows * tables * f * size
    # per function and position: the sums over z of each (x, y) column, then over the columns
    n = case["degree"] + 1
    mads = points * 8 * 4 if case["method"] == "pp" else tables * points + tables * n * n if tables == 5 \
        else 3 * points + 5 * n * n if tables == 2 else 3 * points + 7 * n * n
    b = 24.0 * case["pos"] + table
    fl = 2.0 * mads * case["pos"] * f
    if not adjoint:
        return b + 5.0 * case["pos"] * f * out, fl
    # upstream read, dL/dr written, each coefficient gradient written; about twice the arithmetic
    return b + 5.0 * case["pos"] * f * out + 24.0 * case["pos"] + tables * grid * f * out, 2.0 * fl


def work(case):
    if case["kind"] == "slater":
        c = 2 if case["bloch"] else 1
        p = case["walkers"] * (case["n_up"] + case["n_dn"])
        used = case["walkers"] * (case["n_up"] ** 2 + case["n_dn"] ** 2)
        return {"bytes": 5.0 * used * 4 * c + 24.0 * p * c + case["walkers"] * 8.0 * (1 + 2 * c),
                "flops": 2.0 * (4 if case["bloch"] else 1) * case["walkers"] * (case["n_up"] ** 3 + case["n_dn"] ** 3)}
    if case["kind"] == "batch":
        w = [_spline_work(_orbital_case("eval", nx=g, ny=g, nz=g, orb=o, pos=p, storage=case["storage"]), False)
             for o, g, p, _, _ in _cells(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if case["kind"] == "autograd":   # forward (outputs written), then the adjoint
        f, a = _spline_work(case, False), _spline_work(case, True)
        return {"bytes": f[0] + a[0], "flops": f[1] + a[1]}
    b, fl = _spline_work(case, case["kind"] == "backward")
    return {"bytes": b, "flops": fl}


# -------------------------------------------------------------- the same results in 64 bits

def _multipliers(kind, n, dims):
    """The basis' division in Fourier space: 1 / gamma (smoothing), or 1 / prod(1 + cos(th) / 2)
    (interpolating; periodic in n, so it may be applied before the folding)."""
    th = 2.0 * math.pi * n / np.asarray(dims)
    if kind == "smooth":
        return 1.0 / (1.5 * np.sinc(th / (2.0 * math.pi)) ** 4).prod(1)
    return 1.0 / (1.0 + 0.5 * np.cos(th)).prod(1)


def _table64(n, c, dims):
    """sum_G c_G e^{iG.r} on the grid, [N, O] complex."""
    dev, (nx, ny, nz) = _dev(), dims
    idx = torch.from_numpy(((n[:, 0] % nx) * ny + n[:, 1] % ny) * nz + n[:, 2] % nz).long().to(dev)
    out = torch.empty((nx * ny * nz, len(c)), dtype=torch.complex128, device=dev)
    for o in range(0, len(c), 16):
        grid = torch.zeros((len(c[o:o + 16]), nx * ny * nz), dtype=torch.complex128, device=dev)
        grid.index_add_(1, idx, torch.from_numpy(c[o:o + 16]).to(dev))
        out[:, o:o + 16] = torch.fft.ifftn(grid.view(-1, nx, ny, nz), dim=(1, 2, 3), norm="forward").reshape(len(grid), -1).T
    return out


def _weights64(t):
    """Cubic weights of offsets -1 .. 2 and their first three derivatives: [4][P, 4]."""
    s = 1.0 - t
    one = torch.ones_like(t)
    return [torch.stack(w, 1) for w in (
        (0.25 * s ** 3, 0.75 * t ** 3 - 1.5 * t ** 2 + 1.0, 0.75 * s ** 3 - 1.5 * s ** 2 + 1.0, 0.25 * t ** 3),
        (-0.75 * s ** 2, 2.25 * t ** 2 - 3.0 * t, -(2.25 * s ** 2 - 3.0 * s), 0.75 * t ** 2),
        (1.5 * s, 4.5 * t - 3.0, 4.5 * s - 3.0, 1.5 * t),
        (-1.5 * one, 4.5 * one, -4.5 * one, 1.5 * one))]


class _Stencil:
    """Cells, weights and flat grid indices of some positions."""

    def __init__(self, pos, lat, dims):
        self.dims = dims
        u = pos @ torch.from_numpy(np.linalg.inv(lat).T).to(pos.device)
        u = (u - torch.floor(u)) * torch.tensor(dims, dtype=torch.float64, device=pos.device)
        i = torch.floor(u)
        self.w = [_weights64(u[:, x] - i[:, x]) for x in range(3)]
        self.i = [i[:, x].long() for x in range(3)]

    def points(self):
        nx, ny, nz = self.dims
        for l in range(4):
            for m in range(4):
                col = ((self.i[0] + l - 1) % nx * ny + (self.i[1] + m - 1) % ny) * nz
                for n in range(4):
                    yield (l, m, n), col + (self.i[2] + n - 1) % nz

    def weight(self, pt, order):
        return (self.w[0][order[0]][:, pt[0]] * self.w[1][order[1]][:, pt[1]] * self.w[2][order[2]][:, pt[2]])[:, None]

    def sums(self, table, orders):
        """The stencil sum of `table` [N, F] with each of the derivative orders."""
        out = [torch.zeros((len(self.i[0]), table.shape[1]), dtype=table.dtype, device=table.device) for _ in orders]
        for pt, idx in self.points():
            rows = table[idx]
            for o, order in zip(out, orders):
                o.addcmul_(rows, self.weight(pt, order).to(rows.dtype))
        return out


_E = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
_add = lambda *t: tuple(sum(x) for x in zip(*t))  # noqa: E731


def _tables64(method, lat, n, c, dims, lap, grads, kpoint):
    """Value table, Laplacian table or None, gradient tables or None; real or complex [N, O]."""
    g = 2.0 * math.pi * (n + np.asarray(kpoint)) @ np.linalg.inv(lat)
    m = _multipliers(method, n, dims)
    out = [_table64(n, c * m, dims)]
    out.append(_table64(n, c * m * -(g * g).sum(1), dims) if lap else None)
    out.append([_table64(n, c * m * 1j * g[:, x], dims) for x in range(3)] if grads else None)
    if not any(kpoint):
        out = [out[0].real.contiguous(), None if out[1] is None else out[1].real.contiguous(),
               None if out[2] is None else [t.real.contiguous() for t in out[2]]]
    return out


def _eval64(tables, lat, dims, pos, kpoint, dtype):
    """val [P, O], grad [P, 3, O], lap [P, O] in 64 bits."""
    dev = pos.device
    val_t, lap_t, grad_t = tables
    j = torch.from_numpy(np.linalg.inv(lat) * np.asarray(dims)[:, None]).to(dev)   # dt_i / dr_a
    metric = j @ j.T
    k = torch.tensor([2.0 * math.pi * x for x in np.asarray(kpoint) @ np.linalg.inv(lat)], dtype=torch.float64, device=dev)
    P, O = len(pos), val_t.shape[1]
    val, lap = (torch.empty((P, O), dtype=dtype, device=dev) for _ in range(2))
    grad = torch.empty((P, 3, O), dtype=dtype, device=dev)
    step = max(1, (1 << 27) // (O * 16))
    for p0 in range(0, P, step):
        st = _Stencil(pos[p0:p0 + step], lat, dims)
        e = slice(p0, p0 + step)
        if grad_t is not None:
            v, = st.sums(val_t, [(0, 0, 0)])
            g = [st.sums(t, [(0, 0, 0)])[0] for t in grad_t]
        else:
            v, *gt = st.sums(val_t, [(0, 0, 0)] + _E)
            g = [sum(gt[i] * j[i, a] for i in range(3)) for a in range(3)]
        if lap_t is not None:
            q, = st.sums(lap_t, [(0, 0, 0)])
        else:
            pairs = [(a, b) for a in range(3) for b in range(a, 3)]
            h = st.sums(val_t, [_add(_E[a], _E[b]) for a, b in pairs])
            q = sum(x * metric[a, b] * (1.0 if a == b else 2.0) for x, (a, b) in zip(h, pairs))
            if any(kpoint):
                q = q + 2j * sum(k[a] * g[a] for a in range(3)) - (k @ k) * v
        if any(kpoint):
            if grad_t is None:
                g = [g[a] + 1j * k[a] * v for a in range(3)]
            ph = torch.exp(1j * (pos[p0:p0 + step] @ k))[:, None]
            v, g, q = v * ph, [x * ph for x in g], q * ph
        val[e], lap[e] = v, q
        for a in range(3):
            grad[e, a] = g[a]
        del v, g, q
    return val, grad, lap


def _backward64(tables, lat, dims, pos, up):
    """dL/dr [P, 3] and the gradients of the tables, real orbitals in 64 bits."""
    dev = pos.device
    val_t, lap_t, _ = tables
    j = torch.from_numpy(np.linalg.inv(lat) * np.asarray(dims)[:, None]).to(dev)
    metric = j @ j.T
    pairs = [(a, b) for a in range(3) for b in range(3)]
    dval = torch.zeros_like(val_t)
    dlap = None if lap_t is None else torch.zeros_like(lap_t)
    dpos = torch.empty((len(pos), 3), dtype=torch.float64, device=dev)
    step = max(1, (1 << 27) // (val_t.shape[1] * 16))
    for p0 in range(0, len(pos), step):
        e = slice(p0, p0 + step)
        st = _Stencil(pos[e], lat, dims)
        wv, wl = up[0][e].double(), up[2][e].double()
        wg = [up[1][e, a].double() for a in range(3)]
        gt = [sum(j[i, a] * wg[a] for a in range(3)) for i in range(3)]
        for pt, idx in st.points():
            v = wv * st.weight(pt, (0, 0, 0))
            for i in range(3):
                v.addcmul_(gt[i], st.weight(pt, _E[i]))
            if dlap is None:
                v.addcmul_(wl, sum(metric[a, b] * st.weight(pt, _add(_E[a], _E[b])) for a, b in pairs))
            else:
                dlap.index_add_(0, idx, wl * st.weight(pt, (0, 0, 0)))
            dval.index_add_(0, idx, v)
        u = torch.zeros((len(wv), 3), dtype=torch.float64, device=dev)
        terms = [(0, 0, 0)] + _E
        for i in range(3):
            parts = st.sums(val_t, [_add(_E[i], t) for t in terms])
            acc = parts[0] * wv + sum(x * y for x, y in zip(parts[1:], gt))
            if lap_t is None:
                h = st.sums(val_t, [_add(_E[i], _E[a], _E[b]) for a, b in pairs if a <= b])
                acc += wl * sum(x * metric[a, b] * (1.0 if a == b else 2.0)
                                for x, (a, b) in zip(h, [q for q in pairs if q[0] <= q[1]]))
            else:
                acc += wl * st.sums(lap_t, [_E[i]])[0]
            u[:, i] = acc.sum(1)
        dpos[e] = u @ j
    return [dpos, dval.view(*dims, -1)] + ([] if dlap is None else [dlap.view(*dims, -1)])


def _slater64(case, seed):
    val, grad, lap = _slater_inputs(case, seed)
    W, ne = case["walkers"], case["n_up"] + case["n_dn"]
    d = torch.complex128 if case["bloch"] else torch.float64
    logdet, sign = torch.zeros(W, dtype=torch.float64, device=_dev()), torch.ones(W, dtype=d, device=_dev())
    kin, drift = torch.zeros(W, dtype=d, device=_dev()), torch.empty((W, ne, 3), dtype=d, device=_dev())
    val, grad, lap = val.view(W, ne, -1), grad.view(W, ne, 3, -1), lap.view(W, ne, -1)
    for e0, n in ((0, case["n_up"]), (case["n_up"], case["n_dn"])):
        for w0 in range(0, W, 256):
            w = slice(w0, w0 + 256)
            a = val[w, e0:e0 + n, :n].to(d)
            x = torch.linalg.inv(a)
            x = x + x @ (torch.eye(n, dtype=d, device=_dev()) - a @ x)   # one refinement step
            s, ld = torch.linalg.slogdet(a)
            logdet[w] += ld.real
            sign[w] *= s
            kin[w] -= 0.5 * torch.einsum("wji,wij->w", x, lap[w, e0:e0 + n, :n].to(d))
            drift[w, e0:e0 + n] = torch.einsum("wji,wicj->wic", x, grad[w, e0:e0 + n, :, :n].to(d))
    return logdet, sign, kin, drift


def exact(case, seed):
    if case["kind"] == "slater":
        return _slater64(case, seed)
    if case["kind"] == "batch":
        out = []
        for i, (orb, grid, pos, a, ecut) in enumerate(_cells(case)):
            n, c = _coefficients(a, 0.0, ecut, 4.0, False, orb, [seed, 5, i])
            lat, dims = _lattice(a, 0.0), (grid,) * 3
            t = _tables64("smooth", lat, n, c, dims, True, False, (0, 0, 0))
            out.append(_eval64(t, lat, dims, _positions(lat, pos, [seed, 6, i]), (0, 0, 0), torch.float64))
        return out
    if case["degree"] != 3 or case["method"] not in ("smooth", "interp") or (case["kind"] != "eval" and case["bloch"]):
        return None
    lat, n, c, pos = _orbital_inputs(case, seed)
    dims = (case["nx"], case["ny"], case["nz"])
    k = _KPOINT if case["bloch"] else (0, 0, 0)
    tables = _tables64(case["method"], lat, n, c, dims, case["lap_table"], case["grad_tables"], k)
    d = torch.complex128 if case["bloch"] else torch.float64
    if case["kind"] == "eval":
        return _eval64(tables, lat, dims, pos, k, d)
    back = _backward64(tables, lat, dims, pos, _upstream(case, seed))
    return back if case["kind"] == "backward" else list(_eval64(tables, lat, dims, pos, k, d)) + back
