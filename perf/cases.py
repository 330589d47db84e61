"""What the solver is used for, as timed cases.

A case is one pass of work through the public entry points (``ehs.Solver`` / ``ehs.solver_for``
and ``autograd.solve``) on seeded synthetic media.  ``kind`` says which:

apply     K x and K_s x, the operator and its shifted form, which a program applies to form residuals
          of its own
cycle     one multigrid cycle of the shifted operator, the preconditioner of every iteration
solve     preconditioned FGMRES to a 1e-6 residual with a context the program keeps
fwi       one gradient of a frequency-domain inversion with a kept context: forward solves of all
          sources, receiver residual, adjoint solves, gradient with respect to the medium
autograd  the same gradient for a new medium, which is what every later step of an inversion and
          every new model pays for: ``autograd.solve`` builds the hierarchy, solves, and goes back

``exact`` restates the method in plain torch (complex128, assembled sparse operators); it shares no
code with the package.
"""
import math

import numpy as np
import torch

from paper_1806_11277_gb300 import autograd, ehs, synth

# coarsest inverses of the complex64 cycle by name (opts.coarse_fmt)
FMT = {"df": 0, "c64": 1, "fp16": 2, "bf16": 3}


def _case(name, kind, shape, **kw):
    """shape: (n_y, n_x) or (n_z, n_y, n_x).  split, overlap: subdomains per axis of the coarsest
    grid (1: exact coarsest solve).  dd: top-level subdomains per axis (1: none)."""
    c = dict(name=name, kind=kind, nz=shape[0] if len(shape) == 3 else 0, ny=shape[-2], nx=shape[-1], media=1, nrhs=1,
             levels=3, alpha=0.2, cycle=1, prec="c64", fmt="df", table16=0, split=1, overlap=2, dd=1)
    c.update(kw)
    return c


# the 16-bit storage and the 16x16-cell subdomains of the benchmark's MG-DD preconditioner
_MGDD = dict(fmt="fp16", table16=1, overlap=3)


def listed():
    return [
        # the smallest calls: what a call costs when there is next to nothing to compute
        _case("apply_64_c128", "apply", (64, 64), prec="c128"),
        _case("cycle_64", "cycle", (64, 64)),
        # one pass of the operator over a large model
        _case("apply_1024", "apply", (1024, 1024), levels=6, alpha=0.4),
        # W-cycle with the exact coarsest solve on a ragged grid (no power of two, no tile size)
        _case("cycle_200x344_w", "cycle", (200, 344), levels=4, alpha=0.4, cycle=2),
        # the plain FP64 form
        _case("cycle_256_c128", "cycle", (256, 256), levels=4, alpha=0.4, prec="c128"),
        _case("solve_64_c128", "solve", (64, 64), prec="c128"),
        # the preconditioner and the solve of the 512x512 benchmark, several media in a batch
        _case("cycle_512_mgdd", "cycle", (512, 512), split=8, **_MGDD),
        _case("solve_512_mgdd", "solve", (512, 512), media=2, split=8, **_MGDD),
        # the 16-source gradient of the benchmark's inversion line
        _case("fwi_256_16src", "fwi", (256, 256), nrhs=16, split=4, **_MGDD),
        # a gradient for a new medium (hierarchy setup included)
        _case("autograd_256", "autograd", (256, 256), nrhs=4, split=4, **_MGDD),
        # 3D: one hierarchy with complex64 storage, and overlapping subdomains with 16-bit storage
        _case("solve_64x64x64", "solve", (64, 64, 64), nrhs=2, levels=4, alpha=0.5, fmt="c64"),
        _case("solve_96x96x96_dd", "solve", (96, 96, 96), levels=4, alpha=0.5, dd=2, split=2, table16=1, fmt="fp16"),
    ]


def draw(rng):
    def logint(lo, hi, step):
        return step * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step))

    kind = rng.choice(["apply", "cycle", "cycle", "cycle", "solve", "solve", "fwi", "autograd"])
    prec = rng.choice(["c64", "c64", "c128"])
    if kind == "apply":
        shape = (logint(64, 1024, 32), logint(64, 1024, 32))
        # enough levels that the coarsest grid, which this case does not use, is small
        return _drawn("apply", shape, levels=6 if max(shape) > 512 and min(shape) >= 64 else 5, alpha=0.4, prec=prec,
                      media=rng.choice([1, 2]))
    if kind == "solve" and rng.random() < 0.35:
        shape = tuple(logint(24, 64, 8) for _ in range(3))
        return _drawn("solve", shape, levels=3 if min(shape) < 32 else 4, alpha=0.5, nrhs=rng.choice([1, 2]),
                      fmt=rng.choice(["c64", "fp16"]), table16=rng.choice([0, 1]), split=2, overlap=1)
    if rng.random() < 0.6:                # MG-DD: coarsest subdomains of 12 to 16 cells, 3 levels
        top = 6 if kind == "cycle" else 4
        split = rng.randint(2, top)
        cells = [split * rng.choice([12, 14, 16]) * 4 for _ in range(2)]
        return _drawn(kind, tuple(cells), nrhs=rng.choice([1, 3, 4]) if kind != "cycle" else 1, split=split,
                      media=rng.choice([1, 2]) if kind in ("cycle", "solve") and split < 4 else 1,
                      fmt=rng.choice(["c64", "fp16", "bf16"]), table16=rng.choice([0, 1, 2]), overlap=3)
    shape = (logint(64, 288, 8), logint(64, 288, 8))
    return _drawn(kind, shape, levels=4, alpha=0.4, cycle=rng.choice([1, 2]), prec=prec if kind == "cycle" else "c64",
                  nrhs=rng.choice([1, 2]), fmt=rng.choice(["df", "df", "c64", "fp16"]))


def _drawn(kind, shape, **kw):
    c = _case("", kind, shape, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _shape(c):
    return (c["nz"], c["ny"], c["nx"]) if c["nz"] else (c["ny"], c["nx"])


def _weights(c):
    return [0.5, 0.5, 0.2] if c["nz"] else [0.75, 0.5, 0.25, 0.25, 0.25]


def _options(c):
    d = 3 if c["nz"] else 2
    axes = lambda s: tuple(s if k < d else 1 for k in range(3))
    kw = dict(levels=c["levels"], alpha=c["alpha"], w=_weights(c), cycle=c["cycle"], nrhs=c["nrhs"],
              prec=ehs.EHS_C128 if c["prec"] == "c128" else ehs.EHS_C64, coarse_fmt=FMT[c["fmt"]],
              coef_half=c["table16"], coarse_dd=axes(c["split"]) if not c["nz"] else (c["split"], c["split"], 1),
              coarse_dd_overlap=c["overlap"])
    if c["dd"] > 1:
        kw.update(precond=ehs.EHS_PRECOND_DD, dd=axes(c["dd"]), dd_overlap=4, dd_pad=8)
    return kw


def _abl(c):
    return max(4, min(20, min(_shape(c)) // 10))


def _media(c, seed):
    """Smooth random media, wavelengths resolved by 8 points; 3D: perturbed layers."""
    shape = _shape(c)
    if c["nz"]:
        full = synth.layered_3d(n=max(shape), seed=seed, corr=10.0, abl=_abl(c))
        cut = tuple(slice(0, s) for s in shape)
        return [synth.Medium(full.lam[cut], full.mu[cut], full.rho[cut], full.omega, full.h, full.abl_cells)]
    sigmas = (0.25, 0.4, 0.45, 0.49)
    return [synth.random_2d(n=shape[0], nx=shape[1], sigma=sigmas[(seed + k) % 4], seed=seed + k, abl=_abl(c))
            for k in range(c["media"])]


def _vector(c, gen, scale=1.0):
    """Random slot vectors of all items, zero on the Dirichlet slots."""
    shape = _shape(c)
    d = len(shape)
    v = scale * torch.randn((c["media"] * c["nrhs"], d + 1) + shape, dtype=torch.complex128, generator=gen,
                            device="cuda")
    for k in range(d):
        v[:, k].select(d - k, 0).zero_()
    return v


def _inputs(c, seed):
    """Media and vectors of a case, from the seed alone."""
    meds = _media(c, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.complex128 if c["prec"] == "c128" else torch.complex64
    s = dict(meds=meds)
    if c["kind"] in ("apply", "cycle"):
        s["b"] = _vector(c, gen).to(dt)
        return s
    rng = np.random.default_rng(seed)
    shape, d = _shape(c), len(_shape(c))
    lo, a = _abl(c) + 2, _abl(c)
    q = np.zeros((c["media"] * c["nrhs"], d + 1) + shape, dtype=np.complex128)
    for i in range(len(q)):     # unit x-forces on a line below the absorbing layer
        at = (lo, shape[1] // 2) if d == 3 else (lo,)
        q[(i, 0) + at + (int(rng.integers(a + 1, shape[-1] - a)),)] = 1.0
    s["q"] = torch.from_numpy(q).cuda()
    if c["kind"] in ("fwi", "autograd"):
        xs = np.unique(np.linspace(a + 2, shape[-1] - a - 2, min(200, shape[-1] - 2 * a - 4)).round().astype(int))
        s["rx"], s["ry"] = torch.from_numpy(xs).cuda(), lo
        s["data"] = 0.05 * torch.randn((c["nrhs"], len(xs)), dtype=torch.complex128, generator=gen, device="cuda")
    return s


def prepare(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    s["kind"] = c["kind"]
    if c["kind"] == "autograd":
        m = s["meds"][0]
        s["model"] = [torch.from_numpy(np.ascontiguousarray(v[None])).cuda().requires_grad_() for v in
                      (m.lam, m.mu, m.rho)]
        s["args"] = (m.omega, m.h, m.abl_cells)
        s["options"] = _options(c)
        return s
    s["solver"] = ehs.solver_for(s["meds"], **_options(c))
    v = s.get("b", s.get("q"))
    s["out"] = torch.zeros_like(v)
    if c["kind"] == "apply":
        s["shifted"] = torch.zeros_like(v)
    if c["kind"] == "fwi":
        s["adj"], s["g"] = torch.zeros_like(v), torch.zeros_like(v)
        s["grad"] = [torch.empty((1,) + _shape(c), dtype=torch.float64, device="cuda") for _ in range(3)]
    return s


# --------------------------------------------------------------------- run
def run(state):
    s, kind = state, state["kind"]
    if kind == "apply":
        s["solver"].op_apply(s["b"], s["out"])
        s["solver"].op_apply(s["b"], s["shifted"], shifted=True)
        return [s["out"], s["shifted"]]
    if kind == "cycle":
        s["solver"].vcycle(s["b"], s["out"])
        return s["out"]
    if kind == "solve":
        s["solver"].fgmres_solve(s["q"], s["out"])
        return s["out"]
    if kind == "fwi":
        S, u, w, g = s["solver"], s["out"], s["adj"], s["g"]
        S.fgmres_solve(s["q"], u)
        g[:, 0, s["ry"], s["rx"]] = u[:, 0, s["ry"], s["rx"]] - s["data"]
        S.adjoint_solve(g, w)
        S.gradient(u, w, out=s["grad"])
        return [u, w] + s["grad"]
    lam, mu, rho = s["model"]
    x = autograd.solve(lam, mu, rho, s["q"], *s["args"], **s["options"])
    misfit = 0.5 * (x[:, 0, s["ry"], s["rx"]] - s["data"]).abs().square().sum()
    return [x.detach()] + list(torch.autograd.grad(misfit, s["model"]))


# -------------------------------------------------------------------- work
def _cycle_work(c):
    """Bytes and flops of one cycle and one operator product per item batch, and the setup's flops: vectors in
    and out, the operator's coefficients, every level's stencil table and the coarsest inverses read once."""
    shape, d = _shape(c), len(_shape(c))
    cells, items = math.prod(shape), c["media"] * c["nrhs"]
    z = 16 if c["prec"] == "c128" else 8
    vec = cells * (d + 1) * z
    byt = items * 2 * vec + c["media"] * cells * 4 * (z // 2)
    flo = items * cells * (d + 1) * 8 * 20
    visits, inv = 1, 0
    for l in range(1, c["levels"]):
        n = cells // 2 ** (d * l)
        visits *= c["cycle"] if l < c["levels"] - 1 else 1
        if l < c["levels"] - 1 or c["split"] > 1:
            stored = (45 if l == 1 else 69) if d == 2 else (440 if l == 1 else 480)   # half of the symmetric stencil
            byt += c["media"] * n * stored * (4 if c["table16"] else z)
            flo += items * visits * n * stored * 2 * 8 * 5
        if l == c["levels"] - 1:
            if c["split"] > 1:
                ns = c["split"] ** 2
                ext = [s / 2 ** l for s in shape]
                box = math.prod(e / c["split"] + 2 * c["overlap"] if k >= len(ext) - 2 else e for k, e in enumerate(ext))
                live = min((d + 1) * box, (d + 1) * n)
            else:
                ns, live = 1, (d + 1) * n
            inv = c["media"] * ns * live
            byt += inv * live / 2 * (16 if c["prec"] == "c128" or c["fmt"] == "df" else 8 if c["fmt"] == "c64" else 4)
            flo += items * visits * ns * live * live * 8
    return byt, flo, items * cells * (d + 1), inv * live * live * 4


def work(case):
    c = dict(case)
    shape, d = _shape(c), len(_shape(c))
    cells, items = math.prod(shape), c["media"] * c["nrhs"]
    z = 16 if c["prec"] == "c128" else 8
    if c["kind"] == "apply":
        return {"bytes": items * cells * (d + 1) * 3 * z + c["media"] * cells * 2 * z,
                "flops": 2 * items * cells * 8 * (d * (2 * d + 3) + 2 * d + 1)}
    byt, flo, n, setup = _cycle_work(c)
    if c["kind"] == "cycle":
        return {"bytes": byt, "flops": flo}
    # iterations of a 1e-6 solve on these media, each with one cycle, one operator product and an orthogonalisation
    # that reads about half of ten basis vectors and the new one and writes one
    its = 16 if cells <= 4096 else 24 if d == 2 else 40
    one = byt + n * (5 + 2 + 3) * 16
    solves = 1 if c["kind"] == "solve" else 2
    out = {"bytes": solves * its * one, "flops": solves * its * (flo + n * 8 * 2 * 2 * 5)}
    if c["kind"] == "autograd":
        out["flops"] += setup
    return out


# ------------------------------------------- the method in plain torch, 64 bits
class _Grid:
    """Cells of a grid in slot numbering: slot (a, cell) is a * ncell + cell; u_k lives on the low face of its cell
    along direction k (numpy axis d - 1 - k), slots with index 0 along k are not unknowns."""

    def __init__(self, shape):
        self.shape, self.d, self.n = tuple(shape), len(shape), math.prod(shape)
        self.id = torch.arange(self.n, device="cuda").reshape(self.shape)
        self.i = [torch.arange(self.shape[self.d - 1 - k], device="cuda").reshape(
            [-1 if a == self.d - 1 - k else 1 for a in range(self.d)]).expand(self.shape) for k in range(self.d)]

    def at(self, k, off, v=None):
        """The neighbour `off` cells along k, clamped to the grid (of the cell numbers, or of a cell array v)."""
        v = self.id if v is None else v
        a, m = self.d - 1 - k, self.shape[self.d - 1 - k]
        return v.index_select(a, (torch.arange(m, device=v.device) + off).clamp(0, m - 1))

    def live(self):
        return torch.cat([(self.i[k] >= 1).reshape(-1) for k in range(self.d)] +
                         [torch.ones(self.n, dtype=torch.bool, device="cuda")])


def _entries(g, lam, mu, rho, omega, h, abl, alpha):
    """(row, column, value) of K (alpha = 0) or of the shifted operator, values differentiable in the medium."""
    d, n = g.d, g.n
    ramp = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    for k in range(d):
        m = g.shape[d - 1 - k]
        depth = torch.maximum(abl - g.i[k], g.i[k] - (m - 1 - abl)).clamp(min=0).double()
        ramp = torch.maximum(ramp, (depth / abl) ** 2)
    gamma = 0.01 * math.pi + omega * ramp
    rows, cols, vals = [], [], []

    def add(mask, a, b, to, v):
        rows.append(a * n + g.id[mask])
        cols.append(b * n + to[mask])
        vals.append(v[mask] * torch.ones((), dtype=torch.complex128, device="cuda"))

    for k in range(d):
        ok = g.i[k] >= 1
        m = g.shape[d - 1 - k]
        low = g.at(k, -1, mu)
        total = mu + low
        add(ok & (g.i[k] + 1 < m), k, k, g.at(k, 1), -mu / h ** 2)
        add(ok & (g.i[k] - 1 >= 1), k, k, g.at(k, -1), -low / h ** 2)
        for j in range(d):
            if j == k:
                continue
            for off in (1, -1):
                w = 0.25 * (mu + low + g.at(j, off, mu) + g.at(j, off, low))
                total = total + w
                inside = g.i[j] + 1 < g.shape[d - 1 - j] if off > 0 else g.i[j] >= 1
                add(ok & inside, k, k, g.at(j, off), -w / h ** 2)
        face = lambda v: 0.5 * (v + g.at(k, -1, v))
        mass = torch.complex(face(rho), -face(rho * gamma) / omega)
        add(ok, k, k, g.id, total / h ** 2 - omega ** 2 * mass + 1j * alpha * omega ** 2 * face(rho))
        one = torch.ones(g.shape, dtype=torch.float64, device="cuda") / h
        add(ok, k, d, g.id, one)
        add(ok, k, d, g.at(k, -1), -one)
        add(ok, d, k, g.id, one)
        add(g.i[k] + 1 < m, d, k, g.at(k, 1), -one)
    add(g.id >= 0, d, d, g.id, -1.0 / (lam + mu))
    return torch.cat(rows), torch.cat(cols), torch.cat(vals)


class _Sparse:
    def __init__(self, r, c, v, m, n):
        self.coo = torch.sparse_coo_tensor(torch.stack([r, c]), v, (m, n)).coalesce()
        self._csr()

    def _csr(self):
        self.csr = self.coo.to_sparse_csr()
        i = self.coo.indices()
        self.keys, self.vals, self.width = i[0] * self.coo.shape[1] + i[1], self.coo.values(), self.coo.shape[1]

    def __matmul__(self, x):
        return self.csr @ x

    def get(self, r, c):
        """Entries at (r, c), zero where none is stored."""
        key = r * self.width + c
        at = torch.searchsorted(self.keys, key).clamp(max=len(self.keys) - 1)
        return torch.where(self.keys[at] == key, self.vals[at], torch.zeros_like(self.vals[at]))

    @staticmethod
    def of(coo):
        s = _Sparse.__new__(_Sparse)
        s.coo = coo.coalesce()
        s._csr()
        return s


def _prolongation(gc):
    """The grid twice as fine from gc: u_k linear along k between faces, 3/4 and 1/4 across; p 3/4 and 1/4 with
    clamped ghosts (u: zero ghosts)."""
    d = gc.d
    gf = _Grid([2 * s for s in gc.shape])
    rows, cols, vals = [], [], []
    for a in range(d + 1):
        terms = [(torch.zeros_like(gf.id), torch.ones(gf.shape, dtype=torch.float64, device="cuda"))]
        for k in range(d):
            j, m = gf.i[k], gc.shape[d - 1 - k]
            stride = math.prod(gc.shape[d - k:]) if k else 1
            if a == k:
                even = (j % 2 == 0).double()
                two = [(j // 2, 0.5 + 0.5 * even), ((j + 1) // 2, 0.5 - 0.5 * even)]
                two = [(J, w * ((J >= 1) & (J <= m - 1) & (j >= 1))) for J, w in two]
            else:
                near = j // 2
                nb = torch.where(j % 2 == 1, near + 1, near - 1)
                inside = (nb >= 0) & (nb < m)
                two = [(near, torch.where(inside, 0.75, 1.0 if a == d else 0.75).double()), (nb, 0.25 * inside)]
            terms = [(t + J.clamp(0, m - 1) * stride, w * v) for t, w in terms for J, v in two]
        for t, w in terms:
            ok = w != 0
            rows.append(a * gf.n + gf.id[ok])
            cols.append(a * gc.n + t[ok])
            vals.append(w[ok].to(torch.complex128))
    return _Sparse(torch.cat(rows), torch.cat(cols), torch.cat(vals), (d + 1) * gf.n, (d + 1) * gc.n)


class _Cycle:
    """Multigrid cycle of the shifted operator: red-black economic cell relaxation, Galerkin coarse operators, the
    coarsest grid solved exactly or by one sweep over overlapping boxes, colour by colour."""

    def __init__(self, c, g, entries):
        self.c, self.levels = c, c["levels"]
        n = (g.d + 1) * g.n
        self.g, self.A, self.P, self.blocks = [g], [_Sparse(*entries, n, n)], [], []
        for l in range(self.levels - 1):
            gc = _Grid([s // 2 for s in self.g[-1].shape])
            P = _prolongation(gc)
            A = self.A[-1].coo
            R = P.coo.transpose(0, 1).coalesce()
            self.blocks.append(self._block_inverses(self.g[-1], self.A[-1], _weights(c)[min(l, len(_weights(c)) - 1)]))
            self.A.append(_Sparse.of(torch.sparse.mm(R, torch.sparse.mm(A, P.coo))))
            P.rt = R.to_sparse_csr()
            self.P.append(P)
            self.g.append(gc)
        self._coarsest()

    @staticmethod
    def _block_inverses(g, A, w):
        d, n = g.d, g.n
        dofs, ok = [], []
        for side in (0, 1):
            for k in range(d):
                dofs.append((k * n + (g.id if side == 0 else g.at(k, 1))).reshape(-1))
                ok.append((g.i[k] >= 1 if side == 0 else g.i[k] + 1 < g.shape[d - 1 - k]).reshape(-1))
        dofs.append(d * n + g.id.reshape(-1))
        ok.append(torch.ones(n, dtype=torch.bool, device="cuda"))
        dofs, ok = torch.stack(dofs, 1), torch.stack(ok, 1)
        m = 2 * d + 1
        B = torch.eye(m, dtype=torch.complex128, device="cuda").repeat(n, 1, 1)
        for a in range(m):
            for b in range(m):
                if a == b or a == 2 * d or b == 2 * d:
                    both = ok[:, a] & ok[:, b]
                    B[both, a, b] = A.get(dofs[both, a], dofs[both, b])
        parity = sum(g.i).reshape(-1) % 2
        inv = w * torch.linalg.inv(B)
        return [(dofs[parity == p], ok[parity == p], inv[parity == p]) for p in (0, 1)]

    def _relax(self, l, b, x):
        for dofs, ok, inv in self.blocks[l]:
            r = (b - self.A[l] @ x)[dofs] * ok[:, :, None]
            x = x.index_put((dofs.reshape(-1),), ((inv @ r) * ok[:, :, None]).reshape(-1, b.shape[1]), accumulate=True)
        return x

    def _coarsest(self):
        g, A = self.g[-1], self.A[-1]
        N = (g.d + 1) * g.n
        split = [self.c["split"] if k < 2 or not self.c["nz"] else 1 for k in range(g.d)]
        over = self.c["overlap"]
        edges = []
        for k in range(g.d):
            m, s = g.shape[g.d - 1 - k], split[k]
            cut = [0]
            for q in range(s):
                cut.append(cut[-1] + m // s + (1 if q < m % s else 0))
            edges.append([(max(cut[q] - over, 0), min(cut[q + 1] + over, m)) if s > 1 else (0, m) for q in range(s)])
        boxes = [[]]
        for k in range(g.d):
            boxes = [b + [(q, lohi)] for b in boxes for q, lohi in enumerate(edges[k])]
        live = g.live()
        i = A.coo.indices()
        self.boxes = {}
        for b in boxes:
            colour = sum((q % 2) << k for k, (q, _) in enumerate(b))
            inside = torch.ones(g.shape, dtype=torch.bool, device="cuda")
            for k, (_, (lo, hi)) in enumerate(b):
                inside = inside & (g.i[k] >= lo) & (g.i[k] < hi)
            sel = [(inside & (g.i[k] - 1 >= b[k][1][0])).reshape(-1) for k in range(g.d)] + [inside.reshape(-1)]
            idx = torch.nonzero(torch.cat(sel) & live).reshape(-1)
            at = torch.full((N,), -1, dtype=torch.long, device="cuda")
            at[idx] = torch.arange(len(idx), device="cuda")
            both = (at[i[0]] >= 0) & (at[i[1]] >= 0)
            M = torch.zeros((len(idx), len(idx)), dtype=torch.complex128, device="cuda")
            M[at[i[0][both]], at[i[1][both]]] = A.vals[both]
            self.boxes.setdefault(colour, []).append((idx, torch.linalg.lu_factor(M)))

    def _coarse(self, b):
        x = torch.zeros_like(b)
        for colour in sorted(self.boxes):
            r = b - self.A[-1] @ x
            for idx, lu in self.boxes[colour]:
                x[idx] += torch.linalg.lu_solve(*lu, r[idx])
        return x

    def __call__(self, b, l=0, x=None):
        if l == self.levels - 1:
            return self._coarse(b)
        x = self._relax(l, b, torch.zeros_like(b) if x is None else x)
        rc = self.P[l].rt @ (b - self.A[l] @ x)
        e = None
        for _ in range(1 if l + 2 == self.levels else self.c["cycle"]):
            e = self(rc, l + 1, e)
        return self._relax(l, b, x + self.P[l] @ e)


def _gmres(K, M, q, tol=1e-12, most=150):
    """Solutions of K u = q for the columns of q: right-preconditioned GMRES without restarts, all columns at once."""
    beta = torch.linalg.norm(q, dim=0)
    V, Z, H = [q / beta], [], []
    for j in range(most):
        Z.append(M(V[j]))
        w = K @ Z[j]
        h = []
        for _ in range(2):
            B = torch.stack(V)
            p = torch.einsum("ink,nk->ik", B.conj(), w)
            w = w - torch.einsum("ink,ik->nk", B, p)
            h.append(p)
        nrm = torch.linalg.norm(w, dim=0)
        V.append(w / nrm)
        H.append(torch.cat([h[0] + h[1], nrm[None].to(h[0].dtype)]).cpu())
        Hm = torch.zeros((q.shape[1], j + 2, j + 1), dtype=torch.complex128)
        for t, col in enumerate(H):
            Hm[:, : t + 2, t] = col.T
        e = torch.zeros((q.shape[1], j + 2, 1), dtype=torch.complex128)
        e[:, 0, 0] = beta.cpu()
        y = torch.linalg.lstsq(Hm, e).solution
        if float((torch.linalg.norm(e - Hm @ y, dim=1)[:, 0] / beta.cpu()).max()) < tol:
            break
    return torch.einsum("ink,ik->nk", torch.stack(Z), y[:, :, 0].T.to(q.device))


def exact(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    if c["kind"] == "solve" and c["nz"] and math.prod(_shape(c)) > 64 ** 3:
        return None         # assembling and factorising the 3D hierarchy this size takes too long
    shape, per = _shape(c), c["nrhs"]
    g = _Grid(shape)
    n = (g.d + 1) * g.n
    outs, grads = [], []
    for k, m in enumerate(s["meds"]):
        model = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (m.lam, m.mu, m.rho)]
        args = (m.omega, m.h, m.abl_cells)
        K = _Sparse(*_entries(g, *model, *args, 0.0), n, n)
        cols = lambda v: v[k * per:(k + 1) * per].to(torch.complex128).reshape(per, n).T.contiguous()
        back = lambda v: v.T.reshape((per, g.d + 1) + shape)
        if c["kind"] == "apply":
            Ks = _Sparse(*_entries(g, *model, *args, c["alpha"]), n, n)
            outs.append(back(K @ cols(s["b"])))
            grads.append(back(Ks @ cols(s["b"])))
            continue
        C = _Cycle(c, g, _entries(g, *model, *args, c["alpha"]))
        if c["kind"] == "cycle":
            outs.append(back(C(cols(s["b"]))))
            continue
        u = _gmres(K, C, cols(s["q"]))
        outs.append(back(u))
        if c["kind"] == "solve":
            continue
        e = torch.zeros_like(outs[0])
        e[:, 0, s["ry"], s["rx"]] = outs[0][:, 0, s["ry"], s["rx"]] - s["data"]
        w = _gmres(K, C, cols(e).conj().resolve_conj()).conj().resolve_conj()   # K is symmetric: K^H = conj(K)
        model = [v.requires_grad_() for v in model]
        r, col, val = _entries(g, *model, *args, 0.0)
        grads = torch.autograd.grad(-(w[r].conj() * u.detach()[col]).sum(1).mul(val).real.sum(), model)
        grads = [back(w)] * (c["kind"] == "fwi") + [v[None] for v in grads]
    out = torch.cat(outs)
    if c["kind"] == "apply":
        return [out, torch.cat(grads)]
    return [out] + list(grads) if c["kind"] in ("fwi", "autograd") else out
