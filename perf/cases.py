"""The work this library is measured on: what a program that uses it has it do.

Three kinds of work, each through the public entry points:

  solve    ALB generation from a random block to a residual tolerance
           (dgdft_alb_solve), the start of a calculation;
  step     one SCF step of ALB generation (dgdft_alb_scf_step: three LOBPCG
           iterations from the previous block under a new potential), what a
           calculation spends most of its ALB time on;
  dg       what follows the ALBs: the DG Hamiltonian's block rows
           (dgdft_dg_assemble) and, for small systems, the density by dense
           diagonalisation (dgdft_dg_density).

Systems are of the repository's own kinds: extended elements of a puckered
monolayer (37.56 x 51.72 x 24 bohr on 48 x 64 x 40 or 48 x 64 x 48 points, 144
atoms, two projectors each) and standalone boxes of random atoms of uneven
size.  Potentials and projectors are built here from seeded atom positions:
the screened local pseudopotential -Z erf(r / rc) / r as a Fourier series, s
and p Gaussians cut at 2 bohr as Kleinman-Bylander projectors.

A box is written nx x ny x nz / m / J: its grid, the eigenpairs computed and
the ALBs kept; "4*48x64x40/48/40" is four of them.
"""

import ctypes
import math

import numpy as np
import torch

from paper_1506_08147_gb300 import binding as B

Z_ION, RC_LOC, SIGMA_KB, RCUT_KB = 5.0, 0.8, 0.5, 2.0
LAYER_L = (37.56, 51.72, 24.0)   # the monolayer's extended element (bohr) on 48 x 64 points in-plane
CELL_X, CELL_Y = 6.26, 8.62      # its primitive cell
PUCKER = ((0.0, 0.10, -2.0), (0.5, 0.40, -2.0), (0.5, 0.60, 2.0), (0.0, 0.90, 2.0))


def listed():
    return [
        # The smallest system the DG part is used on: a cube of 27 elements with few functions each; launches count.
        {"name": "dg_cube", "kind": "dg", "ne": "3x3x3", "nq": "18x18x18", "J": 6, "arith": 0, "density": False},
        # The 576-atom monolayer's DG Hamiltonian (36 elements, 40 functions on 32 x 42 x 80 points), once per SCF step.
        {"name": "dg_layer", "kind": "dg", "ne": "6x6x1", "nq": "48x64x40", "J": 40, "arith": 0, "density": False},
        # The same with the pair-arithmetic option.
        {"name": "dg_layer_pairs", "kind": "dg", "ne": "6x6x1", "nq": "48x64x40", "J": 40, "arith": 1, "density": False},
        # Density of a small layer: 72 functions in all.
        {"name": "density_small", "kind": "dg", "ne": "3x3x1", "nq": "24x24x30", "J": 8, "arith": 0, "density": True},
        # Density of the 576-atom monolayer by dense diagonalisation (1,440 functions, half of them occupied).
        {"name": "density_layer", "kind": "dg", "ne": "6x6x1", "nq": "48x64x40", "J": 40, "arith": 0, "density": True},
        # An SCF step of one monolayer element: what a rank with a single element does.
        {"name": "step_one", "kind": "step", "system": "layer", "boxes": "1*48x64x40/48/40", "mixed": True, "cut": 0.0},
        # An SCF step of the whole 576-atom monolayer: 36 elements, 1,440 ALBs.
        {"name": "step_layer", "kind": "step", "system": "layer", "boxes": "36*48x64x40/48/40", "mixed": True, "cut": 0.0},
        # An SCF step of unlike boxes in one batch, few to many functions each.
        {"name": "step_uneven", "kind": "step", "system": "box",
         "boxes": "1*24x24x24/32/24 1*32x32x32/48/38 1*40x40x48/72/58 1*32x32x32/104/85 1*48x48x64/88/72 1*24x24x24/64/52",
         "mixed": True, "cut": 0.0},
        # An SCF step of elements of the 3,456-atom monolayer: 144 computed, 120 kept.
        {"name": "step_large", "kind": "step", "system": "layer", "boxes": "2*48x64x48/144/120", "mixed": True, "cut": 0.0},
        # An SCF step in plain FP64, the comparison arithmetic.
        {"name": "step_fp64", "kind": "step", "system": "layer", "boxes": "4*48x64x40/48/40", "mixed": False, "cut": 0.0},
        # A single small box solved from a random block to 1e-8 Ha in FP64: the smallest whole call.
        {"name": "solve_box", "kind": "solve", "system": "box", "boxes": "1*16x16x16/16/16", "mixed": False, "cut": 0.0,
         "tol": 1e-8},
        # Monolayer elements solved from random blocks to 1e-6 Ha: the benchmark's call on a few elements.
        {"name": "solve_layer", "kind": "solve", "system": "layer", "boxes": "3*48x64x40/48/40", "mixed": True, "cut": 0.0,
         "tol": 1e-6},
    ]


GRID_X = (16, 18, 20, 24, 30, 32, 36, 40, 48)          # even, factors 2, 3, 5
GRID_YZ = (15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64)


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_box(rng, max_j):
    n = (rng.choice(GRID_X), rng.choice(GRID_YZ), rng.choice(GRID_YZ))
    # at most a hundredth of the planewaves: the pencils of 3 m vectors stay well conditioned
    j = min(_spread(rng, 8, max_j), max(4, n[0] * n[1] * n[2] // 160))
    m = j + max(1, math.ceil(0.2 * j)) + rng.randrange(3)
    return "1*%dx%dx%d/%d/%d" % (*n, m, j)


def draw(rng):
    kind = rng.choice(("dg", "dg", "density", "step", "step", "layer", "solve"))
    if kind in ("dg", "density"):
        ne = tuple(rng.choice((1, 3, 4)) for _ in range(2)) + (1,) if rng.random() < 0.7 else (3, 3, 3)
        nq = (rng.choice((12, 18, 24, 30, 36, 48)), rng.choice((12, 15, 18, 24, 27, 36, 48)), rng.choice((12, 18, 20, 27, 30, 40)))
        n_elem = ne[0] * ne[1] * ne[2]
        j = _spread(rng, 3, min(48, nq[0] * nq[1] * nq[2] // 400 + 4))
        if kind == "density":
            j = min(j, max(3, 800 // n_elem))
        return {"kind": "dg", "ne": "%dx%dx%d" % ne, "nq": "%dx%dx%d" % nq, "J": j,
                "arith": rng.choice((0, 0, 1)) if kind == "dg" else 0, "density": kind == "density"}
    if kind == "layer":
        m = rng.randrange(24, 49)
        return {"kind": "step", "system": "layer", "boxes": "%d*48x64x%d/%d/%d" % (_spread(rng, 1, 24), rng.choice((40, 48)), m, m - rng.randrange(4, 9)),
                "mixed": True, "cut": rng.choice((0.0, 0.0, 0.9137))}
    if kind == "step":
        boxes = [_draw_box(rng, 96) for _ in range(_spread(rng, 1, 6))]
        return {"kind": "step", "system": "box", "boxes": " ".join(boxes), "mixed": rng.random() < 0.7, "cut": rng.choice((0.0, 0.0, 0.9137))}
    n = (rng.choice((16, 18, 20, 24)), rng.choice((15, 16, 18, 20, 24)), rng.choice((16, 18, 20, 24, 25)))
    m = rng.randrange(10, 29)
    return {"kind": "solve", "system": "box", "boxes": "1*%dx%dx%d/%d/%d" % (*n, m, m - rng.randrange(3, 6)), "mixed": rng.random() < 0.5,
            "cut": 0.0, "tol": 1e-6}


# ------------------------------------------------------------------ systems

def _three(text):
    return tuple(int(v) for v in text.split("x"))


def _boxes(case):
    out = []
    for word in case["boxes"].split():
        count, rest = word.split("*")
        grid, m, j = rest.split("/")
        out += [(_three(grid), int(m), int(j))] * int(count)
    return out


def _lengths(case, n):
    if case["system"] == "layer":
        return (LAYER_L[0] * n[0] / 48, LAYER_L[1] * n[1] / 64, LAYER_L[2])
    return tuple(0.78 * v for v in n)


def _atoms(case, n, L, J, gen):
    """Positions in the box: a perturbed puckered layer, or random with a least distance."""
    if case["system"] == "layer":
        return _layer_atoms(max(1, round(L[0] / CELL_X)), max(1, round(L[1] / CELL_Y)), L, gen)
    n_at = max(3, min(4 + round((J - 16) * 36 / 80), int(np.prod(L) / 160)))
    return _random_atoms(n_at, np.asarray(L), gen)


def _layer_atoms(cx, cy, L, gen):
    base = [((i + fx) / cx * L[0], (j + fy) / cy * L[1], L[2] / 2 + z) for j in range(cy) for i in range(cx) for fx, fy, z in PUCKER]
    return np.mod(np.array(base) + gen.uniform(-0.2, 0.2, (len(base), 3)), L)


def _random_atoms(count, L, gen):
    got = []
    for tries in range(20000):
        r = gen.uniform(0, 1, 3) * L
        far = 2.5 if tries < 4000 else 1.5
        d = np.array(got).reshape(-1, 3) - r
        d -= np.round(d / L) * L
        if not len(got) or np.min(np.sum(d * d, axis=1)) > far * far:
            got.append(r)
            if len(got) == count:
                break
    return np.array(got)


def _freq(n, length):
    return torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device="cuda") * (2 * math.pi / length)


def _symbol(n, L):
    """|G|^2 / 2 on the (nz, ny, nx/2 + 1) half spectrum."""
    gx = _freq(n[0], L[0])[: n[0] // 2 + 1]
    return 0.5 * (_freq(n[2], L[2])[:, None, None] ** 2 + _freq(n[1], L[1])[None, :, None] ** 2 + gx[None, None, :] ** 2)


def _local_coeffs(atoms, n, L):
    """Fourier coefficients of the local pseudopotential over the full grid of frequencies, and these."""
    g = [_freq(k, l) for k, l in zip(n, L)]
    g2 = g[2][:, None, None] ** 2 + g[1][None, :, None] ** 2 + g[0][None, None, :] ** 2
    v = -(4 * math.pi * Z_ION / float(np.prod(L))) * torch.exp(-g2 * RC_LOC ** 2 / 4) / torch.where(g2 == 0, torch.ones_like(g2), g2)
    v[0, 0, 0] = 0.0
    r = torch.as_tensor(atoms, dtype=torch.float64, device="cuda")
    e = [torch.exp(-1j * torch.outer(r[:, d], g[d])) for d in range(3)]
    plane = e[1][:, :, None] * e[0][:, None, :]                       # atom, y, x
    sf = torch.matmul(e[2].T, plane.reshape(len(atoms), -1)).reshape(g2.shape)
    return v * sf, g


def _series_at(coef, g, pts):
    """The series at the tensor points pts = (xs, ys, zs); (nz, ny, nx)."""
    e = [torch.exp(1j * torch.outer(gd, torch.as_tensor(p, dtype=torch.float64, device="cuda"))) for gd, p in zip(g, pts)]
    v = coef @ e[0]                                                   # z, y, x'
    v = torch.einsum("zyx,yb->zbx", v, e[1])
    v = torch.einsum("zbx,zc->cbx", v, e[2])
    return v.real.contiguous()


def _near(atom, pts, cell):
    """Tensor points within the cut of an atom (minimum image): flat indices, distances squared, z offsets."""
    d = [np.asarray(p) - a for p, a in zip(pts, atom)]
    d = [v - np.round(v / c) * c for v, c in zip(d, cell)]
    ii, jj, kk = (np.nonzero(np.abs(v) <= RCUT_KB)[0] for v in d)
    r2 = d[2][kk][:, None, None] ** 2 + d[1][jj][None, :, None] ** 2 + d[0][ii][None, None, :] ** 2
    flat = ii[None, None, :] + len(pts[0]) * (jj[None, :, None] + len(pts[1]) * kk[:, None, None])
    keep = r2 <= RCUT_KB ** 2
    dz = np.broadcast_to(d[2][kk][:, None, None], r2.shape)
    return flat[keep], r2[keep], dz[keep]


def _kb(atoms, pts, cell, unit):
    """KB projectors at tensor points as CSR rows (ids, row_ptr, idx, val). unit: rows of Euclidean
    norm 1 (the ALB problem's), else functions of unit L2 norm (the DG problem's)."""
    pid, ptr, idx, val = [], [0], [], []
    r = np.linspace(0, RCUT_KB, 4001)
    gr = np.exp(-(r / SIGMA_KB) ** 2)
    l2 = [math.sqrt(np.trapezoid(4 * math.pi * r ** 2 * gr, r)), math.sqrt(np.trapezoid(4 * math.pi / 3 * r ** 4 * gr, r))]
    for a, r0 in enumerate(atoms):
        flat, r2, dz = _near(r0, pts, cell)
        g = np.exp(-r2 / (2 * SIGMA_KB ** 2))
        for ell, b in enumerate((g, dz * g)):
            norm = math.sqrt(float(np.sum(b * b))) if unit else l2[ell]
            if len(flat) == 0 or norm == 0.0:
                continue
            pid.append(2 * a + ell)
            idx.append(flat)
            val.append(b / norm)
            ptr.append(ptr[-1] + len(flat))
    cat = lambda v, t: np.concatenate(v).astype(t) if v else np.zeros(0, t)  # noqa: E731
    return np.asarray(pid, np.int32), np.asarray(ptr, np.int64), cat(idx, np.int32), cat(val, np.float64)


def _e_box(n):
    """E_K inside Q_K: the middle third in-plane, all of z."""
    lo = (math.ceil(n[0] / 3), math.ceil(n[1] / 3), 0)
    return lo, (math.ceil(2 * n[0] / 3), math.ceil(2 * n[1] / 3), n[2])


def _element(case, k, n, m, J, seed):
    """One element's inputs; the same on every call with the same arguments."""
    gen = np.random.default_rng([seed, 11, k])
    L = _lengths(case, n)
    atoms = _atoms(case, n, L, J, gen)
    pts = [np.arange(nd) * (ld / nd) for nd, ld in zip(n, L)]
    coef, g = _local_coeffs(atoms, n, L)
    v = _series_at(coef, g, pts)
    pid, ptr, idx, val = _kb(atoms, pts, L, True)
    gamma = gen.uniform(0.5, 2.0, 2 * len(atoms))[pid]
    tg = torch.Generator(device="cuda").manual_seed(seed * 4096 + k)
    x = torch.randn((m, n[2], n[1], n[0]), generator=tg, device="cuda", dtype=torch.float64)
    if case["kind"] == "step":
        # a block as an earlier step leaves it: smooth, and largest where the potential is low
        x = torch.fft.irfftn(torch.fft.rfftn(x, dim=(1, 2, 3)) * torch.exp(-_symbol(n, L)), s=(n[2], n[1], n[0]), dim=(1, 2, 3))
        x = x / (1.0 + torch.exp((v - v.mean()) / v.std()))
    x = x.reshape(m, -1)
    x = (x / x.norm(dim=1, keepdim=True)).contiguous()
    return {"n": n, "L": L, "m": m, "J": J, "v": v.reshape(-1), "ptr": ptr, "idx": idx, "val": val, "gamma": gamma, "x0": x}


def _ecut(case, els):
    """The cutoff of Eq. Ngecut (the sphere inscribed in the coarsest axis of the batch), times cut."""
    low = min(min((math.pi * nd / ld) ** 2 / 2 for nd, ld in zip(e["n"], e["L"])) for e in els)
    return case["cut"] * low


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    return _prepare_dg(case, seed) if case["kind"] == "dg" else _prepare_alb(case, seed)


def run(state):
    return _run_dg(state) if state["case"]["kind"] == "dg" else _run_alb(state)


def _prepare_alb(case, seed):
    els = [_element(case, k, n, m, J, seed) for k, (n, m, J) in enumerate(_boxes(case))]
    descs = []
    for e in els:
        lo, hi = _e_box(e["n"])
        descs.append({"n": e["n"], "L": e["L"], "e_lo": lo, "e_hi": hi, "m": e["m"], "J": e["J"]})
    stream = torch.cuda.Stream()
    ctx = B.Context(descs, precision=B.DGDFT_PREC_MIXED if case["mixed"] else B.DGDFT_PREC_FP64, tol=case.get("tol", 1e-6),
                    maxit=800, ecut=_ecut(case, els), stream=stream.cuda_stream)
    for k, e in enumerate(els):
        ctx.dgdft_alb_set_projectors(k, e["ptr"], e["idx"], e["val"], e["gamma"])
    phi = [torch.empty((e["J"], int(np.prod(np.subtract(d["e_hi"], d["e_lo"])))), dtype=torch.float64, device="cuda")
           for e, d in zip(els, descs)]
    torch.cuda.synchronize()
    return {"case": case, "ctx": ctx, "stream": stream, "v": [e["v"] for e in els], "x0": [e["x0"] for e in els], "phi": phi}


def _run_alb(state):
    """The potential and the block go in, the step or solve runs, the ALBs and their eigenvalues come out.

    The columns of phi are fixed up to their signs and, where two singular values are close, a
    rotation, so a program does not compare them; what they span on E_K is seen at every point by
    sum_j phi_j(x)^2.  A solve fixes its vectors only to the tolerance over a gap: its eigenvalues
    are what a program relies on.  A mixed step's iterations run in FP32 and no FP64 stage refines
    them, so FP32 is the type its numbers are kept in."""
    ctx, case = state["ctx"], state["case"]
    with torch.cuda.stream(state["stream"]):
        for k, (v, x0) in enumerate(zip(state["v"], state["x0"])):
            ctx.dgdft_alb_set_potential(k, v)
            ctx.dgdft_alb_set_initial(k, x0)
        if case["kind"] == "step":
            ctx.dgdft_alb_scf_step(3)
        else:
            ctx.dgdft_alb_solve(check=True)
        eig, res = [], []
        for k, phi in enumerate(state["phi"]):
            _, e, r = ctx.dgdft_alb_get_basis(k, phi)
            eig.append(e)
            res.append(r)
        eig, res = np.concatenate(eig), np.concatenate(res)
        if case["kind"] == "solve":
            return {"eig": eig}
        span = [phi.square().sum(0) for phi in state["phi"]]
        if case["mixed"]:
            eig, res, span = eig.astype(np.float32), res.astype(np.float32), [s.float() for s in span]
        return {"eig": eig, "res": res, "span": span}


class _Domain:
    """The periodic cell of a DG case, its elements and their grids."""

    def __init__(self, case):
        self.ne, self.nq, self.J, self.alpha = _three(case["ne"]), _three(case["nq"]), case["J"], 20.0
        self.span = tuple(3 if n > 1 else 1 for n in self.ne)
        # the monolayer's spacings; a box that spans the cell along z is as deep as the layer
        h = (LAYER_L[0] / 48, LAYER_L[1] / 64, LAYER_L[2] / 40)
        self.lq = tuple(n * d for n, d in zip(self.nq, h))
        self.le = tuple(l / s for l, s in zip(self.lq, self.span))
        self.cell = tuple(l * n for l, n in zip(self.le, self.ne))
        self.nl = tuple(max(2, 2 * round(n / s)) for n, s in zip(self.nq, self.span))
        self.off = tuple(l * (s // 2) for l, s in zip(self.le, self.span))
        self.n_elem = int(np.prod(self.ne))

    def atoms(self, gen):
        if self.ne[2] == 1:
            return _layer_atoms(max(1, round(self.cell[0] / CELL_X)), max(1, round(self.cell[1] / CELL_Y)), self.cell, gen)
        return _random_atoms(max(2, int(np.prod(self.cell) / 290)), np.asarray(self.cell), gen)

    def series_grid(self):
        return tuple(min(128, 2 * round(n * q / s / 2)) for n, q, s in zip(self.ne, self.nq, self.span))

    def corner(self, k):
        i = (k % self.ne[0], k // self.ne[0] % self.ne[1], k // (self.ne[0] * self.ne[1]))
        return tuple(a * l for a, l in zip(i, self.le))


def _columns(dom, k, seed):
    """J smooth functions on Q_K's grid, (J, N): a random Fourier series, damped."""
    tg = torch.Generator(device="cuda").manual_seed(seed * 4096 + 2048 + k)
    nx, ny, nz = dom.nq
    x = torch.randn((dom.J, nz, ny, nx), generator=tg, device="cuda", dtype=torch.float64)
    x = torch.fft.irfftn(torch.fft.rfftn(x, dim=(1, 2, 3)) * torch.exp(-_symbol(dom.nq, dom.lq)), s=(nz, ny, nx), dim=(1, 2, 3))
    x = x.reshape(dom.J, -1)
    return (x / x.square().mean(dim=1, keepdim=True).sqrt()).contiguous()


def _dg_system(dom, seed):
    gen = np.random.default_rng([seed, 12])
    atoms = dom.atoms(gen)
    gamma = gen.uniform(0.5, 2.0, 2 * len(atoms))
    coef, g = _local_coeffs(atoms, dom.series_grid(), dom.cell)
    return atoms, gamma, coef, g


def _prepare_dg(case, seed):
    dom = _Domain(case)
    atoms, gamma, coef, g = _dg_system(dom, seed)
    dg = B.DG(dom.ne, dom.cell, dom.span, dom.nq, dom.nl, dom.J, dom.alpha, 2 * len(atoms), dfloat=bool(case["arith"]))
    dg.dgdft_dg_set_gamma(gamma)
    for k in range(dom.n_elem):
        pts = dg.dgdft_dg_lgl_points(k)
        dg.dgdft_dg_set_potential(k, _series_at(coef, g, pts).reshape(-1))
        dg.dgdft_dg_set_projectors(k, *_kb(atoms, pts, dom.cell, False))
    cols = [_columns(dom, k, seed) for k in range(dom.n_elem)]
    state = {"case": case, "dom": dom, "dg": dg, "cols": cols}
    if case["density"]:
        dg.dgdft_dg_assemble(cols)
        state["rho"] = torch.empty((dom.n_elem, int(np.prod(dom.nl))), dtype=torch.float64, device="cuda")
    else:
        state["rows"] = [torch.empty((len(dg.dgdft_dg_neighbours(k)), dom.J, dom.J), dtype=torch.float64, device="cuda")
                         for k in range(dom.n_elem)]
    torch.cuda.synchronize()
    return state


def _run_dg(state):
    dg, cols = state["dg"], state["cols"]
    if state["case"]["density"]:
        eig, rho = dg.dgdft_dg_density(cols, dg.n_elem * dg.J // 2, out=state["rho"])
        return {"eig": eig, "rho": rho}
    dg.dgdft_dg_assemble(cols)
    for k, row in enumerate(state["rows"]):
        # the C entry point, so that the rows stay on the device
        status = dg.lib.dgdft_dg_get_row(dg.h, k, ctypes.c_void_p(row.data_ptr()), 1)
        if status != B.DGDFT_OK:
            raise RuntimeError("dgdft_dg_get_row: status %d" % status)
    return {"rows": list(state["rows"])}


# ------------------------------------------------------------------ work

def work(case):
    """Bytes: inputs read and outputs written once; the working blocks of an ALB iteration are
    neither. Operations: multiply-adds as two, of the products each step cannot do without."""
    if case["kind"] == "dg":
        dom = _Domain(case)
        nq, nl, J = float(np.prod(dom.nq)), float(np.prod(dom.nl)), dom.J
        lx, ly, lz = dom.nl
        qx, qy, qz = dom.nq
        interp = 2.0 * J * (lx * qx * qy * qz + lx * ly * qy * qz + lx * ly * lz * qz)
        basis = 2.0 * nl * J * J                     # mass matrix (half) and its inverse factor applied (half)
        if case["density"]:
            n, occ = dom.n_elem * J, dom.n_elem * J // 2
            flops = dom.n_elem * (interp + basis + 2.0 * nl * J * J) + 4.0 / 3 * n ** 3 + 2.0 * n * n * occ + 2.0 * n * J * 27 * occ
            return {"bytes": 8.0 * (dom.n_elem * (nq * J + nl) + n * n + occ), "flops": flops}
        grad = 2.0 * J * nl * (lx + ly + lz)
        volume = 4.0 * nl * J * J                    # four symmetric products
        nb = float(np.prod([min(3, n) for n in dom.ne]))
        return {"bytes": 8.0 * dom.n_elem * (nq * J + nl + nb * J * J), "flops": dom.n_elem * (interp + basis + grad + volume)}
    b = f = 0.0
    steps = 3 if case["kind"] == "step" else 50      # a solve takes 50 to 200 iterations
    for n, m, J in _boxes(case):
        ng = float(np.prod(n))
        lo, hi = _e_box(n)
        ne = float(np.prod(np.subtract(hi, lo)))
        b += 8.0 * (ng + ng * m + ne * J + 2 * J)
        # per iteration: three H applies (two transforms each), twelve products (half of two thirds by
        # symmetry), X', P', HP' updates; the initial block's; the restriction's products
        fft = 2 * 2.5 * ng * math.log2(ng) * m
        f += steps * (3 * fft + 2 * 12 * ng * m * m + 2 * 8 * ng * m * m) + 2 * fft + 8 * ng * m * m + 4 * ne * J * J
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits

def exact(case, seed):
    with torch.no_grad():
        return _exact_dg(case, seed) if case["kind"] == "dg" else _exact_alb(case, seed)


class _Hamiltonian:
    """The local problem's operators on rows of grid values, by torch's FFT."""

    def __init__(self, e, ecut):
        self.n, self.shape = e["n"], (e["n"][2], e["n"][1], e["n"][0])
        self.t = _symbol(e["n"], e["L"])
        self.mask = (self.t <= ecut) if ecut > 0 else None
        self.v = e["v"]
        ng = int(np.prod(e["n"]))
        to = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
        rows = np.repeat(np.arange(len(e["gamma"])), np.diff(e["ptr"]))
        self.b = torch.sparse_coo_tensor(torch.stack([to(rows), to(e["idx"].astype(np.int64))]), to(e["val"]),
                                         (len(e["gamma"]), ng)).coalesce()
        self.bt = self.b.transpose(0, 1).coalesce()
        self.gamma = to(e["gamma"])

    def _filter(self, x, f):
        y = torch.fft.rfftn(x.reshape(-1, *self.shape), dim=(1, 2, 3)) * f
        return torch.fft.irfftn(y, s=self.shape, dim=(1, 2, 3)).reshape(x.shape)

    def project(self, x):
        return x if self.mask is None else self._filter(x, self.mask)

    def kinetic(self, x):
        return self._filter(x, self.t)

    def __call__(self, x):
        c = torch.sparse.mm(self.b, x.T) * self.gamma[:, None]
        return self.kinetic(x) + x * self.v + torch.sparse.mm(self.bt, c).T

    def teter(self, r, t):
        s = self.t[None] / t[:, None, None, None]
        num = 27 + s * (18 + s * (12 + s * 8))
        return self._filter(r, num / (num + 16 * s ** 4))


def _ritz(s, hs, m, limit):
    a, b = s @ hs.T, s @ s.T
    d = torch.rsqrt(torch.diagonal(b))
    a, b = 0.5 * (a + a.T) * d[:, None] * d, 0.5 * (b + b.T) * d[:, None] * d
    if float(torch.linalg.cond(b)) > limit:
        return None
    low = torch.linalg.cholesky(b)
    c = torch.linalg.solve_triangular(low, a, upper=False)
    c = torch.linalg.solve_triangular(low, c.T, upper=False)
    th, z = torch.linalg.eigh(0.5 * (c + c.T))
    return th[:m], torch.linalg.solve_triangular(low.T, z[:, :m], upper=True) * d[:, None]


def _lobpcg(h, x, keep, tol, maxit):
    """Eigenvalues, residual norms and vectors after maxit iterations, or at a residual of tol."""
    m = x.shape[0]
    x = h.project(x)
    th, y = _ritz(x, h(x), m, 1e15)
    x = y.T @ x
    p = None
    for it in range(maxit + 1):
        hx = h(x)
        xx = (x * x).sum(1)
        th = (x * hx).sum(1) / xx
        r = h.project(hx - th[:, None] * x)
        res = r.norm(dim=1) / xx.sqrt()
        if it == maxit or float(res[:keep].max()) <= tol:
            return th, res, x
        w = h.teter(r, (x * h.kinetic(x)).sum(1) / xx)
        w = w - (w @ x.T) @ x
        got = None
        for s in ([x, w, p], [x, w]) if p is not None else ([x, w],):
            s = torch.cat(s)
            got = _ritz(s, h(s), m, 1e14)
            if got is not None:
                break
        y = got[1]
        p = h.project(y[m:].T @ s[m:])
        x = h.project(y[:m].T @ s[:m] + p)


def _exact_alb(case, seed):
    els = [_element(case, k, n, m, J, seed) for k, (n, m, J) in enumerate(_boxes(case))]
    ecut = _ecut(case, els)
    eig, res, span = [], [], []
    for e in els:
        tol, maxit = (0.0, 3) if case["kind"] == "step" else (0.05 * case["tol"], 400)
        J, n = e["J"], e["n"]
        th, r, x = _lobpcg(_Hamiltonian(e, ecut), e["x0"], J, tol, maxit)
        eig.append(th[:J])
        res.append(r[:J])
        lo, hi = _e_box(n)
        f = x[:J].reshape(J, n[2], n[1], n[0])[:, lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]].reshape(J, -1)
        f = torch.linalg.solve_triangular(torch.linalg.cholesky(f @ f.T), f, upper=False)
        span.append(f.square().sum(0) / float(np.prod(e["L"]) / np.prod(n)))
    if case["kind"] == "solve":
        return {"eig": torch.cat(eig).cpu().numpy()}
    return {"eig": torch.cat(eig).cpu().numpy(), "res": torch.cat(res).cpu().numpy(), "span": span}


def _lgl(n):
    """Legendre-Gauss-Lobatto nodes and weights on [-1, 1] and the differentiation matrix."""
    leg = np.polynomial.legendre
    c = np.zeros(n)
    c[-1] = 1.0
    x = np.array([-1.0, 1.0])
    if n > 2:
        d1 = leg.legder(c)
        r = np.sort(leg.legroots(d1).real)
        for _ in range(4):
            r = r - leg.legval(r, d1) / leg.legval(r, leg.legder(d1))
        x = np.concatenate([[-1.0], r, [1.0]])
    w = 2.0 / (n * (n - 1) * leg.legval(x, c) ** 2)
    p = leg.legval(x, c)
    diff = x[:, None] - x[None, :] + np.eye(n)
    d = p[:, None] / p[None, :] / diff
    np.fill_diagonal(d, 0.0)
    np.fill_diagonal(d, -d.sum(axis=1))
    return x, w, d


def _trig(n, length, pts):
    """Samples at k length / n -> the real trigonometric interpolant at pts."""
    t = pts[:, None] - np.arange(n)[None, :] * (length / n)
    out = np.ones(t.shape)
    for m in range(1, (n - 1) // 2 + 1):
        out += 2.0 * np.cos(2 * math.pi * m * t / length)
    return (out + np.cos(math.pi * n * t / length) if n % 2 == 0 else out) / n


def _exact_dg(case, seed):
    dom = _Domain(case)
    atoms, gamma, coef, g = _dg_system(dom, seed)
    to = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    J, shape = dom.J, (dom.nl[2], dom.nl[1], dom.nl[0])
    ref = [_lgl(n) for n in dom.nl]
    local = [(x + 1) * (l / 2) for (x, _, _), l in zip(ref, dom.le)]
    w1 = [to(w * (l / 2)) for (_, w, _), l in zip(ref, dom.le)]
    D = [to(d * (2 / l)) for (_, _, d), l in zip(ref, dom.le)]
    T = [to(_trig(n, l, o + p)) for n, l, o, p in zip(dom.nq, dom.lq, dom.off, local)]
    w = (w1[2][:, None, None] * w1[1][None, :, None] * w1[0]).reshape(-1)
    along = lambda f, d, a: torch.einsum(("ai,jcbi->jcba", "bi,jcia->jcba", "ci,jiba->jcba")[d], a, f)  # noqa: E731
    n_elem, gam = dom.n_elem, to(gamma)
    H = torch.zeros((n_elem, J, n_elem, J), dtype=torch.float64, device="cuda")
    kb = torch.zeros((n_elem, len(gamma), J), dtype=torch.float64, device="cuda")
    face, phis = [], []
    for k in range(n_elem):
        f = _columns(dom, k, seed).reshape(J, dom.nq[2], dom.nq[1], dom.nq[0])
        for d in range(3):
            f = along(f, d, T[d])
        f = f.reshape(J, -1)
        low = torch.linalg.cholesky((f * w) @ f.T)
        phi = torch.linalg.solve_triangular(low, f, upper=False)
        grid = phi.reshape(J, *shape)
        grads = [along(grid, d, D[d]) for d in range(3)]
        pts = [c + p for c, p in zip(dom.corner(k), local)]
        H[k, :, k, :] += (phi * (w * _series_at(coef, g, pts).reshape(-1))) @ phi.T
        for gd in grads:
            gd = gd.reshape(J, -1)
            H[k, :, k, :] += 0.5 * (gd * w) @ gd.T
        pid, ptr, idx, val = _kb(atoms, pts, dom.cell, False)
        for r, p in enumerate(pid):
            i = torch.as_tensor(idx[ptr[r]:ptr[r + 1]].astype(np.int64), device="cuda")
            kb[k, int(p)] = phi[:, i] @ (w[i] * to(val[ptr[r]:ptr[r + 1]]))
        end = lambda a, d, hi: a.select(3 - d, dom.nl[d] - 1 if hi else 0).reshape(J, -1)  # noqa: E731
        face.append([[(end(grid, d, hi), end(grads[d], d, hi)) for hi in (False, True)] for d in range(3)])
        phis.append(phi if case["density"] else None)
    near, at = [], lambda i: (i[0] % dom.ne[0]) + dom.ne[0] * ((i[1] % dom.ne[1]) + dom.ne[1] * (i[2] % dom.ne[2]))  # noqa: E731
    for k in range(n_elem):
        i = (k % dom.ne[0], k // dom.ne[0] % dom.ne[1], k // (dom.ne[0] * dom.ne[1]))
        near.append(sorted({at((i[0] + a, i[1] + b, i[2] + c)) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)}))
        for q in near[k]:
            H[k, :, q, :] += (kb[k] * gam[:, None]).T @ kb[q]
        for d in range(3):
            o = [e for e in (2, 1, 0) if e != d]
            wf = (w1[o[0]][:, None] * w1[o[1]]).reshape(-1)
            step = list(i)
            step[d] += 1
            b = at(step)
            jump, mean = {}, {}
            for e, sign, (u, du) in ((k, 1.0, face[k][d][1]), (b, -1.0, face[b][d][0])):
                jump[e] = jump.get(e, 0) + sign * u
                mean[e] = mean.get(e, 0) + 0.5 * du
            for p in jump:
                for q in jump:
                    H[p, :, q, :] += dom.alpha * (jump[p] * wf) @ jump[q].T - 0.5 * (jump[p] * wf) @ mean[q].T - 0.5 * (mean[p] * wf) @ jump[q].T
    if not case["density"]:
        return {"rows": [torch.stack([H[k, :, q, :] for q in near[k]]) for k in range(n_elem)]}
    n = n_elem * J
    A = H.reshape(n, n)
    lam, c = torch.linalg.eigh(0.5 * (A + A.T))
    c = c[:, : n // 2].reshape(n_elem, J, n // 2)
    rho = []
    for k in range(n_elem):
        # rho = sum over (j, j') of phi_j P phi_j', P the occupied projector's block
        rho.append((phis[k] * ((c[k] @ c[k].T) @ phis[k])).sum(0))
    return {"eig": lam[: n // 2].cpu().numpy(), "rho": torch.stack(rho)}
