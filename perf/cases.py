"""What is measured of this library: its public calls, over the sizes that users bring.

Molecules are synthetic (centres uniform in a ball with a 1.5 A minimum spacing, radii
U[1.2, 2.0] A, charges N(0, 0.4) e rounded to 0.01 e; 2,000 atoms in a ball of 20 A), as in the
repository's benchmark.  Solves run to a relative residual of 1e-12, so that the potential is
settled to the digits of its type, whatever the order in which a solver sums.
"""
import math

import numpy as np
import torch

import paper_2502_09323_gb300 as pb
from paper_2502_09323_gb300 import _native as N

RTOL = 1e-12
EPS_IN, EPS_OUT, SALT_M, TEMP_K = 2.0, 80.0, 0.145, 298.15
SPACING = 1.5


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # the operator alone, as a user's own Krylov or eigenvalue loop calls it: the smallest
        # call there is, and the FP32 operator of a full-size grid
        {"name": "apply_fp64_33", "kind": "apply", "nx": 33, "ny": 33, "nz": 33, "atoms": 30,
         "bc": pb.BC_ZERO, "fp32": False},
        {"name": "apply_fp32_257", "kind": "apply", "nx": 257, "ny": 257, "nz": 257, "atoms": 2000,
         "bc": pb.BC_ZERO, "fp32": True},
        # a new molecule up to its solve (grid, crossing edges, coefficients, boundary values,
        # Coulomb sums): a ragged explicit box with Debye-Hueckel boundary values, and the
        # 257^3 cube of the benchmark
        {"name": "setup_ragged_dh", "kind": "setup", "nx": 141, "ny": 95, "nz": 63, "atoms": 300,
         "bc": pb.BC_DH},
        {"name": "setup_257", "kind": "setup", "nx": 257, "ny": 257, "nz": 257, "atoms": 2000,
         "bc": pb.BC_ZERO},
        # one solve of a prepared system: a small molecule with Coulomb boundary values, a
        # ragged box, and the benchmark's 257^3 grid
        {"name": "solve_65", "kind": "solve", "nx": 65, "ny": 65, "nz": 65, "atoms": 150,
         "bc": pb.BC_COULOMB, "fp32": True},
        {"name": "solve_ragged", "kind": "solve", "nx": 150, "ny": 97, "nz": 118, "atoms": 500,
         "bc": pb.BC_DH, "fp32": True},
        {"name": "solve_257", "kind": "solve", "nx": 257, "ny": 257, "nz": 257, "atoms": 2000,
         "bc": pb.BC_ZERO, "fp32": True},
        # the plain FP64 solver, which a user takes to check the mixed one
        {"name": "solve_fp64_97", "kind": "solve", "nx": 97, "ny": 97, "nz": 97, "atoms": 400,
         "bc": pb.BC_ZERO, "fp32": False},
        # one molecule from its atoms to its energies
        {"name": "molecule_129", "kind": "molecule", "n": 129, "atoms": 1000},
        # a screening batch: uneven molecules on 0.5 A grids, solved together
        {"name": "batch_24", "kind": "batch", "count": 24, "lo": 200, "hi": 3000},
        # a large complex on a brick octree (0.25 / 0.5 / 1.0 A), from its atoms to its energies
        {"name": "octree_20000", "kind": "octree", "atoms": 20000},
        # the serving loop with its queue full: octree requests of uneven size
        {"name": "serve_8", "kind": "serve", "count": 8, "lo": 300, "hi": 5000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "setup", "solve", "solve", "molecule", "batch", "octree", "serve"])
    if kind in ("apply", "setup", "solve"):
        n = [_log(rng, 33, 257) for _ in range(3)]
        if rng.random() < 0.5:
            n = [n[0]] * 3
        c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2],
             "bc": rng.choice([pb.BC_ZERO, pb.BC_COULOMB, pb.BC_DH])}
        # about the benchmark's spacing of 0.25 to 0.5 A
        h = rng.uniform(0.25, 0.5)
        c["atoms"] = max(10, min(2000, int(2000 * (max(0.33 * h * (min(n) - 1) - 1.0, 3.0) / 20.0) ** 3)))
        if kind == "apply":
            c["fp32"] = rng.random() < 0.5
        if kind == "solve":
            c["fp32"] = rng.random() < 0.75 or n[0] * n[1] * n[2] > 4000000
        return c
    if kind == "molecule":
        return {"kind": kind, "n": _log(rng, 65, 257), "atoms": _log(rng, 100, 2000)}
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 4, 24), "lo": 200, "hi": 2500}
    if kind == "octree":
        return {"kind": kind, "atoms": _log(rng, 100, 15000)}
    return {"kind": kind, "count": rng.randint(2, 7), "lo": 300, "hi": 4000}


# ----------------------------------------------------------------- inputs --
def ball_radius(n):
    return 20.0 * (n / 2000.0) ** (1.0 / 3.0)


def molecule(n, rng):
    """(n, 5) rows x, y, z, R, 0: random sequential addition, a block of candidates at a time."""
    rb = ball_radius(n)
    cell = 0.999 * SPACING / math.sqrt(3.0)  # at most one centre per cell
    dim = int(2.0 * rb / cell) + 8
    occ = np.full(dim ** 3, -1, np.int64)
    pts = np.empty((n, 3))
    near = [(z * dim + y) * dim + x for z in range(-2, 3) for y in range(-2, 3) for x in range(-2, 3)
            if (x, y, z) != (0, 0, 0)]
    have = 0
    for _ in range(1000):
        if have == n:
            break
        m = int(1.2 * (n - have)) + 16
        v = rng.standard_normal((m, 3))
        p = v / np.linalg.norm(v, axis=1, keepdims=True) * (rb * rng.random((m, 1)) ** (1.0 / 3.0))
        k = np.floor((p + rb) / cell).astype(np.int64) + 3
        key = (k[:, 2] * dim + k[:, 1]) * dim + k[:, 0]
        first = np.sort(np.unique(key, return_index=True)[1])
        first = first[occ[key[first]] < 0]
        p, key = p[first], key[first]
        at = have + np.arange(len(key))
        every = np.concatenate([pts[:have], p])
        occ[key] = at
        good = np.ones(len(key), bool)
        for off in near:
            o = occ[key + off]
            # an earlier centre or candidate closer than the spacing
            c = (o >= 0) & (o < at)
            d = every[o[c]] - p[c]
            good[np.flatnonzero(c)[(d * d).sum(1) < SPACING * SPACING]] = False
        occ[key] = -1
        p, key = p[good][: n - have], key[good][: n - have]
        occ[key] = have + np.arange(len(key))
        pts[have: have + len(p)] = p
        have += len(p)
    if have < n:
        raise RuntimeError("no room for %d atoms" % n)
    a = np.zeros((n, 5))
    a[:, :3] = pts
    a[:, 3] = rng.uniform(1.2, 2.0, n)
    return a


def params(bc):
    return pb.Params(eps_in=EPS_IN, eps_out=EPS_OUT, ionic_strength_M=SALT_M, temperature_K=TEMP_K, bc=bc)


def opts(mixed=True):
    return pb.SolveOpts(precision=pb.MIXED if mixed else pb.FP64, rtol=RTOL)


def box(case):
    """An explicit grid around the molecule: its shortest side is 1.5 times the molecule."""
    n = (case["nx"], case["ny"], case["nz"])
    h = 3.0 * (ball_radius(case["atoms"]) + 2.0) / (min(n) - 1)
    return pb.GridSpec(n=n, origin=tuple(-0.5 * h * (m - 1) for m in n), h=h, fill=0.0)


def screen_spec(atoms):
    """A 0.5 A grid of 32 k + 1 nodes per axis that is 1.5 times the molecule."""
    lo = (atoms[:, :3] - atoms[:, 3:4]).min(0)
    hi = (atoms[:, :3] + atoms[:, 3:4]).max(0)
    n = 32 * max(2, math.ceil(3.0 * (ball_radius(len(atoms)) + 2.0) / 0.5 / 32.0)) + 1
    o = 0.5 * (lo + hi) - 0.25 * (n - 1)
    return pb.GridSpec(n=(n, n, n), origin=tuple(float(x) for x in o), h=0.5, fill=0.0)


def sizes(case):
    u = np.random.default_rng(4000 + case["count"]).random(case["count"])
    return np.exp(math.log(case["lo"]) + u * math.log(case["hi"] / case["lo"])).astype(int)


def molecules(case, seed):
    """The molecules of a case.  Their shapes belong to the case, so that lists of surface points
    and bricks have one length; the seed mirrors them and gives them their charges."""
    shape, rng = np.random.default_rng(1000 + case.get("atoms", 0) + case.get("count", 0)), np.random.default_rng(seed)
    out = []
    for n in sizes(case) if "count" in case else [case["atoms"]]:
        a = molecule(int(n), shape)
        a[:, :3] *= rng.choice([-1.0, 1.0], 3)
        a[:, 4] = np.round(rng.normal(0.0, 0.4, len(a)), 2)
        out.append(a)
    return out


def prepare(case, seed):
    kind = case["kind"]
    mols = molecules(case, seed)
    s = {"kind": kind, "case": case, "mols": mols}
    if kind in ("apply", "solve"):
        g = pb.pb_build_grid(box(case), mols[0])
        s["system"] = pb.pb_assemble_coeffs(g, params(case["bc"]))
    if kind == "apply":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s["x"] = torch.randn(g.N, generator=gen, device="cuda",
                             dtype=torch.float32 if case["fp32"] else torch.float64)
    if kind == "solve":
        s["phi"] = torch.empty(g.N, dtype=torch.float64, device="cuda")
    if kind == "batch":
        s["systems"] = [pb.pb_assemble_coeffs(pb.pb_build_grid(screen_spec(a), a), params(pb.BC_ZERO))
                        for a in mols]
    if kind == "serve":
        from paper_2502_09323_gb300 import serving
        s["serving"] = serving
        s["server"] = serving.Server(capacity=64, params=params(pb.BC_ZERO), opts=opts(), h=0.25,
                                     grid="octree")
    return s


# -------------------------------------------------------------------- run --
_DTYPES = {np.float64: torch.float64, np.int64: torch.int64, np.uint8: torch.uint8, np.int8: torch.int8}


def fetch(obj, name):
    """One array of a grid or system in a new device tensor (the C call with a device target)."""
    which, dtype, kind = pb._ARRAYS[name]
    g, s = (obj.grid, obj) if isinstance(obj, pb.System) else (obj, None)
    n = {"N": g.info.n_nodes, "nc": g.info.n_cross, "nc3": 3 * g.info.n_cross}[kind]
    out = torch.empty(int(n), dtype=_DTYPES[dtype], device="cuda")
    if n:
        N.check(N.lib().pb_get_array(g.handle, s.handle if s else None, which, out.data_ptr(),
                                     out.numel() * out.element_size(), N.DEVICE,
                                     torch.cuda.current_stream().cuda_stream))
    return out


GRID_OUT = ("inside", "cross_id", "cross_alpha", "cross_rp", "cross_sign", "mc_weight", "mc_normal")
SYS_OUT = ("Wx", "Wy", "Wz", "diag", "rhs", "bc", "phi_surf", "psi_surf", "psi_n")


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "apply":
        return pb.pb_apply(s["system"], s["x"], pb.MIXED if case["fp32"] else pb.FP64)
    if kind == "setup":
        g = pb.pb_build_grid(box(case), s["mols"][0])
        y = pb.pb_assemble_coeffs(g, params(case["bc"]))
        pb.pb_coulomb_terms(y, pb.CT_SURFACE | pb.CT_PAIRS)
        out = {k: fetch(g, k) for k in GRID_OUT}
        out.update({k: fetch(y, k) for k in SYS_OUT})
        return out
    if kind == "solve":
        pb.pb_solve(s["system"], opts(case["fp32"]), phi_out=s["phi"])
        return s["phi"]
    if kind == "molecule":
        r = pb.solve_molecule(s["mols"][0], n=case["n"], fill=1.5, params=params(pb.BC_ZERO), opts=opts())
        return {"energy": r["energy"], "phi": fetch(r["system"], "phi")}
    if kind == "batch":
        pb.pb_solve_batch(s["systems"], opts())
        return [fetch(y, "phi") for y in s["systems"]]
    if kind == "octree":
        r = pb.solve_molecule(s["mols"][0], spec=pb.OctreeSpec(), params=params(pb.BC_ZERO), opts=opts())
        return {"energy": r["energy"], "phi": fetch(r["system"], "phi")}
    rec = s["server"].run([s["serving"].Request(rid=i, atoms=a, arrival_s=0.0) for i, a in enumerate(s["mols"])])
    return [r["energy"] for r in sorted(rec, key=lambda r: r["rid"])]


# ------------------------------------------------------------------- work --
def _nodes(n_atoms, h):
    """Nodes of a cube of spacing h that is 1.5 times a molecule."""
    return (3.0 * (ball_radius(n_atoms) + 1.6) / h + 1.0) ** 3


def work(case):
    # bytes: a solve reads the operator (three weights and a diagonal), the right-hand side and
    # writes the potential; a set-up writes what the solve reads.  flops: the operator once per
    # decimal digit of a solve; 20 a pair for the Coulomb sums at the surface points (290 an
    # atom at 0.25 A).
    kind = case["kind"]
    digits = -math.log10(RTOL)
    solve = lambda nodes: (48.0 * nodes, 14.0 * digits * nodes)  # noqa: E731
    pairs = lambda a, h: 20.0 * 290.0 * a * a * (0.25 / h) ** 2  # noqa: E731
    if kind in ("apply", "setup", "solve"):
        nodes = float(case["nx"] * case["ny"] * case["nz"])
        if kind == "apply":  # x, y and what the operator needs: a byte a node, or its four arrays
            return {"bytes": nodes * (9.0 if case["fp32"] else 48.0), "flops": 14.0 * nodes}
        if kind == "solve":
            b, f = solve(nodes)
            return {"bytes": b, "flops": f}
        return {"bytes": 49.0 * nodes, "flops": pairs(case["atoms"], box(case).h)}
    if kind == "molecule":
        b, f = solve(float(case["n"]) ** 3)
        h = 3.0 * (ball_radius(case["atoms"]) + 1.6) / (case["n"] - 1)
        return {"bytes": b, "flops": f + pairs(case["atoms"], h)}
    if kind == "batch":
        every = [solve(_nodes(int(a), 0.5)) for a in sizes(case)]
        return {"bytes": sum(b for b, _ in every), "flops": sum(f for _, f in every)}
    # octree: two shells of 3 A about the surface at 0.25 A, about 2,080 unknowns an atom at
    # 20,000 atoms and more for small molecules
    atoms = [case["atoms"]] if kind == "octree" else \
        [int(a) for a in sizes(case)]
    b = f = 0.0
    for a in atoms:
        nodes = 4.0 / 3.0 * math.pi * ((ball_radius(a) + 5.0) / 0.25) ** 3
        bb, ff = solve(nodes)
        b, f = b + bb, f + ff + pairs(a, 0.25)
    return {"bytes": b, "flops": f}


# ------------------------------------------------- the same in plain torch --
E_CHARGE, K_BOLTZ, EPS0, AVOGADRO = 1.602176634e-19, 1.380649e-23, 8.8541878128e-12, 6.02214076e23
L_B = E_CHARGE ** 2 / (4.0 * math.pi * EPS0 * K_BOLTZ * TEMP_K) * 1e10
# 1:1 salt: eps_s k_D^2 = 2 N_A 10^3 I e^2 / (eps_0 k_B T), in 1/A^2
KAP2 = 2.0 * AVOGADRO * 1e3 * SALT_M * E_CHARGE ** 2 / (EPS0 * K_BOLTZ * TEMP_K) * 1e-20


class Plain:
    """Grid, coefficients, sums and solve of one molecule in 64 bits, with torch alone."""

    def __init__(self, atoms, n, origin, h, bc):
        self.n, self.o, self.h, self.bc = n, origin, h, bc
        self.a = torch.from_numpy(atoms).cuda()
        self.nx, self.ny, self.nz = n
        self.N = n[0] * n[1] * n[2]
        self.stride = (1, n[0], n[0] * n[1])
        self._inside()
        self._edges()

    def _inside(self):
        a, h = self.a, self.h
        m = int(float(a[:, 3].max()) / h) + 2
        r = torch.arange(-m, m + 1, device="cuda")
        dz, dy, dx = (t.reshape(-1) for t in torch.meshgrid(r, r, r, indexing="ij"))
        self.inside = torch.zeros(self.N, dtype=torch.bool, device="cuda")
        for q in torch.split(a, max(1, 4_000_000 // dx.numel())):
            idx, d2 = [], 0.0
            ok = True
            for d, off in enumerate((dx, dy, dz)):
                c = torch.round((q[:, d] - self.o[d]) / h).long()[:, None] + off[None]
                x = self.o[d] + c.double() * h - q[:, d, None]
                d2 = d2 + x * x
                ok = ok & (c >= 0) & (c < self.n[d])
                idx.append(c)
            ok = ok & (d2 < (q[:, 3] ** 2)[:, None])
            node = (idx[2] * self.ny + idx[1]) * self.nx + idx[0]
            self.inside[node[ok]] = True

    def _along(self, d):
        """(edge node, t0, t1) of the pieces that single balls cover of edges along axis d."""
        a, h = self.a, self.h
        e, f = [x for x in range(3) if x != d]
        m = int(float(a[:, 3].max()) / h) + 2
        r = torch.arange(-m, m + 1, device="cuda")
        df, de, dd = (t.reshape(-1) for t in torch.meshgrid(r, r, r, indexing="ij"))
        found = []
        for q in torch.split(a, max(1, 4_000_000 // dd.numel())):
            ci = [torch.round((q[:, x] - self.o[x]) / h).long()[:, None] for x in range(3)]
            ce, cf, cd = ci[e] + de, ci[f] + df, ci[d] + dd
            xe = self.o[e] + ce.double() * h - q[:, e, None]
            xf = self.o[f] + cf.double() * h - q[:, f, None]
            s2 = (q[:, 3] ** 2)[:, None] - (xe * xe + xf * xf)
            s = s2.clamp(min=0.0).sqrt()
            x0 = q[:, d, None] - (self.o[d] + cd.double() * h)
            t0, t1 = ((x0 - s) / h).clamp(min=0.0), ((x0 + s) / h).clamp(max=1.0)
            ok = (s2 > 0) & (t1 > t0) & (ce >= 0) & (ce < self.n[e]) & (cf >= 0) & (cf < self.n[f])
            ok &= (cd >= 0) & (cd < self.n[d] - 1)
            c = [None] * 3
            c[d], c[e], c[f] = cd, ce, cf
            node = (c[2] * self.ny + c[1]) * self.nx + c[0]
            found.append((node[ok], t0[ok], t1[ok]))
        return [torch.cat(x) for x in zip(*found)]

    def _edges(self):
        ids, alpha = [], []
        self.W = []
        i = torch.arange(self.N, device="cuda")
        coord = (i % self.nx, (i // self.nx) % self.ny, i // (self.nx * self.ny))
        for d in range(3):
            node, t0, t1 = self._along(d)
            node, order = torch.sort(node)
            t0, t1 = t0[order], t1[order]
            edge, inv, cnt = torch.unique_consecutive(node, return_inverse=True, return_counts=True)
            place = torch.arange(node.numel(), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[inv]
            K = int(cnt.max())
            lo = torch.full((edge.numel(), K), 2.0, dtype=torch.float64, device="cuda")
            hi = lo.clone()
            lo[inv, place], hi[inv, place] = t0, t1
            lo, by = torch.sort(lo, dim=1)
            hi = torch.gather(hi, 1, by)
            cover, reach = torch.zeros_like(lo[:, 0]), torch.zeros_like(lo[:, 0])
            for k in range(K):
                real = lo[:, k] < 1.5
                cover += torch.where(real, (hi[:, k] - torch.maximum(lo[:, k], reach)).clamp(min=0.0), 0.0)
                reach = torch.where(real, torch.maximum(reach, hi[:, k]), reach)
            cover = torch.where(cover > 1.0 - 1e-12, 1.0, cover)
            al = torch.zeros(self.N, dtype=torch.float64, device="cuda")
            al[edge] = cover
            ex = coord[d] < self.n[d] - 1
            there = torch.zeros_like(self.inside)
            there[: self.N - self.stride[d]] = self.inside[self.stride[d]:]
            mixed = ex & (self.inside != there)
            mark = ex & (mixed | ((al > 0.0) & (al < 1.0)))
            at = torch.nonzero(mark).reshape(-1)
            ids.append(at + d * self.N)
            alpha.append(al[at])
            w = self.h * torch.where(self.inside, EPS_IN, EPS_OUT).double()
            w[at] = 1.0 / (al[at] / EPS_IN + (1.0 - al[at]) / EPS_OUT) * self.h
            self.W.append(torch.where(ex, w, 0.0))
        self.id, self.alpha = torch.cat(ids), torch.cat(alpha)
        self.coord = coord
        self.face = torch.zeros_like(self.inside)
        for d in range(3):
            self.face |= (coord[d] == 0) | (coord[d] == self.n[d] - 1)
        # crossing points and signs
        d = self.id // self.N
        lo = self.id % self.N
        hi = lo + torch.tensor(self.stride, device="cuda")[d]
        a, b = self.inside[lo], self.inside[hi]
        self.sign = (a & ~b).to(torch.int8) - (b & ~a).to(torch.int8)
        at = torch.where(self.sign > 0, self.alpha, torch.where(self.sign < 0, 1.0 - self.alpha, 0.5))
        x = torch.stack([self.o[k] + coord[k][lo].double() * self.h for k in range(3)], 1)
        x[torch.arange(len(d), device="cuda"), d] += at * self.h
        self.rp, self.d, self.lo, self.hi = x, d, lo, hi
        kap = KAP2 * self.h ** 3 * (~self.inside).double()
        diag = torch.zeros(self.N, dtype=torch.float64, device="cuda")
        for k in range(3):
            diag += self.W[k]
            diag[self.stride[k]:] += self.W[k][: -self.stride[k]]
        self.diag = torch.where(self.face, 0.0, diag + kap)

    def rhs(self):
        a, h = self.a, self.h
        f = torch.zeros(self.N, dtype=torch.float64, device="cuda")
        u = [(a[:, d] - self.o[d]) / h for d in range(3)]
        c = [x.floor().long().clamp(0, self.n[d] - 2) for d, x in enumerate(u)]
        t = [x - y.double() for x, y in zip(u, c)]
        for k in range(8):
            b = (k & 1, (k >> 1) & 1, k >> 2)
            node = ((c[2] + b[2]) * self.ny + c[1] + b[1]) * self.nx + c[0] + b[0]
            w = 4.0 * math.pi * L_B * a[:, 4]
            for d in range(3):
                w = w * (t[d] if b[d] else 1.0 - t[d])
            f.index_add_(0, node, w)
        self.g = torch.zeros_like(f)
        if self.bc != pb.BC_ZERO:
            at = torch.nonzero(self.face).reshape(-1)
            k_d = math.sqrt(KAP2 / EPS_OUT) if self.bc == pb.BC_DH else 0.0
            x = torch.stack([self.o[d] + self.coord[d][at].double() * h for d in range(3)], 1)
            got = []
            for q in torch.split(x, 20_000_000 // len(a) + 1):
                r = torch.sqrt(((q[:, None] - a[None, :, :3]) ** 2).sum(2))
                got.append((L_B / EPS_OUT * a[:, 4] * torch.exp(-k_d * r) / r).sum(1))
            self.g[at] = torch.cat(got)
            lift = torch.zeros_like(f)
            for d in range(3):
                s = self.stride[d]
                lift[:-s] += self.W[d][:-s] * self.g[s:]
                lift[s:] += self.W[d][:-s] * self.g[:-s]
            f = f + lift
        return torch.where(self.face, 0.0, f)

    def apply(self, x):
        x = torch.where(self.face, 0.0, x)
        y = self.diag * x
        for d in range(3):
            s = self.stride[d]
            y[:-s] -= self.W[d][:-s] * x[s:]
            y[s:] -= self.W[d][:-s] * x[:-s]
        return torch.where(self.face, 0.0, y)

    def solve(self):
        f = self.rhs()
        dinv = torch.where(self.face, 0.0, 1.0 / self.diag.clamp(min=1e-300))
        x, r = torch.zeros_like(f), f.clone()
        z = dinv * r
        p, rho, f2 = z.clone(), torch.dot(r, z), torch.dot(f, f)
        for it in range(5000):
            q = self.apply(p)
            alpha = rho / torch.dot(p, q)
            x += alpha * p
            r -= alpha * q
            if it % 20 == 0 and float(torch.dot(r, r) / f2) < 1e-28:
                break
            z = dinv * r
            rho, old = torch.dot(r, z), rho
            p = z + rho / old * p
        return x + self.g

    def surface(self):
        """Phi and Psi (along the edge, outward) at the crossing points of the flux edges."""
        phi = torch.zeros(len(self.id), dtype=torch.float64, device="cuda")
        psi = torch.zeros_like(phi)
        a = self.a
        for at in torch.split(torch.nonzero(self.sign).reshape(-1), 20_000_000 // len(a) + 1):
            v = self.rp[at][:, None] - a[None, :, :3]
            r = torch.sqrt((v * v).sum(2))
            phi[at] = (a[:, 4] / r).sum(1)
            along = torch.gather(v, 2, self.d[at][:, None, None].expand(-1, len(a), 1))[:, :, 0]
            psi[at] = self.sign[at].double() * (a[:, 4] * along / r ** 3).sum(1)
        return phi, psi

    def energy(self, u):
        phi, psi = self.surface()
        inn, out = torch.where(self.sign >= 0, self.lo, self.hi), torch.where(self.sign >= 0, self.hi, self.lo)
        w = torch.stack(self.W)[self.d, self.lo]
        flux = torch.where(self.sign != 0, w * (u[inn] - u[out]), 0.0)
        S = float((flux * phi).sum()) / (4.0 * math.pi)
        a = self.a
        coul = 0.0
        for k in range(0, len(a), 500):
            r = torch.cdist(a[k:k + 500, :3], a[:, :3], compute_mode="donot_use_mm_for_euclid_dist")
            qq = a[k:k + 500, 4, None] * a[None, :, 4]
            i = torch.arange(k, min(k + 500, len(a)), device="cuda")[:, None]
            coul += float(torch.where(i < torch.arange(len(a), device="cuda")[None], qq / r, 0.0).sum())
        return {"e_coul": L_B / EPS_IN * coul, "e_pol": 0.5 * (1.0 / EPS_OUT - 1.0 / EPS_IN) * S,
                "e_ion_flux": -0.5 * S / EPS_OUT, "e_ion_surf": None, "e_ion_mc": None, "e_total": None,
                "flux_charge": float(flux.sum()) / (4.0 * math.pi * L_B)}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("octree", "serve"):  # a composite grid with hanging nodes
        return None
    mols = molecules(case, seed)
    if kind == "batch":
        out = []
        for a in mols:
            s = screen_spec(a)
            out.append(Plain(a, s.n, s.origin, s.h, pb.BC_ZERO).solve())
        return out
    if kind == "molecule":
        a, n = mols[0], case["n"]
        lo, hi = (a[:, :3] - a[:, 3:4]).min(0), (a[:, :3] + a[:, 3:4]).max(0)
        side = 1.5 * float((hi - lo).max())
        p = Plain(a, (n, n, n), tuple(float(v) for v in 0.5 * (lo + hi) - 0.5 * side), side / (n - 1), pb.BC_ZERO)
        u = p.solve()
        return {"energy": p.energy(u), "phi": u}
    s = box(case)
    p = Plain(mols[0], s.n, s.origin, s.h, case["bc"])
    if kind == "apply":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(p.N, generator=gen, device="cuda",
                        dtype=torch.float32 if case["fp32"] else torch.float64)
        return p.apply(x.double())
    if kind == "solve":
        return p.solve()
    phi, psi = p.surface()
    f = p.rhs()
    return {"inside": p.inside.to(torch.uint8), "cross_id": p.id, "cross_alpha": p.alpha,
            "cross_rp": p.rp.reshape(-1), "cross_sign": p.sign, "mc_weight": None, "mc_normal": None,
            "Wx": p.W[0], "Wy": p.W[1], "Wz": p.W[2], "diag": p.diag, "rhs": f, "bc": p.g,
            "phi_surf": phi, "psi_surf": psi, "psi_n": None}
