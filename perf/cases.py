"""The work a user of the library has it do, as cases that can be timed: one
V-cycle or one whole solve on a mesh the user keeps, with new data every time,
through the Python binding.  Sizes follow the tests and the benchmark: cubes of
1 to 64 sub-cubes of six macro-tetrahedra, refined 3 to 8 times.
"""

import itertools
import math

import numpy as np
import torch

from paper_1506_06185_gb300 import autograd, hhg

SHEAR = [[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]]
RECOVERY = {"none": hhg.HHG_RECOVERY_NONE, "lr": hhg.HHG_RECOVERY_LR, "dd": hhg.HHG_RECOVERY_DD,
            "dn": hhg.HHG_RECOVERY_DN}


def _case(name, call, sub, levels, **kw):
    c = {"name": name, "call": call, "sx": sub[0], "sy": sub[1], "sz": sub[2], "levels": levels,
         "shape": "cube",          # cube | sheared | corners (moved sub-cube corners)
         "coeff": "one",           # one | lognormal, per macro-tetrahedron
         "tuned": False,           # the mesh was autotuned after its creation
         "mixed": False, "recovery": "none", "rtol": 1e-8}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest mesh of the tests: nothing but launches, the coarse solve and the read-back
        _case("cycle_smallest", "cycle", (1, 1, 1), 3),
        # the paper's small experiment: a fault in one tetrahedron, two local recovery cycles
        _case("solve_small_lr", "solve", (2, 2, 2), 4, recovery="lr", rtol=1e-10),
        # an ordinary cycle on a box whose sides differ (three different stencil weights, ragged work lists)
        _case("cycle_box", "cycle", (3, 2, 1), 6),
        # a tuned mesh of 27 sub-cubes, Dirichlet-Neumann recovery of one macro in the middle
        _case("solve_dn", "solve", (3, 3, 3), 6, tuned=True, recovery="dn"),
        # the benchmark's workload: FP64, one sub-cube lost, Dirichlet-Dirichlet recovery
        _case("solve_large_dd", "solve", (2, 2, 2), 8, tuned=True, recovery="dd"),
        # the same in FP32 cycles inside FP64 iterative refinement
        _case("solve_large_mixed", "solve", (2, 2, 2), 8, tuned=True, recovery="dd", mixed=True),
        # a service that gets its right-hand side on the host and sends the solution back there
        _case("solve_from_host", "solve_host", (2, 2, 2), 7, tuned=True, mixed=True),
        # a sheared domain with a coefficient per macro: all 15 stencil weights
        _case("cycle_sheared", "cycle", (2, 2, 2), 7, shape="sheared", coeff="lognormal"),
        # a polyhedral domain of general tetrahedra, solved
        _case("solve_corners", "solve", (2, 2, 1), 6, shape="corners"),
        # an unstructured macro mesh given as vertices and tetrahedra, with local recovery
        _case("solve_general", "solve_general", (2, 2, 1), 5, shape="corners", recovery="lr"),
        # gradients with respect to the load and the coefficients: forward and adjoint solve
        _case("gradient", "gradient", (4, 4, 4), 5, coeff="lognormal", tuned=True, rtol=1e-10),
        # many small recovery problems at once, one persistent launch
        _case("batch_small", "batch", (2, 1, 1), 5, tasks=48, cycles=3),
    ]


def draw(rng):
    call = rng.choice(["cycle", "cycle", "cycle15", "solve", "solve", "mixed", "host", "corners", "general",
                       "gradient", "batch"])
    pick = lambda n: (rng.randint(1, n), rng.randint(1, n), rng.randint(1, n))  # noqa: E731
    rec = rng.choice(["none", "lr", "dd", "dn"])
    tuned = rng.random() < 0.5
    rtol = 10.0 ** -rng.randint(6, 10)
    if call == "cycle":
        c = _case("", "cycle", pick(4), rng.randint(3, 6), tuned=tuned, coeff=rng.choice(["one", "lognormal"]))
    elif call == "cycle15":
        c = _case("", "cycle", pick(3), rng.randint(3, 6), shape=rng.choice(["sheared", "corners"]),
                  coeff=rng.choice(["one", "lognormal"]))
    elif call == "solve":
        c = _case("", "solve", pick(3), rng.randint(4, 7), tuned=tuned, recovery=rec, rtol=rtol)
    elif call == "mixed":
        c = _case("", "solve", pick(3), rng.randint(4, 7), tuned=tuned, recovery=rec, mixed=True, rtol=rtol)
    elif call == "host":
        c = _case("", "solve_host", pick(3), rng.randint(4, 7), tuned=tuned, mixed=rng.random() < 0.5, rtol=rtol)
    elif call == "corners":
        c = _case("", "solve", pick(2), rng.randint(4, 6), shape="corners", rtol=rtol)
    elif call == "general":
        c = _case("", "solve_general", pick(2), rng.randint(3, 5), shape="corners", rtol=rtol,
                  recovery=rng.choice(["none", "lr", "dd"]))
    elif call == "gradient":
        c = _case("", "gradient", pick(4), rng.randint(3, 5), coeff="lognormal", tuned=tuned, rtol=1e-10)
    else:
        c = _case("", "batch", (rng.randint(1, 2), 1, 1), rng.randint(4, 5), tasks=rng.randint(8, 60),
                  cycles=rng.randint(1, 4))
    del c["name"]
    return c


# --- inputs -------------------------------------------------------------------

def _sub(case):
    return case["sx"], case["sy"], case["sz"]


def _n_macro(case):
    return 6 * case["sx"] * case["sy"] * case["sz"]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _corners(case):
    """Positions of the sub-cube corners, moved by up to 0.12 of an edge."""
    s = _sub(case)
    z, y, x = np.meshgrid(*(np.arange(n + 1) for n in reversed(s)), indexing="ij")
    pos = np.stack([x / s[0], y / s[1], z / s[2]], -1)
    return pos + np.random.default_rng(7).uniform(-0.12, 0.12, pos.shape) / np.array(s)


def _coeff(case, seed):
    if case["coeff"] == "one":
        return None
    return np.exp(np.random.default_rng(seed).standard_normal(_n_macro(case)))


def _tets(case):
    """The macro-tetrahedra of every sub-cube as corner ids."""
    sx, sy, sz = _sub(case)
    out = []
    for c, b, a in itertools.product(range(sz), range(sy), range(sx)):
        for p in itertools.permutations(range(3)):
            v, tet = [a, b, c], []
            for step in (None, *p):
                if step is not None:
                    v[step] += 1
                tet.append((v[2] * (sy + 1) + v[1]) * (sx + 1) + v[0])
            out.append(tet)
    return np.array(out, dtype=np.int32)


def _fault(case):
    """The macros lost: a sub-cube (DD, LR on larger meshes), or one macro."""
    n = _n_macro(case)
    if case["recovery"] == "dn":
        return [n // 2]
    return [0] if case["levels"] <= 4 or n <= 6 else list(range(6))


def _solve_args(case):
    kw = dict(rtol=case["rtol"], max_cycles=80, mixed_precision=case["mixed"])
    if case["recovery"] != "none":
        kw.update(fault_cycle=3, fault_ids=_fault(case), recovery=RECOVERY[case["recovery"]])
        kw.update(dict(n_local=2) if case["recovery"] == "lr" else dict(n_global=3, eta=4.0))
    return kw


def _grid(case):
    N = 1 << case["levels"]
    return tuple(s * N + 1 for s in reversed(_sub(case)))


def _inner(shape):
    return tuple(slice(1, n - 1) for n in shape)


def _fields(case, seed, shape):
    """A random load, zero on the boundary, and an iterate with smooth
    Dirichlet values: zero inside, but for a batch, whose faults erase parts
    of a smooth iterate."""
    f = torch.zeros(shape, dtype=torch.float64, device="cuda")
    i = _inner(shape)
    f[i] = torch.rand(f[i].shape, generator=_gen(seed), dtype=torch.float64, device="cuda") * 2 - 1
    z, y, x = (torch.linspace(0, 1, n, dtype=torch.float64, device="cuda") for n in shape)
    u = torch.exp(x)[None, None, :] * torch.cos(y)[None, :, None] * (1 + z)[:, None, None] * float(shape[0]) ** -1
    if case["call"] != "batch":
        u[i] = 0
    return f, u.contiguous()


def _mesh(case, seed):
    kw = {"precision": 32 if case["mixed"] else 64, "coeff": _coeff(case, seed)}
    if case["shape"] == "sheared":
        kw["affine"] = np.array(SHEAR)
    elif case["shape"] == "corners":
        kw["vertex_pos"] = _corners(case)
    M = hhg.Mesh(_sub(case), case["levels"], **kw)
    if case["tuned"]:
        hhg.hhg_autotune(M.h, case["levels"] - 1)
    return M


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        tasks, fields = [], []
        for t in range(case["tasks"]):
            sub = (case["sx"] if t % 2 else 1, 1, 1)
            one = dict(case, sx=sub[0])
            M = hhg.Mesh(sub, case["levels"])
            f, u0 = _fields(one, seed * 1000 + t, M.shape)
            M.set_problem(f, u0)
            tasks.append((M, _task_fault(one, t), case["cycles"]))
            fields.append((f, u0, torch.empty_like(f)))
        return {"case": case, "tasks": tasks, "fields": fields, "batch": hhg.Batch(tasks)}
    if call == "solve_general":
        M = hhg.Mesh.general(_corners(case).reshape(-1, 3), _tets(case), case["levels"])
        f, u0 = _fields(case, seed, _grid(case))
        ids = torch.from_numpy(_general_nodes(case)).cuda()
        f, u0 = f.reshape(-1)[ids].contiguous(), u0.reshape(-1)[ids].contiguous()
    else:
        M = _mesh(case, seed)
        f, u0 = _fields(case, seed, M.shape)
    st = {"case": case, "mesh": M, "f": f, "u0": u0}
    if call == "solve_host":
        st.update({k: st[k].cpu().pin_memory() for k in ("f", "u0")})
        st["out"] = torch.empty(M.shape, dtype=torch.float64, pin_memory=True)
    elif call == "gradient":
        st["k"] = torch.from_numpy(_coeff(case, seed)).cuda()
        st["target"] = torch.rand(M.shape, generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
    else:
        st["out"] = torch.empty_like(f)
    return st


def _task_fault(case, t):
    """A fault of one or two macros of a small batch problem."""
    r = np.random.default_rng(t)
    return sorted({int(v) for v in r.integers(0, _n_macro(case), size=2)})


# --- one pass -----------------------------------------------------------------

def run(st):
    case = st["case"]
    if case["call"] == "batch":
        for (M, _, _), (f, u0, _) in zip(st["tasks"], st["fields"]):
            M.set_problem(f, u0)
        st["batch"].launch_persistent(timed=False)
        return {"u": [M.get_solution(out) for (M, _, _), (_, _, out) in zip(st["tasks"], st["fields"])]}
    M = st["mesh"]
    if case["call"] == "gradient":
        f, k = st["f"].detach().requires_grad_(), st["k"].detach().requires_grad_()
        u = autograd.solve(M, f, k, g=st["u0"], rtol=case["rtol"])
        df, dk = torch.autograd.grad(0.5 * ((u - st["target"]) ** 2).sum(), (f, k))
        return {"u": u.detach(), "df": df, "dk": dk}
    M.set_problem(st["f"], st["u0"])
    if case["call"] == "cycle":
        res = M.vcycle()
        return {"u": M.get_solution(st["out"]), "res": res}
    M.solve(**_solve_args(case))
    return {"u": M.get_solution(st["out"])}


def work(case):
    """The load and the iterate read, the solution written; the arithmetic of
    the V(3,3) cycles (24 Gauss-Seidel colour sweeps, a residual, transfers, on
    all levels) that bring a random load's residual to rtol."""
    n = math.prod(_grid(case))
    seven = case["shape"] == "cube"
    per_cycle = (6 * 12 + 14 + 15 if seven else 6 * 28 + 30 + 15) * 8 / 7 * n
    if case["call"] == "batch":
        n_all = sum(math.prod(_grid(dict(case, sx=case["sx"] if t % 2 else 1))) for t in range(case["tasks"]))
        # a task's cycles run on one or two of its 6 or 12 macros
        return {"bytes": 24.0 * n_all, "flops": per_cycle / n * n_all * case["cycles"] / 6}
    cycles = 1 if case["call"] == "cycle" else math.ceil(math.log(case["rtol"]) / math.log(0.12 if seven else 0.33))
    if case["call"] == "gradient":
        return {"bytes": 40.0 * n, "flops": 2.0 * cycles * per_cycle}
    return {"bytes": 24.0 * n, "flops": float(cycles * per_cycle)}


# --- the same in plain torch, 64 bits -------------------------------------------

OFFS = [o for o in itertools.product((0, 1), repeat=3) if any(o)]
OFFS = OFFS + [tuple(-v for v in o) for o in OFFS]          # (x, y, z) edges of the Freudenthal triangulation
PERMS = list(itertools.permutations(range(3)))


def _at(a, off):
    """The values at the interior nodes' neighbours (x, y, z) + off."""
    n = a.shape
    return a[tuple(slice(1 + o, n[q] - 1 + o) for q, o in enumerate(reversed(off)))]


class _Level:
    def __init__(self, sub, r, B, k, faulty=None):
        """B: (macro, 3, 3) image of a sub-cube's axes in each macro; k: its
        coefficients; faulty: the unknowns are those strictly inside them."""
        N = 1 << r
        nx, ny, nz = (s * N for s in sub)
        self.shape = (nz + 1, ny + 1, nx + 1)
        cell = [torch.arange(n, device="cuda") for n in (nx, ny, nz)]
        box = [c // N for c in cell]
        sc = (box[2][:, None, None] * sub[1] + box[1][None, :, None]) * sub[0] + box[0][None, None, :]
        loc = [4 * (c % N) for c in cell]
        gref = torch.zeros(6, 4, 3, dtype=torch.float64, device="cuda")
        verts = []
        for p, (a, b, c) in enumerate(PERMS):
            for v, ax, s in ((0, a, -1), (1, a, 1), (1, b, -1), (2, b, 1), (2, c, -1), (3, c, 1)):
                gref[p, v, ax] += s
            v = np.zeros((4, 3), int)
            v[1:, a] += 1
            v[2:, b] += 1
            v[3:, c] += 1
            verts.append(v)
        G = torch.einsum("mij,pvj->mpvi", torch.linalg.inv(B).transpose(1, 2), gref)
        vol = torch.linalg.det(B).abs() / (6 * N)
        self.K = torch.einsum("mpvi,mpwi,m->mpvw", G, G, vol)           # without the coefficient
        Kk = self.K * k[:, None, None, None]
        self.verts, self.macro = verts, []
        W = {o: None for o in [(0, 0, 0)] + OFFS}
        full = {o: torch.zeros(self.shape, dtype=torch.float64, device="cuda") for o in W}
        healthy = torch.zeros(self.shape, dtype=torch.bool, device="cuda") if faulty is not None else None
        for p, (a, b, c) in enumerate(PERMS):
            bx, by, bz = (loc[q] + (3, 2, 1)[PERMS[p].index(q)] for q in range(3))
            bx, by, bz = bx[None, None, :], by[None, :, None], bz[:, None, None]
            xy, yz, xz = bx > by, by > bz, bx > bz
            perm = torch.where(xy, torch.where(yz, 0, torch.where(xz, 1, 4)), torch.where(xz, 2, torch.where(yz, 3, 5)))
            macro = 6 * sc + perm
            self.macro.append(macro)
            for v, w in itertools.product(range(4), repeat=2):
                val = Kk[:, p, v, w]
                if not bool(val.any()):
                    continue
                off = tuple(int(t) for t in verts[p][w] - verts[p][v])
                full[off][self._cells(verts[p][v])] += val[macro]
            if faulty is not None:
                bad = ~faulty[macro]
                for v in range(4):
                    healthy[self._cells(verts[p][v])] |= bad
        i = _inner(self.shape)
        scale = float(full[(0, 0, 0)].abs().max())
        for o in W:
            w = full.pop(o)[i]
            W[o] = w.contiguous() if float(w.abs().max()) > 1e-13 * scale else None
        self.diag, self.W = W.pop((0, 0, 0)), {o: w for o, w in W.items() if w is not None}
        zi, yi, xi = (torch.arange(1, n - 1, device="cuda") for n in self.shape)
        colour = (zi[:, None, None] + yi[None, :, None] + xi[None, None, :]) % 4
        self.free = ~healthy[i] if faulty is not None else torch.ones_like(colour, dtype=torch.bool)
        self.colours = [(colour == c) & self.free for c in range(4)]

    def _cells(self, v):
        return tuple(slice(int(o), n - 1 + int(o)) for o, n in zip(reversed(v), self.shape))

    def off(self, u):
        s = torch.zeros_like(self.diag)
        for o, w in self.W.items():
            s.addcmul_(w, _at(u, o))
        return s

    def smooth(self, u, f, steps):
        i = _inner(self.shape)
        for _ in range(steps):
            for m in self.colours:
                u[i] = torch.where(m, (f[i] - self.off(u)) / self.diag, u[i])

    def residual(self, u, f):
        i = _inner(self.shape)
        r = torch.zeros_like(f)
        r[i] = torch.where(self.free, f[i] - self.diag * u[i] - self.off(u), 0.0)
        return r

    def dense(self):
        n = self.diag.numel()
        idx = torch.full(self.shape, -1, device="cuda")
        idx[_inner(self.shape)] = torch.where(self.free, torch.arange(n, device="cuda").view(self.diag.shape), -1)
        A = torch.diag(self.diag.reshape(-1))
        me = _at(idx, (0, 0, 0))
        for o, w in self.W.items():
            to = _at(idx, o)
            ok = (me >= 0) & (to >= 0)
            A[me[ok], to[ok]] = w[ok]
        return A


class _Plain:
    """V(3,3) cycles on the global node grid."""

    def __init__(self, case, seed, faulty=None):
        sub = _sub(case)
        pos = np.stack(np.meshgrid(*(np.arange(n + 1) / n for n in sub), indexing="ij"), -1).transpose(2, 1, 0, 3)
        if case["shape"] == "corners":
            pos = _corners(case)
        elif case["shape"] == "sheared":
            pos = pos @ np.array(SHEAR).T
        pos = pos.reshape(-1, 3)
        B = np.zeros((_n_macro(case), 3, 3))
        for m, t in enumerate(_tets(case)):
            for s, ax in enumerate(PERMS[m % 6]):
                B[m, :, ax] = pos[t[s + 1]] - pos[t[s]]
        k = _coeff(case, seed)
        self.k = torch.ones(len(B), dtype=torch.float64, device="cuda") if k is None else torch.from_numpy(k).cuda()
        bad = None
        if faulty is not None:
            bad = torch.zeros(len(B), dtype=torch.bool, device="cuda")
            bad[list(faulty)] = True
        self.lv = [_Level(sub, r, torch.from_numpy(B).cuda(), self.k, bad) for r in range(2, case["levels"] + 1)]
        self.A0 = torch.linalg.lu_factor(self.lv[0].dense())

    def cycle(self, u, f, l=None):
        l = len(self.lv) - 1 if l is None else l
        L = self.lv[l]
        i = _inner(L.shape)
        if l == 0:
            u[i] = torch.linalg.lu_solve(*self.A0, torch.where(L.free, f[i], 0.0).reshape(-1, 1)).view(L.diag.shape)
            return u
        C = self.lv[l - 1]
        L.smooth(u, f, 3)
        r = L.residual(u, f)
        fc, uc = (torch.zeros(C.shape, dtype=torch.float64, device="cuda") for _ in range(2))
        even = lambda off: tuple(slice(2 + o, n - 2 + o, 2) for o, n in zip(reversed(off), L.shape))  # noqa: E731
        fc[_inner(C.shape)] = r[even((0, 0, 0))] + 0.5 * sum(r[even(o)] for o in OFFS)
        self.cycle(uc, fc, l - 1)
        e = torch.zeros_like(u)
        for par in itertools.product((0, 1), repeat=3):                 # (x, y, z) parity
            lo = tuple(slice(0, n - p) for n, p in zip(C.shape, reversed(par)))
            hi = tuple(slice(p, n) for n, p in zip(C.shape, reversed(par)))
            to = tuple(slice(p, None, 2) for p in reversed(par))
            e[to] = uc[lo] if not any(par) else 0.5 * (uc[lo] + uc[hi])
        u[i] += torch.where(L.free, e[i], 0.0)
        L.smooth(u, f, 3)
        return u

    def solve(self, u, f):
        """Cycles until rounding holds the residual up."""
        best, since = math.inf, 0
        for _ in range(400):
            r = float(self.lv[-1].residual(u, f).norm())
            since = 0 if r < 0.9 * best else since + 1
            if since > 2 or r == 0.0:
                break
            best = min(best, r)
            self.cycle(u, f)
        return u


def _general_nodes(case):
    """Grid index of every node of the general mesh, in the library's order:
    interface nodes by key, then the volume nodes macro by macro."""
    N, n1 = 1 << case["levels"], (1 << case["levels"]) + 1
    sx, sy, _ = _sub(case)
    shape = _grid(case)
    tets = _tets(case).astype(np.int64)
    corner = np.stack([tets % (sx + 1), tets // (sx + 1) % (sy + 1), tets // ((sx + 1) * (sy + 1))], -1)
    k, j, i = np.meshgrid(*(np.arange(N + 1),) * 3, indexing="ij")
    w = np.stack([N - i - j - k, i, j, k], -1).reshape(-1, 4)
    w = w[w[:, 0] >= 0]
    pos = np.einsum("nv,tvx->tnx", w, corner)
    gid = (pos[..., 2] * shape[1] + pos[..., 1]) * shape[2] + pos[..., 0]
    inner = (w > 0).all(1)
    code = np.where(w[None] > 0, tets[:, None, :] * n1 + w[None], np.iinfo(np.int64).max)[:, ~inner]
    code.sort(-1)
    count = (w[~inner] > 0).sum(1)
    key = np.concatenate([np.broadcast_to(count, code.shape[:2])[..., None], code], -1).reshape(-1, 5)
    _, first = np.unique(key, axis=0, return_index=True)
    return np.concatenate([gid[:, ~inner].reshape(-1)[first], gid[:, inner].reshape(-1)])


def exact(case, seed):
    call = case["call"]
    if call == "batch":
        out, made = [], {}
        for t in range(case["tasks"]):
            one = dict(case, sx=case["sx"] if t % 2 else 1)
            lost = tuple(_task_fault(one, t))
            key = (one["sx"], lost)
            if key not in made:
                made[key] = _Plain(one, seed, lost)
            f, u = _fields(one, seed * 1000 + t, _grid(one))
            i = _inner(u.shape)
            u[i] = torch.where(made[key].lv[-1].free, 0.0, u[i])
            for _ in range(case["cycles"]):
                made[key].cycle(u, f)
            out.append(u)
        return {"u": out}
    P = _Plain(case, seed)
    f, u = _fields(case, seed, _grid(case))
    if call == "cycle":
        P.cycle(u, f)
        return {"u": u, "res": float(P.lv[-1].residual(u, f).norm())}
    P.solve(u, f)
    if call == "solve_general":
        return {"u": u.reshape(-1)[torch.from_numpy(_general_nodes(case)).cuda()]}
    if call != "gradient":
        return {"u": u}
    L = P.lv[-1]
    rhs = u - torch.rand(u.shape, generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
    lam = P.solve(torch.zeros_like(u), rhs)
    dk = torch.zeros_like(P.k)
    for p in range(6):
        lv, uv = (torch.stack([a[L._cells(L.verts[p][v])] for v in range(4)]) for a in (lam, u))
        val = torch.zeros_like(uv[0])
        for v, w in itertools.product(range(4), repeat=2):
            val += L.K[:, p, v, w][L.macro[p]] * lv[v] * uv[w]
        dk -= torch.bincount(L.macro[p].reshape(-1), val.reshape(-1), minlength=len(dk))
    return {"u": u, "df": lam, "dk": dk}
