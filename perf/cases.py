"""The work a user of gbcg has it do, as cases that can be timed and checked.

Every case goes through the public Python entry points (``gbcg.Solver``,
``gbcg.BatchSolver``, ``gbcg.Net``, ``gbcg.cg_solve_noalloc``) on the
matrices the repository is about: Q1 hexahedral FEM systems on a box of
ex x ey x ez elements (27 entries per inner row), air with iron blobs,
assembled here on the GPU from the seed.

Right-hand sides are seeded source currents (b = M_L J, the time-stepping
load of the batched workload).  Solves run to the paper's tolerance 1e-10
(Table I), or for a fixed number of iterations (a user's own budget, or the
116 the paper reports).
"""
import functools
import math

import numpy as np
import torch

from paper_1107_0538_gb300 import gbcg, problems

TOL = 1e-10   # the paper's tolerance (Table I)
COILS = 3     # boxes of source current per right-hand side


def listed():
    return [
        # y = A x alone on the paper-sized matrix: a user's own Krylov loop,
        # one short launch per call, the matrix in L2
        {"name": "spmv_50", "kind": "spmv", "ex": 50, "ey": 50, "ez": 50},
        # the same on a matrix larger than L2: bound by memory
        {"name": "spmv_100", "kind": "spmv", "ex": 100, "ey": 100, "ez": 100},
        # the smallest system in use (the smoke test's 8^3 box): one solve of
        # a small model, latency only
        {"name": "cg_8", "kind": "cg", "ex": 8, "ey": 8, "ez": 8, "contrast": 1e2, "maxit": 0},
        # the 20^3 uniform system of the parity tests, solved to 1e-10
        {"name": "cg_20", "kind": "cg", "ex": 20, "ey": 20, "ez": 20, "contrast": 1.0, "maxit": 0},
        # the paper-sized system (N = 132651): plain FP64 CG, the headline path
        {"name": "cg_50", "kind": "cg", "ex": 50, "ey": 50, "ez": 50, "contrast": 1e3, "maxit": 0},
        # FP64 Jacobi-PCG on an uneven box of about that size, the form most
        # users would run there
        {"name": "pcg_57x44x61", "kind": "pcg", "ex": 57, "ey": 44, "ez": 61, "contrast": 1e3, "maxit": 0},
        # plain FP64 CG on the large system, a budget of 200 iterations: the
        # matrix streams from HBM
        {"name": "cg_100", "kind": "cg", "ex": 100, "ey": 100, "ez": 100, "contrast": 1e3, "maxit": 200},
        # mixed precision (FP32 inner CG with Jacobi, FP64 refinement) on the
        # large system
        {"name": "ir32_100", "kind": "ir", "ex": 100, "ey": 100, "ez": 100, "contrast": 1e3, "values": "fp32"},
        # batched time stepping: uneven boxes with 4 right-hand sides each
        {"name": "batch_16", "kind": "batch", "nsys": 16, "emin": 20, "emax": 40, "sizes": 1000,
         "nrhs": 4, "values": "fp32"},
        # flexible CG with the learned preconditioner on the large system
        {"name": "learned_100", "kind": "learned", "ex": 100, "ey": 100, "ez": 100, "contrast": 1e3},
        # training: loss and gradient of one mini-batch of 8 pairs at 50^3
        {"name": "grad_50", "kind": "grad", "ex": 50, "ey": 50, "ez": 50, "contrast": 1e3, "pairs": 8},
        # the allocation-free solve of a caller's device CSR arrays, for the
        # number of iterations the paper reports (Table I)
        {"name": "noalloc_50", "kind": "noalloc", "ex": 50, "ey": 50, "ez": 50, "contrast": 1e3, "maxit": 116},
    ]


def draw(rng):
    """One more case of the listed kinds, over the sizes each is used at."""
    def edge(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):
        e = edge(lo, hi)
        return {k: min(hi, max(lo, int(round(e * rng.uniform(0.75, 1.3))))) for k in ("ex", "ey", "ez")}

    contrast = round(10.0 ** rng.uniform(1.0, 3.0), 3)
    kind = rng.choice(["spmv", "cg", "pcg", "ir", "batch", "learned", "grad", "noalloc"])
    if kind == "spmv":
        return {"kind": kind, **box(32, 100)}
    if kind == "cg":
        return {"kind": kind, **box(8, 90), "contrast": contrast, "maxit": 0}
    if kind == "pcg":
        return {"kind": kind, **box(8, 90), "contrast": contrast, "maxit": 0}
    if kind == "ir":
        return {"kind": kind, **box(16, 90), "contrast": contrast, "values": rng.choice(["fp32", "bf16"])}
    if kind == "batch":
        return {"kind": kind, "nsys": rng.randint(1, 24), "emin": rng.randint(8, 20), "emax": rng.randint(21, 40),
                "sizes": rng.randint(0, 9999), "nrhs": rng.randint(1, 4), "values": rng.choice(["fp32", "fp32", "bf16"])}
    if kind == "learned":
        return {"kind": kind, **box(12, 80), "contrast": contrast}
    if kind == "grad":
        return {"kind": kind, **box(12, 56), "contrast": contrast, "pairs": rng.randint(1, 8)}
    return {"kind": kind, **box(8, 60), "contrast": contrast, "maxit": 0}


# ------------------------------------------------------------------ matrices

class _System:
    """One Q1 system: the numpy CSR the entry points take, and what the
    64-bit values below need (27 columns and values per row, on the GPU)."""

    def __init__(self, ex, ey, ez, contrast, seed):
        self.grid = g = problems.Grid(ex, ey, ez, 1.0 / max(ex, ey, ez))
        self.rowptr, self.colidx, self.cols, self.inside = _pattern(ex, ey, ez)
        self.n = g.n
        self.nu = problems.nu_blobs(g, seed=10 * seed + 1, nu_iron=1.0 / contrast)
        nu = torch.nn.functional.pad(torch.from_numpy(self.nu).cuda(), (1, 1, 1, 1, 1, 1))
        one = torch.nn.functional.pad(torch.ones_like(torch.from_numpy(self.nu)).cuda(), (1, 1, 1, 1, 1, 1))
        nx, ny, nz = g.nodes

        def shared(field, dz, dy, dx):   # sum over the elements that hold a node and its neighbour
            rng = [(0,) if d == 1 else ((-1,) if d == -1 else (-1, 0)) for d in (dz, dy, dx)]
            acc = 0.0
            for sz in rng[0]:
                for sy in rng[1]:
                    for sx in rng[2]:
                        acc = acc + field[1 + sz:1 + sz + nz, 1 + sy:1 + sy + ny, 1 + sx:1 + sx + nx]
            return acc.reshape(-1)

        mass = (g.h ** 3 / 8.0) * shared(one, 0, 0, 0)
        ell = torch.empty((self.n, 27), dtype=torch.float64, device="cuda")
        for t, (dz, dy, dx) in enumerate(_offsets()):
            nd = abs(dz) + abs(dy) + abs(dx)
            ell[:, t] = g.h * problems.Q1_UNIT_STIFFNESS[nd] * shared(nu, dz, dy, dx)
        ell[:, 13] += 1e-2 * mass
        ell *= self.inside
        self.mass, self.ell = mass, ell
        self.vals_dev = ell[self.inside]
        self.vals = self.vals_dev.cpu().numpy()

    def times(self, v):
        """A v in FP64; v is (n,) or (n, m)."""
        out = 0.0
        for t in range(27):
            a = self.ell[:, t]
            out = out + (a if v.dim() == 1 else a[:, None]) * v[self.cols[:, t]]
        return out

    def currents(self, seed, steps=1):
        """(steps, n) right-hand sides: M_L J of a few boxes of source current."""
        u = problems.uniform01(10 * seed + 2, 8 * COILS).reshape(COILS, 8)
        g = self.grid
        nx, ny, nz = g.nodes
        ax = [torch.arange(m, device="cuda", dtype=torch.float64) / max(m - 1, 1) for m in (nx, ny, nz)]
        out = torch.zeros((steps, self.n), dtype=torch.float64, device="cuda")
        for c in range(COILS):
            lo, hi = 0.1 + 0.5 * u[c, 0:3], 0.2 + 0.5 * u[c, 0:3] + 0.3 * u[c, 3:6]
            m = [((a >= lo[i]) & (a <= hi[i])).double() for i, a in enumerate(ax)]
            box = (m[2][:, None, None] * m[1][None, :, None] * m[0][None, None, :]).reshape(-1)
            for s in range(steps):
                out[s] += (0.5 + 1.5 * u[c, 6]) * math.sin(2 * math.pi * (s / steps + u[c, 7])) * box
        return out * self.mass + 1e-3 * self.mass

    @property
    def nnz(self):
        return int(self.colidx.size)


def _offsets():
    return [(dz, dy, dx) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]


@functools.lru_cache(maxsize=4)
def _pattern(ex, ey, ez):
    """Row pointers, columns, and per row its 27 neighbours and which exist."""
    nx, ny, nz = ex + 1, ey + 1, ez + 1
    kk, jj, ii = torch.meshgrid(*(torch.arange(m, device="cuda") for m in (nz, ny, nx)), indexing="ij")
    node = (ii + nx * (jj + ny * kk)).reshape(-1)
    cols = torch.empty((node.numel(), 27), dtype=torch.int64, device="cuda")
    inside = torch.empty((node.numel(), 27), dtype=torch.bool, device="cuda")
    for t, (dz, dy, dx) in enumerate(_offsets()):
        ok = ((kk + dz >= 0) & (kk + dz < nz) & (jj + dy >= 0) & (jj + dy < ny) & (ii + dx >= 0)
              & (ii + dx < nx)).reshape(-1)
        cols[:, t] = torch.where(ok, node + dx + nx * (dy + ny * dz), node)
        inside[:, t] = ok
    rowptr = torch.zeros(node.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(inside.sum(dim=1), 0, out=rowptr[1:])
    return rowptr.int().cpu().numpy(), cols[inside].int().cpu().numpy(), cols, inside


def _system(case, seed):
    return _System(case["ex"], case["ey"], case["ez"], case.get("contrast", 1e3), seed)


def _sizes(case):
    """Element counts of the batch's boxes."""
    lo, hi = case["emin"], case["emax"]
    u = problems.uniform01(case["sizes"], 3 * case["nsys"]).reshape(-1, 3)
    return (lo + np.minimum((u * (hi - lo + 1)).astype(int), hi - lo)).tolist()


def _batch(case, seed):
    return [_System(*s, 10.0 ** (2.0 + 2.0 * float(problems.uniform01(seed + 7 * i, 1)[0])), seed + i)
            for i, s in enumerate(_sizes(case))]


def _values(case):
    return {"fp32": gbcg.CG_VALUES_FP32, "bf16": gbcg.CG_VALUES_BF16}[case["values"]]


def _pairs(sys_, case, seed):
    """Training pairs: errors e (uniform, then smoothed by one product, as the
    error after a few CG steps is) and their residuals A e, as floats."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    e = 2.0 * torch.rand((case["pairs"], sys_.n), dtype=torch.float64, device="cuda", generator=g) - 1.0
    return (torch.stack([sys_.times(v) for v in e]).float().contiguous(), e.float().contiguous())


# --------------------------------------------------------------- the entry points

def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "tol": TOL, "maxit": case.get("maxit", 0)}
    if kind == "batch":
        systems = _batch(case, seed)
        st["solver"] = gbcg.BatchSolver(systems, inner_values=_values(case), precond=gbcg.CG_PRECOND_JACOBI)
        st["b"] = torch.cat([s.currents(seed + i, case["nrhs"]) for i, s in enumerate(systems)], dim=1).contiguous()
        st["x"] = torch.zeros_like(st["b"])
        return st
    s = _system(case, seed)
    if kind == "spmv":
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["solver"] = gbcg.Solver(s)
        st["x"] = 2.0 * torch.rand(s.n, dtype=torch.float64, device="cuda", generator=g) - 1.0
        st["y"] = torch.empty_like(st["x"])
        return st
    st["b"] = s.currents(seed)[0].contiguous()
    st["x"] = torch.zeros_like(st["b"])
    if kind in ("cg", "pcg"):
        st["solver"] = gbcg.Solver(s, precond=gbcg.CG_PRECOND_JACOBI if kind == "pcg" else gbcg.CG_PRECOND_NONE)
    elif kind == "ir":
        st["solver"] = gbcg.Solver(s, precond=gbcg.CG_PRECOND_JACOBI, inner_values=_values(case))
    elif kind in ("learned", "grad"):
        st["net"] = gbcg.Net(problems.learn_init_params(seed=seed))
        st["solver"] = gbcg.Solver(s, precond=gbcg.CG_PRECOND_LEARNED)
        st["solver"].set_learned(st["net"], s.grid, problems.node_log_nu(s.grid, s.nu).astype(np.float32))
        if kind == "grad":
            R, E = _pairs(s, case, seed)
            st["set"] = gbcg.LearnSet([st["solver"]], np.zeros(case["pairs"], dtype=np.int32), R, E)
            st["order"] = np.arange(case["pairs"])
    else:
        dev = [torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colidx).cuda(), s.vals_dev.contiguous()]
        st["csr"] = gbcg.cg_csr(s.n, s.nnz, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(),
                                gbcg.CG_MEM_DEVICE)
        st["keep"] = dev
    return st


def run(st):
    kind = st["kind"]
    if kind == "spmv":
        st["solver"].spmv(st["x"], st["y"])
        return st["y"]
    if kind == "grad":
        loss, grad = st["net"].grad(st["set"], st["order"])
        return {"loss": np.float32(loss), "grad": grad}
    st["x"].zero_()
    if kind == "batch":
        st["solver"].solve(st["b"], st["x"], st["tol"])
    elif kind == "noalloc":
        gbcg.cg_solve_noalloc(st["csr"], st["b"].data_ptr(), st["x"].data_ptr(), st["tol"], st["maxit"],
                              torch.cuda.current_stream().cuda_stream)
    else:
        st["solver"].solve(st["b"], st["x"], st["tol"], st["maxit"])
    return st["x"]


# ------------------------------------------------------------------ work, exact values

def _nnz(ex, ey, ez):
    return problems.q1_nnz(ex, ey, ez), (ex + 1) * (ey + 1) * (ez + 1)


def work(case):
    """Matrix (values and 32-bit columns) and vectors once; flops of the
    iterations.  Where the tolerance ends the solve, the number of iterations
    is estimated from the longest edge, as measured on the 20^3 to 100^3 boxes."""
    kind = case["kind"]
    if kind == "batch":
        e = 0.5 * (case["emin"] + case["emax"])
        n1, nnz1 = (e + 1) ** 3, (3 * e + 1) ** 3
        n, nnz, m, iters = case["nsys"] * n1, case["nsys"] * nnz1, case["nrhs"], 16 * e
        return {"bytes": 12 * nnz + 4 * n + 16 * n * m, "flops": iters * m * (2 * nnz + 13 * n)}
    nnz, n = _nnz(case["ex"], case["ey"], case["ez"])
    e = max(case["ex"], case["ey"], case["ez"])
    once = 12 * nnz + 4 * (n + 1) + 16 * n
    conv = 2 * n * 27 * 2 * (16 + 256)   # L and its adjoint: 1->16, 16->16, 16->16, 16->1
    if kind == "spmv":
        return {"bytes": once, "flops": 2 * nnz}
    if kind == "grad":
        return {"bytes": once + 8 * n * case["pairs"], "flops": case["pairs"] * (3 * conv + 2 * nnz)}
    if kind == "learned":
        return {"bytes": once + 4 * n, "flops": 7 * e * (2 * nnz + 13 * n + conv)}
    if kind == "ir":
        return {"bytes": once, "flops": 16 * e * (2 * nnz + 13 * n)}
    iters = case["maxit"] or (7 if kind == "pcg" else 6 + 7 * math.log10(case["contrast"])) * e
    return {"bytes": once, "flops": iters * (2 * nnz + 10 * n + (3 * n if kind == "pcg" else 0))}


def _pcg(s, b, tol, maxit, jacobi):
    """Textbook CG in FP64 (columns of b together); maxit 0: to the tolerance."""
    d = (1.0 / s.ell[:, 13]) if jacobi else torch.ones(s.n, dtype=torch.float64, device="cuda")
    d = d if b.dim() == 1 else d[:, None]
    x, r = torch.zeros_like(b), b.clone()
    z = d * r
    p, rho, bb = z.clone(), (r * z).sum(0), (b * b).sum(0)
    for k in range(maxit or 4000):
        q = s.times(p)
        a = rho / (p * q).sum(0)
        x, r = x + a * p, r - a * q
        if not maxit and k % 10 == 9 and bool(((r * r).sum(0) <= tol * tol * bb).all()):
            break
        z = d * r
        new = (r * z).sum(0)
        p, rho = z + (new / rho) * p, new
    return x


def _net(theta, lognu, shape, dinv):
    """u = L^T L s (before the final D^-1/2) of the preconditioner in 64 bits."""
    nz, ny, nx = shape
    w1, w2, wg = theta[:432].view(16, 1, 3, 3, 3), theta[432:7344].view(16, 16, 3, 3, 3), theta[7344:7776].view(16, 1, 3, 3, 3)
    conv, back = torch.nn.functional.conv3d, torch.nn.functional.conv_transpose3d
    gate = torch.sigmoid(conv((lognu / 8.0).view(1, 1, nz, ny, nx), wg, theta[7776:], padding=1))

    def apply(s):
        h = conv(gate * conv(s.view(1, 1, nz, ny, nx), w1, padding=1), w2, padding=1)
        return back(gate * back(h, w2, padding=1), w1, padding=1).reshape(-1)
    return apply


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return torch.cat([_pcg(s, s.currents(seed + i, case["nrhs"]).T.contiguous(), 1e-14, 0, True).T
                          for i, s in enumerate(_batch(case, seed))], dim=1)
    s = _system(case, seed)
    if kind == "spmv":
        g = torch.Generator(device="cuda").manual_seed(seed)
        return s.times(2.0 * torch.rand(s.n, dtype=torch.float64, device="cuda", generator=g) - 1.0)
    if kind == "grad":
        R, E = (v.double() for v in _pairs(s, case, seed))
        theta = torch.from_numpy(problems.learn_init_params(seed=seed)).double().cuda().requires_grad_(True)
        lognu = torch.from_numpy(problems.node_log_nu(s.grid, s.nu).astype(np.float32)).double().cuda()
        dh = s.ell[:, 13].rsqrt()
        nx, ny, nz = s.grid.nodes
        loss = 0.0
        for r, e in zip(R, E):
            v = dh * r
            sigma = v.square().mean().sqrt()
            w = dh * (_net(theta, lognu, (nz, ny, nx), dh)(v / sigma) - e / (dh * sigma))
            loss = loss + (w * s.times(w)).sum() / (2.0 * s.n * len(R))
        loss.backward()
        return {"loss": loss.detach().cpu().numpy(), "grad": theta.grad.cpu().numpy()}
    b = s.currents(seed)[0]
    if case.get("maxit"):
        return _pcg(s, b, 0.0, case["maxit"], kind == "pcg")
    return _pcg(s, b, 1e-14, 0, True)
