"""The work that a user of this library has it do, as cases that can be timed
and compared: the stencil, the smoother, the coarse operator and the coarse
solve one by one, whole setups and solves, and the learned generator's
training step and inference, each through the package's public calls.

A case is a dict of plain values. `listed` gives the fixed ones, `draw` more
of the same ranges, `prepare` the state a program holds before the call (a
lattice context with its gauge field, clover term and input fields on the
GPU), `run` one pass, `work` what a pass cannot do without, and `exact` the
result of the same inputs in 64 bits, written in plain torch.
"""
import math

import numpy as np
import torch

from paper_1601_03184_gb300 import (MRHS_BF16, MRHS_F16, MRHS_F32, MRHS_F64, MRHS_PREC_FP32, MRHS_PREC_FP64,
                                    MRHS_PREC_MIX_BF16, MRHS_PREC_MIX_FP16, Lattice, mrhs_nn_create,
                                    mrhs_nn_get_grads, mrhs_nn_get_weights, mrhs_nn_infer, mrhs_nn_set_weights,
                                    mrhs_nn_train_step)

DTYPE = {"f64": MRHS_F64, "f32": MRHS_F32, "bf16": MRHS_BF16, "f16": MRHS_F16}
TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
PREC = {"f64": MRHS_PREC_FP64, "f32": MRHS_PREC_FP32, "bf16": MRHS_PREC_MIX_BF16, "f16": MRHS_PREC_MIX_FP16}
EPS, M0, CSW = 0.6, -0.55, 1.5  # roughness, mass (a little heavier than critical) and clover coefficient
LAMBDA, LR = 1.0, 1e-3          # of the training loss and of Adam


def _case(name, kind, dims, agg, **more):
    c = {"kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
         "ax": agg[0], "ay": agg[1], "az": agg[2], "at": agg[3], **more}
    return {"name": name, **c} if name else c


def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _agg(c):
    return (c["ax"], c["ay"], c["az"], c["at"])


def listed():
    a4 = (4, 4, 4, 4)
    return [
        # D on a handful of ragged blocks and an odd count of vectors: the smallest call, all latency
        _case("stencil small odd", "stencil", (4, 6, 4, 8), (2, 3, 2, 2), nrhs=5, dtype="f32"),
        # D on all test vectors of the largest lattice here: residual checks, the network's loss
        _case("stencil large f32", "stencil", (32, 32, 32, 64), a4, nrhs=24, dtype="f32"),
        # D on vectors kept in bf16 (the mixed-precision setup's storage)
        _case("stencil bf16", "stencil", (16, 16, 16, 32), a4, nrhs=32, dtype="bf16"),
        # the refinement's smoother: 4 sweeps of 4 MR steps from the coarse correction
        _case("smoother refine", "smoother", (16, 16, 16, 32), a4, nrhs=20, dtype="f32", sweeps=4, mr=4, guess=True),
        # the initial phase's smoother on the largest lattice here: 5 sweeps from zero
        _case("smoother large", "smoother", (32, 32, 32, 64), a4, nrhs=24, dtype="f32", sweeps=5, mr=4, guess=False),
        # P and D_c from given test vectors, then R, D_c and P once each (what a setup update rebuilds)
        _case("coarse operator f32", "coarse_operator", (16, 16, 16, 32), a4, ntv=32, prec="f32"),
        # the same in the mixed-precision setup on the largest lattice here
        _case("coarse operator bf16", "coarse_operator", (32, 32, 32, 64), a4, ntv=24, prec="bf16"),
        # the coarse solve of all test vectors, even-odd preconditioned, one GMRES cycle
        _case("coarse solve", "coarse_solve", (16, 16, 16, 32), a4, ntv=32, prec="f32", iters=20, even_odd=True),
        # a whole setup: initial phase and three refinements
        _case("setup", "setup", (16, 16, 16, 32), a4, ntv=20, prec="f32", refine=3, iters=10, even_odd=True),
        # one propagator solve with a finished setup (one right-hand side everywhere)
        _case("solve", "solve", (16, 16, 16, 16), a4, ntv=16, prec="f32"),
        # the learned generator: one training step on eight vectors
        _case("train", "train", (16, 16, 16, 16), a4, ntv=8, width=11),
        # and its inference at the wide hidden layers
        _case("infer wide", "infer", (16, 16, 16, 32), a4, ntv=32, width=32),
    ]


def _lattice(rng, most):
    """Extents and aggregates: 4^4 aggregates mostly, an even number of them per direction."""
    agg = rng.choice([(4, 4, 4, 4)] * 4 + [(2, 2, 2, 2), (2, 3, 2, 2), (4, 4, 4, 2), (3, 3, 3, 3)])
    dims = [2 * a for a in agg]
    goal = math.exp(rng.uniform(math.log(np.prod(dims)), math.log(most)))
    while True:
        mu = rng.choice([m for m in range(4) if dims[m] == min(dims)] + [3])
        dims[mu] += 2 * agg[mu]
        if np.prod(dims) > goal:
            dims[mu] -= 2 * agg[mu]
            return tuple(dims), agg


def draw(rng):
    kind = rng.choice(["stencil", "stencil", "smoother", "smoother", "coarse_operator", "coarse_operator",
                       "coarse_solve", "setup", "solve", "train", "infer"])
    if kind == "stencil":
        dims, agg = _lattice(rng, 1 << 20)
        return _case(None, kind, dims, agg, nrhs=rng.choice([1, 3, 4, 8, 12, 16, 20, 24, 32, rng.randint(1, 40)]),
                     dtype=rng.choice(["f32", "f32", "bf16", "f16", "f64"]))
    if kind == "smoother":
        dims, agg = _lattice(rng, 1 << 18)
        return _case(None, kind, dims, agg, nrhs=rng.choice([1, 4, 8, 12, 16, 20, 24, 32, rng.randint(1, 40)]),
                     dtype=rng.choice(["f32", "f32", "f32", "f64"]), sweeps=rng.randint(1, 5), mr=rng.randint(2, 5),
                     guess=rng.choice([True, False]))
    if kind == "coarse_operator":
        dims, agg = _lattice(rng, 1 << 18)
        most = min(32, 3 * int(np.prod(agg)))
        return _case(None, kind, dims, agg, ntv=min(most, rng.choice([8, 12, 16, 20, 24, 32, rng.randint(4, 32)])),
                     prec=rng.choice(["f32", "f32", "bf16", "f16", "f64"]))
    if kind == "coarse_solve":
        dims, agg = _lattice(rng, 1 << 18)
        return _case(None, kind, dims, agg, ntv=rng.choice([8, 12, 16, 20, 24, 32, rng.randint(4, 32)]),
                     prec=rng.choice(["f32", "f32", "bf16"]), iters=rng.randint(4, 20),
                     even_odd=rng.choice([True, True, False]))
    if kind == "setup":
        dims, agg = _lattice(rng, 1 << 17)
        return _case(None, kind, dims, agg, ntv=rng.choice([8, 12, 16, 20, 24, rng.randint(4, 24)]),
                     prec=rng.choice(["f32", "f32", "bf16"]), refine=rng.randint(1, 3), iters=rng.randint(4, 10),
                     even_odd=rng.choice([True, False]))
    a4 = (4, 4, 4, 4)
    dims = rng.choice([(8, 8, 8, 8), (8, 8, 8, 16), (8, 8, 16, 16), (16, 16, 16, 16)])
    if kind == "solve":
        return _case(None, kind, dims, a4, ntv=rng.choice([8, 12, 16, rng.randint(6, 20)]), prec="f32")
    return _case(None, kind, dims, a4, ntv=rng.choice([4, 8, rng.randint(1, 12)]),
                 width=rng.choice([11, 11, 16, 32, rng.randint(6, 32)]))


# ------------------------------------------------------------------ inputs --
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed % (1 << 40)) + salt)
    return g


def _gauge(dims, seed):
    """U[s][mu] = exp(i EPS H) on the GPU, H = sum_a h_a lambda_a / 2 with normal h_a; canonical site order."""
    V = int(np.prod(dims))
    lam = torch.zeros(8, 3, 3, dtype=torch.complex128, device="cuda")
    for k, (i, j) in enumerate([(0, 1), (0, 2), (1, 2)]):
        n = (0, 3, 5)[k]
        lam[n, i, j] = lam[n, j, i] = 1
        lam[n + 1, i, j], lam[n + 1, j, i] = -1j, 1j
    lam[2] = torch.diag(torch.tensor([1, -1, 0]))
    lam[7] = torch.diag(torch.tensor([1, 1, -2])) / math.sqrt(3)
    h = torch.randn(V, 4, 8, generator=_gen(seed, 1), device="cuda", dtype=torch.float64)
    return torch.linalg.matrix_exp(1j * EPS / 2 * torch.einsum("sma,aij->smij", h.to(lam.dtype), lam))


def _normal(n, seed, salt, dtype="f32"):
    """n normal numbers as a field of storage type dtype."""
    return torch.randn(n, generator=_gen(seed, salt), device="cuda").to(TORCH[dtype])


def _weights(width, seed):
    """The generator's starting weights: the identity on the first four channels and noise, rounded to bf16."""
    g, ws = _gen(seed, 6), []
    for cin, cout in ((4, width), (width, width), (width, 4)):
        w = 0.03 * torch.randn(9, cout, cin, 2, generator=g, device="cuda")
        for i in range(4):
            w[0, i, i, 0] += 1.0
        ws.append(w.bfloat16().float().reshape(-1))
    return torch.cat(ws + [0.02 * torch.randn(2 * width, generator=g, device="cuda")]).cpu().numpy()


def prepare(case, seed):
    kind, dims, agg = case["kind"], _dims(case), _agg(case)
    V = int(np.prod(dims))
    n = case.get("ntv") or case["nrhs"]
    prec = case.get("prec") or ("f64" if case.get("dtype") == "f64" else "f32")
    wd = "f64" if prec == "f64" else "f32"
    lat = Lattice(dims, agg, min(n, 8) if kind in ("stencil", "smoother") else n, PREC[prec])
    lat.set_gauge(_gauge(dims, seed).cpu().numpy())
    lat.build_clover(M0, CSW)
    s = {"case": case, "lat": lat, "n": n, "wd": DTYPE[wd], "td": TORCH[wd]}
    fine, coarse = V * 24 * n, lat.nagg * 2 * n * 2 * n
    if kind == "stencil":
        s["x"] = _normal(fine, seed, 2, case["dtype"])
        s["y"] = torch.empty_like(s["x"])
    elif kind == "smoother":
        s["b"] = _normal(fine, seed, 2, wd)
        s["x0"] = _normal(fine, seed, 3, wd) if case["guess"] else None
        s["x"] = torch.empty_like(s["b"])
    elif kind in ("train", "infer"):
        s["v"], s["y"], s["step"] = _normal(fine, seed, 3), None, 0
        mrhs_nn_create(lat.ctx, (4, case["width"], case["width"], 4), 1)
        mrhs_nn_set_weights(lat.ctx, _weights(case["width"], seed))
        if kind == "train":
            lat.set_tv(_normal(fine, seed, 2), MRHS_F32)
            lat.build_P()
        else:
            s["y"] = torch.empty_like(s["v"])
    else:
        s["tv"] = _normal(fine, seed, 2, wd)
        if kind != "solve":
            s["vc"] = _normal(coarse, seed, 4, wd)
            s["yc"] = torch.empty_like(s["vc"])
        if kind in ("coarse_operator", "setup"):
            # the coarse unit vectors, both chiralities of column j in right-hand side j: P of them is P itself
            e = torch.zeros(lat.nagg, 2, n, 2, n, device="cuda", dtype=s["td"])
            e[:, :, torch.arange(n), 0, torch.arange(n)] = 1
            s["unit"], s["P"] = e.reshape(-1), torch.empty_like(s["tv"])
        if kind in ("coarse_solve", "setup"):
            lat.set_coarse_solver(1 if case["even_odd"] else 0)
        if kind == "coarse_solve":
            lat.set_tv(s["tv"], s["wd"])
            lat.build_P()
            lat.build_Dc()
        if kind == "solve":
            lat.set_coarse_solver(1)
            lat.setup_init(s["tv"], s["wd"], 0, 4, 4)
            lat.setup_refine(2, 4, 4, 0.05, 20, 100)
            g = torch.randn(V, 12, 2, generator=_gen(seed, 5), device="cuda", dtype=torch.float64)
            s["b"] = torch.view_as_complex(g).cpu().numpy()
    return s


# ------------------------------------------------------------------- a pass --
def run(state):
    s, c, lat = state, state["case"], state["lat"]
    kind, n, wd = c["kind"], s["n"], s["wd"]
    if kind == "stencil":
        lat.apply_D(s["x"], s["y"], n, DTYPE[c["dtype"]])
        return s["y"]
    if kind == "smoother":
        if s["x0"] is None:
            s["x"].zero_()
        else:
            s["x"].copy_(s["x0"])
        lat.sap(s["b"], s["x"], n, wd, c["sweeps"], c["mr"])
        return s["x"]
    if kind == "coarse_operator":
        lat.set_tv(s["tv"], wd)
        lat.build_P()
        lat.build_Dc()
        lat.restrict(s["tv"], s["vc"], n, wd)
        lat.apply_Dc(s["vc"], s["yc"], n, wd)
        lat.prolong(s["unit"], s["P"], n, wd)
        return {"P": s["P"], "vc": s["vc"], "yc": s["yc"]}
    if kind == "coarse_solve":
        lat.coarse_solve(s["vc"], s["yc"], n, wd, 0.0, 20, c["iters"])
        return s["yc"]
    if kind == "setup":
        lat.setup_init(s["tv"], wd, 0, 5, 4)
        lat.setup_refine(c["refine"], 4, 4, 0.0, 20, c["iters"])
        lat.prolong(s["unit"], s["P"], n, wd)
        lat.apply_Dc(s["vc"], s["yc"], n, wd)
        return {"P": s["P"], "yc": s["yc"]}
    if kind == "solve":
        return lat.solve_fgmres(s["b"], tol=1e-12, restart=25, maxit=200)[0]
    if kind == "infer":
        mrhs_nn_infer(lat.ctx, s["v"], s["y"], n)
        return s["y"]
    s["step"] += 1
    loss = mrhs_nn_train_step(lat.ctx, s["v"], n, LAMBDA, LR, s["step"])
    return {"loss": loss, "grads": mrhs_nn_get_grads(lat.ctx), "weights": mrhs_nn_get_weights(lat.ctx)}


def work(case):
    """Operands once, results once; the products of D (1872 flop per site and vector), P, D_c and the network."""
    kind, dims, agg = case["kind"], _dims(case), _agg(case)
    V, Va = int(np.prod(dims)), int(np.prod(agg))
    n = case.get("ntv") or case["nrhs"]
    e = BYTES[case.get("dtype") or case.get("prec") or "f32"]
    r = 8 if e == 8 else 4
    field, ops = 24 * n * V * e, 144 * r * V
    nc, nagg = 2 * n, V // Va
    dc, cfield = 9 * nc * nc * 2 * r * nagg, nc * 2 * n * r * nagg
    mr_flops = lambda sweeps, mr: V * n * sweeps * (1872 + mr * (1872 + 336))  # noqa: E731
    gs_flops, dc_flops = 2 * 8 * n * n * 12 * V, V * 2 * n * 936 + nagg * 8 * nc * nc * 6 * Va * 2
    if kind == "stencil":
        return {"bytes": ops + 2 * field, "flops": 1872 * V * n}
    if kind == "smoother":
        return {"bytes": ops + (3 if case["guess"] else 2) * field, "flops": mr_flops(case["sweeps"], case["mr"])}
    if kind == "coarse_operator":
        return {"bytes": ops + 24 * n * V * r * 2 + field + dc + 2 * cfield,
                "flops": gs_flops + dc_flops + 2 * 8 * n * n * 12 * V + nagg * 9 * nc * nc * 8 * n}
    if kind == "coarse_solve":
        return {"bytes": dc + 2 * cfield, "flops": case["iters"] * nagg * 9 * nc * nc * 8 * n}
    if kind == "setup":
        k = case["refine"]
        return {"bytes": ops + 24 * n * V * r + 2 * field + dc,
                "flops": mr_flops(5, 4) + k * mr_flops(4, 4) + (k + 1) * (gs_flops + dc_flops)
                + k * (2 * 8 * n * n * 12 * V + case["iters"] * nagg * 9 * nc * nc * 8 * n)}
    if kind == "solve":  # D_c, P and the links once, and what ten V-cycles of one vector compute
        return {"bytes": ops + field + dc, "flops": 10 * V * 4 * (1872 + 4 * 2208) + 100 * nagg * 9 * nc * nc * 8}
    w = case["width"]
    conv = 9 * V * n * (8 * 3 * (4 * w + w * w + 4 * w) + 72 * (4 + 2 * w))
    if kind == "infer":
        return {"bytes": 288 * V + 2 * field, "flops": conv}
    return {"bytes": 288 * V + ops + 3 * field, "flops": 3 * conv + 2 * 1872 * V * n}


# --------------------------------------------------- the same in 64 bits -----
class _Exact:
    """The Wilson-clover operator and the steps of the setup on tensors
    psi[t][z][y][x][spin][colour][vector] in complex128."""

    def __init__(self, dims, agg, U):
        self.dims, self.agg = dims, agg
        self.V, self.Va = int(np.prod(dims)), int(np.prod(agg))
        self.nb = [d // a for d, a in zip(dims, agg)]
        self.nagg = self.V // self.Va
        self.grid = tuple(dims[::-1])
        self.U = [u.contiguous() for u in U.reshape(*self.grid, 4, 3, 3).unbind(4)]
        c = dict(dtype=torch.complex128, device="cuda")
        sig = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], **c)
        self.gamma = torch.zeros(4, 4, 4, **c)
        for k in range(3):
            self.gamma[k, :2, 2:], self.gamma[k, 2:, :2] = -1j * sig[k], 1j * sig[k]
        self.gamma[3, :2, 2:] = self.gamma[3, 2:, :2] = torch.eye(2, **c)
        at = [torch.arange(d, device="cuda") for d in dims]
        self.blk = sum((at[m] // agg[m]).reshape([-1 if k == 3 - m else 1 for k in range(4)]) for m in range(4)) % 2

    def shift(self, f, mu, d, fermion=False):
        """f(x + d mu), antiperiodic in t for fermions."""
        f = torch.roll(f, -d, 3 - mu)
        if fermion and mu == 3:
            f[-1 if d > 0 else 0] *= -1
        return f

    def stays(self, mu, d):
        """1 where x + d mu is in the aggregate of x."""
        at = torch.arange(self.dims[mu], device="cuda") % self.agg[mu]
        m = at != (self.agg[mu] - 1 if d > 0 else 0)
        return m.reshape([-1 if k == 3 - mu else 1 for k in range(4)] + [1, 1, 1])

    def clover(self):
        """A(x) as 12 x 12 matrices."""
        A = torch.zeros(*self.grid, 4, 3, 4, 3, dtype=torch.complex128, device="cuda")
        for mu in range(4):
            for nu in range(mu + 1, 4):
                u, v = self.U[mu], self.U[nu]
                S = self.shift
                um, vm, vn, un = S(u, mu, -1), S(v, mu, -1), S(v, nu, -1), S(u, nu, -1)
                Q = u @ S(v, mu, 1) @ S(u, nu, 1).mH @ v.mH
                Q += v @ S(um, nu, 1).mH @ vm.mH @ um
                Q += um.mH @ S(vm, nu, -1).mH @ S(um, nu, -1) @ vn
                Q += vn.mH @ un @ S(vn, mu, 1) @ u.mH
                sigma = 0.5j * (self.gamma[mu] @ self.gamma[nu] - self.gamma[nu] @ self.gamma[mu])
                A += 0.5j * CSW / 8 * torch.einsum("ij,tzyxab->tzyxiajb", sigma, Q - Q.mH)
        A = A.reshape(*self.grid, 12, 12)
        A.diagonal(dim1=-2, dim2=-1).add_(4 + M0)
        return A

    def hops(self, psi, out, inside):
        """out -= the hopping terms; inside: only those within an aggregate (True), only those that leave one
        (False), or all of them (None)."""
        for mu in range(4):
            for d in (1, -1):
                h = psi if d > 0 else torch.matmul(self.U[mu].mH.unsqueeze(4), psi)
                h = self.shift(h, mu, d, True)
                h = h - d * torch.einsum("ij,tzyxjcn->tzyxicn", self.gamma[mu], h)
                if d > 0:
                    h = torch.matmul(self.U[mu].unsqueeze(4), h)
                if inside is not None:
                    h *= self.stays(mu, d) == inside
                out -= 0.5 * h
        return out

    def D(self, psi, inside=None):
        if not hasattr(self, "A"):
            self.A = self.clover()
        out = (self.A @ psi.reshape(*self.grid, 12, -1)).reshape(psi.shape)
        return self.hops(psi, out, inside)

    # device layouts: sites aggregate by aggregate, [site][component][re, im][vector]
    def load(self, f):
        n = f.numel() // (24 * self.V)
        f = f.double().reshape(self.V, 12, 2, n)
        f = torch.complex(f[:, :, 0], f[:, :, 1])
        f = f.reshape(*self.nb[::-1], *self.agg[::-1], 4, 3, n).permute(0, 4, 1, 5, 2, 6, 3, 7, 8, 9, 10)
        return f.reshape(*self.grid, 4, 3, n)

    def aggregates(self, psi):
        """[aggregate][chirality][site and component][vector]"""
        n = psi.shape[-1]
        p = [x for m in (3, 2, 1, 0) for x in (self.nb[m], self.agg[m])]
        f = psi.reshape(*p, 2, 6, n).permute(0, 2, 4, 6, 8, 1, 3, 5, 7, 9, 10)
        return f.reshape(self.nagg, 2, self.Va * 6, n)

    def sites(self, f):
        n = f.shape[-1]
        f = f.reshape(*self.nb[::-1], 2, *self.agg[::-1], 6, n).permute(0, 5, 1, 6, 2, 7, 3, 8, 4, 9, 10)
        return f.reshape(*self.grid, 4, 3, n)

    def store(self, psi):
        n = psi.shape[-1]
        f = self.aggregates(psi).reshape(self.nagg, 2, self.Va, 6, n).permute(0, 2, 1, 3, 4).reshape(-1, n)
        return torch.stack((f.real, f.imag), 1).reshape(-1)

    def load_c(self, f, ntv):
        f = f.double().reshape(self.nagg, 2 * ntv, 2, -1)
        return torch.complex(f[:, :, 0], f[:, :, 1])

    def store_c(self, f):
        return torch.stack((f.real, f.imag), 2).reshape(-1)

    def smooth(self, b, x, sweeps, mr):
        on = [(self.blk == c).reshape(*self.grid, 1, 1, 1) for c in (0, 1)]
        for _ in range(sweeps):
            for c in (0, 1):
                rho = (b - self.D(x)) * on[c]
                for _ in range(mr):
                    q = self.D(rho, True)
                    a, r = self.aggregates(q), self.aggregates(rho)
                    qq = (a.real.square() + a.imag.square()).sum((1, 2))
                    al = (a.conj() * r).sum((1, 2)) / qq.clamp_min(1e-300)
                    al = al.reshape(self.nagg, 1, 1, -1)
                    x = x + self.sites(al * r)
                    rho = self.sites(r - al * a)
        return x

    def orthonormal(self, v):
        """The Q factor with positive diagonal per aggregate and chirality: Cholesky-QR, repeated."""
        q = self.aggregates(v)
        for _ in range(3):
            L = torch.linalg.cholesky(q.mH @ q)
            q = torch.linalg.solve_triangular(L, q.mH, upper=False).mH
        return q

    def R(self, P, v):
        return (P.mH @ self.aggregates(v)).reshape(self.nagg, -1, v.shape[-1])

    def prolong(self, P, u):
        return self.sites(P @ u.reshape(self.nagg, 2, -1, u.shape[-1]))

    def Dc(self, P, u, inside=None):
        return self.R(P, self.D(self.prolong(P, u), inside))

    def couple(self, P, u):
        """The hop blocks of D_c alone."""
        f = self.prolong(P, u)
        return self.R(P, self.hops(f, torch.zeros_like(f), False))

    def coarse_solve(self, P, b, iters, even_odd):
        if not even_odd:
            return _gmres(lambda x: self.Dc(P, x), b, iters)
        nc = b.shape[1]
        e = torch.eye(nc, dtype=b.dtype, device="cuda").expand(self.nagg, nc, nc).contiguous()
        inv = torch.linalg.inv(torch.cat([self.Dc(P, e[:, :, k:k + 8].contiguous(), True) for k in range(0, nc, 8)], 2))
        corner = [torch.arange(m, device="cuda") for m in self.nb]
        col = sum(corner[m].reshape([-1 if k == 3 - m else 1 for k in range(4)]) for m in range(4)) % 2
        ev = (col == 0).reshape(-1, 1, 1)

        def schur(x):
            u = (inv @ self.couple(P, x)) * ~ev
            return self.Dc(P, x, True) * ev - self.couple(P, u) * ev

        x = _gmres(schur, (b - self.couple(P, (inv @ b) * ~ev)) * ev, iters)
        return x + (inv @ (b - self.couple(P, x))) * ~ev


def _gmres(op, b, iters, restart=20):
    """Restarted GMRES from zero, every vector its own Krylov space, a given number of steps."""
    dot = lambda p, q: (p.conj() * q).sum((0, 1))  # noqa: E731
    x, left = torch.zeros_like(b), iters
    while left > 0:
        r = b - op(x)
        beta = dot(r, r).real.sqrt()
        m = min(left, restart)
        V, H = [r / beta], torch.zeros(b.shape[2], m + 1, m, dtype=b.dtype, device="cuda")
        for k in range(m):
            w = op(V[k])
            for _ in range(2):
                for i in range(k + 1):
                    h = dot(V[i], w)
                    H[:, i, k] += h
                    w = w - h * V[i]
            H[:, k + 1, k] = dot(w, w).real.sqrt()
            V.append(w / H[:, k + 1, k])
        rhs = torch.zeros(b.shape[2], m + 1, 1, dtype=b.dtype, device="cuda")
        rhs[:, 0, 0] = beta
        Qr, Rr = torch.linalg.qr(H)
        y = torch.linalg.solve_triangular(Rr, Qr.mH @ rhs, upper=True)
        for k in range(m):
            x = x + y[:, k, 0] * V[k]
        left -= m
    return x


def _bicgstab(op, b, tol=1e-14, most=4000):
    dot = lambda p, q: (p.conj() * q).sum()  # noqa: E731
    x = torch.zeros_like(b)
    goal = tol * dot(b, b).real.sqrt()
    done = 0
    while done < most:  # restarted from the true residual, so that the answer is as good as 64 bits give
        r = b - op(x)
        if dot(r, r).real.sqrt() <= 10 * goal:
            break
        r0, p = r.clone(), r.clone()
        rho = dot(r0, r)
        for _ in range(400):
            done += 1
            v = op(p)
            al = rho / dot(r0, v)
            t = r - al * v
            w = op(t)
            om = dot(w, t) / dot(w, w)
            x = x + al * p + om * t
            r = t - om * w
            if dot(r, r).real.sqrt() <= goal:
                break
            new = dot(r0, r)
            p = r + new / rho * al / om * (p - om * v)
            rho = new
    return x


def _network(E, W, bias, v):
    """The generator on v: per layer the nine transported neighbours mixed over the channels, modReLU between."""
    h = v
    for layer, w in enumerate(W):
        z = torch.einsum("oc,tzyxcan->tzyxoan", w[0], h)
        for mu in range(4):
            up = torch.matmul(E.U[mu].unsqueeze(4), E.shift(h, mu, 1, True))
            z = z + torch.einsum("oc,tzyxcan->tzyxoan", w[1 + mu], up)
            dn = E.shift(torch.matmul(E.U[mu].mH.unsqueeze(4), h), mu, -1, True)
            z = z + torch.einsum("oc,tzyxcan->tzyxoan", w[5 + mu], dn)
        if layer < 2:
            size = (z.real.square() + z.imag.square()).sum(5, keepdim=True).sqrt()
            z = z * (torch.relu(size + bias[layer].reshape(-1, 1, 1)) / size)
        h = z
    return h


def exact(case, seed):
    kind, n = case["kind"], case.get("ntv") or case["nrhs"]
    wd = "f64" if "f64" in (case.get("prec"), case.get("dtype")) else "f32"
    E = _Exact(_dims(case), _agg(case), _gauge(_dims(case), seed))
    fine, coarse = E.V * 24 * n, E.nagg * 2 * n * 2 * n
    if kind == "stencil":
        return E.store(E.D(E.load(_normal(fine, seed, 2, case["dtype"]))))
    if kind == "smoother":
        out = torch.empty(E.V * 24, n, dtype=torch.float64, device="cuda")
        b = _normal(fine, seed, 2, wd).reshape(-1, n)
        x = _normal(fine, seed, 3, wd).reshape(-1, n) if case["guess"] else torch.zeros_like(b)
        for k in range(0, n, 8):  # a few vectors at a time
            f = E.smooth(E.load(b[:, k:k + 8]), E.load(x[:, k:k + 8]), case["sweeps"], case["mr"])
            out[:, k:k + 8] = E.store(f).reshape(E.V * 24, -1)
        return out.reshape(-1)
    if kind == "solve":
        b = torch.view_as_complex(torch.randn(E.V, 12, 2, generator=_gen(seed, 5), device="cuda", dtype=torch.float64))
        x = _bicgstab(E.D, b.reshape(*E.grid, 4, 3, 1))
        return x.reshape(E.V, 12).cpu().numpy()
    if kind == "infer" or kind == "train":
        flat = torch.from_numpy(_weights(case["width"], seed)).cuda().double().requires_grad_(kind == "train")
        c = (4, case["width"], case["width"], 4)
        W, at = [], 0
        for i, o in zip(c[:3], c[1:]):
            W.append(torch.view_as_complex(flat[at:at + 18 * i * o].reshape(9, o, i, 2)))
            at += 18 * i * o
        bias = flat[at:].reshape(2, -1)
        v = _network(E, W, bias, E.load(_normal(fine, seed, 3)))
        if kind == "infer":
            return E.store(v)
        P = E.orthonormal(E.load(_normal(fine, seed, 2)))
        Dv, q = E.D(v), v - E.prolong(P, E.R(P, v))
        two = lambda f: (f.real.square() + f.imag.square()).sum((0, 1, 2, 3, 4, 5))  # noqa: E731
        loss = ((two(Dv) + LAMBDA * two(q)) / two(v)).sum()
        loss.backward()
        g = flat.grad
        return {"loss": float(loss.detach()), "grads": g.cpu().numpy(),
                "weights": (flat.detach() - LR * g / (g.abs() + 1e-8)).cpu().numpy()}
    tv = E.load(_normal(fine, seed, 2, wd))
    vc = E.load_c(_normal(coarse, seed, 4, wd), n)
    if kind == "coarse_operator":
        P = E.orthonormal(tv)
        vc = E.R(P, tv)
        return {"P": E.store(E.sites(P)), "vc": E.store_c(vc), "yc": E.store_c(E.Dc(P, vc))}
    if kind == "coarse_solve":
        return E.store_c(E.coarse_solve(E.orthonormal(tv), vc, case["iters"], case["even_odd"]))
    # a whole setup
    size = lambda f: (f.real.square() + f.imag.square()).sum((0, 1, 2, 3, 4, 5)).sqrt()  # noqa: E731
    v = E.smooth(tv, torch.zeros_like(tv), 5, 4)
    P = E.orthonormal(v / size(v))
    for _ in range(case["refine"]):
        v = v / size(v)
        v = E.smooth(v, E.prolong(P, E.coarse_solve(P, E.R(P, v), case["iters"], case["even_odd"])), 4, 4)
        P = E.orthonormal(v / size(v))
    return {"P": E.store(E.sites(P)), "yc": E.store_c(E.Dc(P, vc))}
