"""Measured work of the structured-multigrid library: what a user's program has
it do, through paper_2506_21932_gb300.smg (and the C ABI below it).

A case is one call, or the short chain of calls a program makes for one
result:
  vcycle  one V(1,1)-cycle on a hierarchy the program keeps (the
          preconditioner of an outer iteration of the program's own)
  solve   one Krylov solve on a hierarchy the program keeps (a new
          right-hand side per time step, the same matrix)
  tts     set-up plus solve (a new matrix per time step)
  setup   set-up plus the first V-cycle on it
  train   one training pair and one Adam step of the learned post-smoother
  cnn     one forward pass of the learned post-smoother's network
Sizes are those of the repository's configurations (benchmark and tests) or
of the same kind: every level halves all dimensions (or x and y), so extents
are a small number, odd ones among them, times a power of two.

exact() is plain torch in 64 bits, built here from the definitions: Galerkin
products by probing, lexicographic sweeps and ILU(0) by wavefronts, lines by
dense inverses, solves by other methods (sine transforms, Jacobi CG).
"""
import itertools
import math

import torch

from paper_2506_21932_gb300 import inputs as I
from paper_2506_21932_gb300 import smg as S

SMOOTHER = {"sgs": S.SGS, "ilu0": S.ILU0, "lgs": S.LGS}
TRANSFER = {"fw27v": S.FW27V, "pc8c": S.PC8C, "c64c": S.C64C, "c16xy": S.C16XY}
PRECISION = {"fp64": S.FP64, "fp32": S.FP32, "bf16": S.BF16}
KRYLOV = {"pcg": S.PCG, "fpcg": S.FPCG, "fgmres": S.FGMRES}


def _case(name, do, gen, dims, smoother, transfer="fw27v", precision="fp64", krylov="pcg", tol=1e-9, iters=0):
    c = {"do": do, "gen": gen, "nx": dims[0], "ny": dims[1], "nz": dims[2], "smoother": smoother,
         "transfer": transfer, "precision": precision, "krylov": krylov, "tol": tol, "iters": iters}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # small 7-point Poisson problem, symmetric GS, PCG: everything in L2, latency and launches count
        _case("poisson7_32_sgs_solve", "solve", "lap", (32, 32, 32), "sgs", iters=6),
        # small 27-point problem with odd coarsest extents, ILU(0), PCG: a subdomain or a test problem
        _case("aniso27_40x24x56_ilu0_solve", "solve", "q1", (40, 24, 56), "ilu0", iters=26),
        # the headline metric: a new 27-point anisotropic matrix, hierarchy set-up and PCG solve, 16.8 M unknowns
        _case("aniso27_256_ilu0_tts", "tts", "q1", (256, 256, 256), "ilu0", iters=41),
        # the largest configuration's V-cycle, FP64, 56.6 M unknowns
        _case("aniso27_384_ilu0_vcycle", "vcycle", "q1", (384, 384, 384), "ilu0"),
        # the FP32 hierarchy under a flexible FP64 outer iteration
        _case("aniso27_256_ilu0_fp32_vcycle", "vcycle", "q1", (256, 256, 256), "ilu0", precision="fp32",
              krylov="fpcg"),
        # BF16 storage with row scales on a ragged box (coarsest 13 x 9 x 11)
        _case("aniso27_208x144x176_bf16_vcycle", "vcycle", "q1", (208, 144, 176), "ilu0", precision="bf16",
              krylov="fpcg"),
        # three coupled unknowns per cell (layered reservoir), block GS, FGMRES(30)
        _case("block3_128x128x64_fgmres_solve", "solve", "blk", (128, 128, 64), "sgs", "pc8c", krylov="fgmres",
              tol=1e-8, iters=54),
        # variable-coefficient 7-point diffusion, symmetric GS (27-point coarse levels)
        _case("varcoef7_256_sgs_vcycle", "vcycle", "fv", (256, 256, 256), "sgs"),
        # the same family with ILU(0) and the cell-centred transfers: a new matrix every step, one cycle on it
        _case("varcoef7_160x96x224_c64c_setup", "setup", "fv", (160, 96, 224), "ilu0", "c64c", krylov="fpcg"),
        # strong coupling along z: line Gauss-Seidel
        _case("zaniso27_128x112x128_lgs_vcycle", "vcycle", "q1z", (128, 112, 128), "lgs"),
        # the same with x-y semi-coarsening (whole columns on every level) under FGMRES(30)
        _case("zaniso27_64x64x128_semi_tts", "tts", "q1z", (64, 64, 128), "lgs", "c16xy", krylov="fgmres", iters=7),
        # training of the learned post-smoother: forward, backward, update
        _case("cnn_train_64", "train", "fv", (64, 64, 64), "sgs", krylov="fpcg"),
    ]


def _box(rng, lo, hi, semi=False):
    """Extents c * 2^L, 4 <= c <= 13 in every coarsened dimension, volume log-uniform in [lo, hi]."""
    while True:
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        c = [rng.randint(4, 13) for _ in range(3)]
        if semi:
            c[2] = 16 * rng.randint(2, 8) + 2 * rng.randint(0, 7)
            c[0], c[1] = rng.randint(4, 7), rng.randint(4, 7)
        L = max(1, round(math.log2(want / (c[0] * c[1] * c[2])) / (2 if semi else 3)))
        d = [c[0] << L, c[1] << L, c[2] if semi else c[2] << L]
        if lo / 2 <= d[0] * d[1] * d[2] <= hi and max(d) <= 512:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["solve7", "solve27", "tts27", "vcycle27", "vcycle27", "low27", "block", "varcoef", "c64c",
                       "lgs", "semi", "train", "cnn"])
    if kind == "solve7":
        return _case("", "solve", "lap", _box(rng, 2 ** 12, 2 ** 21), "sgs", iters=7)
    if kind == "solve27":
        return _case("", "solve", "q1", _box(rng, 2 ** 13, 2 ** 20), "ilu0", iters=28)
    if kind == "tts27":
        return _case("", "tts", "q1", _box(rng, 2 ** 18, 2 ** 23), "ilu0", iters=36)
    if kind == "vcycle27":
        return _case("", "vcycle", "q1", _box(rng, 2 ** 13, 2 ** 25), rng.choice(["ilu0", "ilu0", "sgs"]))
    if kind == "low27":
        return _case("", "vcycle", "q1", _box(rng, 2 ** 15, 2 ** 25), rng.choice(["ilu0", "ilu0", "sgs"]),
                     precision=rng.choice(["fp32", "bf16"]), krylov="fpcg")
    if kind == "block":
        return _case("", "vcycle", "blk", _box(rng, 2 ** 13, 2 ** 20), "sgs", "pc8c",
                     precision=rng.choice(["fp64", "fp32"]), krylov="fgmres")
    if kind == "varcoef":
        return _case("", "vcycle", "fv", _box(rng, 2 ** 15, 2 ** 24), "sgs")
    if kind == "c64c":
        return _case("", "setup", "fv", _box(rng, 2 ** 15, 2 ** 22), "ilu0", "c64c", krylov="fpcg")
    if kind == "lgs":
        return _case("", "vcycle", "q1z", _box(rng, 2 ** 14, 2 ** 22), "lgs")
    if kind == "semi":
        return _case("", "tts", "q1z", _box(rng, 2 ** 14, 2 ** 19, semi=True), "lgs", "c16xy", krylov="fgmres", iters=7)
    if kind == "train":
        return _case("", "train", "fv", _box(rng, 2 ** 14, 2 ** 19), "sgs", krylov="fpcg")
    return _case("", "cnn", "fv", _box(rng, 2 ** 15, 2 ** 24), "sgs", krylov="fpcg")


def _dims(c):
    return c["nx"], c["ny"], c["nz"]


def _matrix(c, seed, dev="cuda"):
    """(offsets, coefficients, log coefficient field or None)."""
    d = _dims(c)
    if c["gen"] == "lap":
        return I.OFF7, I.laplace7(d, device=dev), None
    if c["gen"] == "q1":
        return I.OFF27, I.q1_aniso27(d, seed, device=dev).contiguous(), None
    if c["gen"] == "q1z":
        return I.OFF27, I.q1_aniso27(d, seed, aniso=(1e-3, 1e-3, 1.0), device=dev).contiguous(), None
    if c["gen"] == "fv":
        A, g = I.varcoef7(d, seed, device=dev)
        return I.OFF7, A.contiguous(), g.contiguous()
    return I.OFF7, I.block7_layered(d, seed, device=dev), None


def _vector(n, seed):
    """Right-hand side: iid uniform on [-1, 1], the benchmark's distribution, drawn on the device."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2 + 1)
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * 2.0 - 1.0


def _normal(n, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2 + 1)
    return torch.randn(n, generator=g, dtype=dtype, device="cuda")


def _build(c, off, A):
    return S.SMG(_dims(c), off, A, block=3 if c["gen"] == "blk" else 1, smoother=SMOOTHER[c["smoother"]],
                 transfer=TRANSFER[c["transfer"]], precision=PRECISION[c["precision"]], krylov=KRYLOV[c["krylov"]])


def prepare(case, seed):
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    s = {"case": c}
    if c["do"] == "cnn":
        s.update(theta=I.cnn_theta(seed).cuda(), in2=_normal(2 * n, seed, torch.float32),
                 out=torch.empty(n, dtype=torch.float32, device="cuda"), ws=S.cnn_workspace(_dims(c)))
        return s
    off, A, logk = _matrix(c, seed)
    if c["do"] == "train":
        theta = I.cnn_theta(seed).cuda()
        s.update(h=_build(c, off, A), logk=logk, e0=_normal(n, seed, torch.float64), theta=theta,
                 m=torch.zeros_like(theta), v=torch.zeros_like(theta), grad=torch.empty_like(theta),
                 loss=torch.empty(1, dtype=torch.float32, device="cuda"), ws=S.cnn_workspace(_dims(c)),
                 in2=torch.empty(2 * n, dtype=torch.float32, device="cuda"),
                 target=torch.empty(n, dtype=torch.float32, device="cuda"), step=0)
        return s
    b = _vector(n * (3 if c["gen"] == "blk" else 1), seed)
    s.update(off=off, b=b, x=torch.empty_like(b))
    if c["do"] in ("tts", "setup"):
        s["A"] = A
    else:
        s["h"] = _build(c, off, A)
    return s


def run(state):
    s, c = state, state["case"]
    if c["do"] == "vcycle":
        s["h"].vcycle(s["b"], s["x"])
        return s["x"]
    if c["do"] == "solve":
        s["x"].zero_()
        it, _, _ = s["h"].solve(s["b"], s["x"], tol=c["tol"], maxit=500)
        return {"x": s["x"], "iterations": it}
    if c["do"] == "tts":
        h = _build(c, s["off"], s["A"])
        s["x"].zero_()
        it, _, _ = h.solve(s["b"], s["x"], tol=c["tol"], maxit=500)
        h.close()
        return {"x": s["x"], "iterations": it}
    if c["do"] == "setup":
        h = _build(c, s["off"], s["A"])
        h.vcycle(s["b"], s["x"])
        h.close()
        return s["x"]
    if c["do"] == "cnn":
        S.cnn_forward(_dims(c), s["theta"], s["in2"], s["out"], s["ws"])
        return s["out"]
    s["grad"].zero_()
    s["loss"].zero_()
    s["h"].learned_sample(s["e0"], s["logk"], s["in2"], s["target"])
    s["h"].learned_loss_grad(s["theta"], s["in2"], s["target"], s["grad"], s["loss"], s["ws"], S.LOSS_RESIDUAL)
    s["step"] += 1
    S.cnn_adam(s["theta"], s["m"], s["v"], s["grad"], s["step"])
    return {"in2": s["in2"], "target": s["target"], "loss": s["loss"], "grad": s["grad"], "theta": s["theta"],
            "m": s["m"], "v": s["v"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _level_dims(c):
    d, out = list(_dims(c)), []
    semi = c["transfer"] == "c16xy"
    while True:
        out.append(tuple(d))
        cut = d[:2] if semi else d
        if min(cut) < 8 or any(t & 1 for t in cut):
            return out
        d = [d[0] // 2, d[1] // 2, d[2] if semi else d[2] // 2]


def _levels(c):
    """(points, stencil entries) of every level."""
    ns = 27 if c["gen"] in ("q1", "q1z") else 7
    out = []
    for d in _level_dims(c):
        out.append((d[0] * d[1] * d[2], ns))
        ns = 7 if c["transfer"] == "pc8c" else 27
    return out


def _vcycle_work(c):
    """A V(1,1)-cycle goes through the matrix of a level twice for the two
    smoothings (an ILU(0) solve pair, or a symmetric sweep: once from zero, so
    half of it) and once or twice for residuals; vectors move between them."""
    val = {"fp64": 8, "fp32": 4, "bf16": 2}[c["precision"]]
    vec = 8 if c["precision"] == "fp64" else 4
    bb, B = (9, 3) if c["gen"] == "blk" else (1, 1)
    lv = _levels(c)
    nbytes = flops = 0.0
    for n, ns in lv[:-1]:
        passes = 4 * ns if c["smoother"] == "ilu0" else 4.5 * ns
        nbytes += n * (passes * bb * val + 14 * B * vec)
        flops += n * 2 * passes * bb
    nc = lv[-1][0] * B
    return nbytes + 8.0 * nc * nc, flops + 2.0 * nc * nc


def _setup_work(c):
    """Read the matrix; write its coarse levels and every level's smoother data."""
    bb = 9 if c["gen"] == "blk" else 1
    lv = _levels(c)
    entries = [n * ns * bb for n, ns in lv]
    flops = sum(2.0 * n * 27 * ns * bb for n, ns in lv[:-1]) + sum(2.0 * e * (8 if c["smoother"] == "ilu0" else 1)
                                                                   for e in entries[:-1])
    nc = lv[-1][0] * (3 if bb == 9 else 1)
    return 8.0 * (entries[0] + 2 * sum(entries[1:]) + 2 * sum(entries[:-1])) + 16.0 * nc * nc, flops + 2.0 * nc ** 3


def work(case):
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    if c["do"] == "cnn":
        return {"bytes": 12.0 * n, "flops": 2.0 * 27 * (2 * 16 + 16 * 16 + 16) * n}
    vb, vf = _vcycle_work(c)
    if c["do"] == "vcycle":
        return {"bytes": vb, "flops": vf}
    if c["do"] == "train":
        # the V-cycle, A applied four times, the network forward and twice backward
        return {"bytes": vb + 4 * n * (7 + 2) * 8.0, "flops": vf + 4 * 14.0 * n + 6.0 * 27 * (32 + 256 + 16) * n}
    B = 3 if c["gen"] == "blk" else 1
    ns = _levels(c)[0][1]
    it = max(1, c["iters"])
    # per iteration: one V-cycle, one product with A, and the Krylov vectors
    solve_b = it * (vb + 8.0 * n * (ns * B * B + 12 * B))
    solve_f = it * (vf + 2.0 * n * (ns * B * B + 6 * B))
    sb, sf = _setup_work(c)
    if c["do"] == "solve":
        return {"bytes": solve_b, "flops": solve_f}
    if c["do"] == "setup":
        return {"bytes": sb + vb, "flops": sf + vf}
    return {"bytes": sb + solve_b, "flops": sf + solve_f}


def tolerance(case):
    c = case
    if c["do"] == "cnn":
        return {"rel": 1e-3}  # BF16 activations between layers, FP32 sums: a sum's order moves a few roundings
    if c["do"] == "train":
        return {"rel": 2e-3, "max": 0.1}  # the same, through the backward pass
    if c["do"] in ("solve", "tts"):
        # both answers leave a residual of tol; the part of the error that rounding moves is far smaller
        return {"rel": 1e-8, "max": 1e-6}
    # one V-cycle: sums of at most 27 terms at the hierarchy's precision, through every level (measured against
    # exact(): 2e-16 to 2e-14 in FP64, 1e-7 in FP32; BF16 is storage only, its sums are FP32)
    return {"rel": 1e-12, "max": 1e-10} if c["precision"] == "fp64" else {"rel": 2e-6, "max": 2e-4}


# ---------------------------------------------------------------------------
# 64-bit references from the definitions
# ---------------------------------------------------------------------------

def _prolong1(c, kind):
    """Interpolation along dimension 0 (n -> 2n)."""
    lo, hi = torch.zeros_like(c), torch.zeros_like(c)
    lo[1:], hi[:-1] = c[:-1], c[1:]
    f = torch.empty((2 * c.shape[0],) + c.shape[1:], dtype=c.dtype, device=c.device)
    if kind == "fw27v":
        f[1::2], f[0::2] = c, 0.5 * (c + lo)
    else:
        f[0::2], f[1::2] = 0.75 * c + 0.25 * lo, 0.75 * c + 0.25 * hi
    return f


def _restrict1(f, kind):
    if kind != "fw27v":
        return f[0::2] + f[1::2]
    nxt = torch.zeros_like(f[0::2])
    nxt[:-1] = f[2::2]
    return 0.5 * (f[1::2] + 0.5 * (f[0::2] + nxt))


class _Level:
    def __init__(self, dims, off, A):
        self.d, self.off, self.A = tuple(dims), [tuple(o) for o in off], A.reshape(*dims, len(off))
        nx, ny, nz = self.d
        self.n = nx * ny * nz
        self.lin = torch.tensor([(o[0] * (ny + 2) + o[1]) * (nz + 2) + o[2] for o in self.off], device="cuda")
        self.ec = self.off.index((0, 0, 0))

    def apply(self, x):
        nx, ny, nz = self.d
        xp = torch.nn.functional.pad(x.reshape(self.d), (1,) * 6)
        y = torch.zeros_like(x.reshape(self.d))
        for e, o in enumerate(self.off):
            y.addcmul_(self.A[..., e], xp[1 + o[0]:1 + o[0] + nx, 1 + o[1]:1 + o[1] + ny, 1 + o[2]:1 + o[2] + nz])
        return y

    def fronts(self):
        """Index tensors (plain, padded) of the points with equal 4i + 2j + k, in order."""
        nx, ny, nz = self.d
        ar = [torch.arange(t, device="cuda") for t in self.d]
        t = (4 * ar[0].view(-1, 1, 1) + 2 * ar[1].view(1, -1, 1) + ar[2].view(1, 1, -1)).reshape(-1).to(torch.int32)
        cnt = torch.bincount(t).tolist()
        idx = torch.sort(t, stable=True)[1]
        k, r = idx % nz, idx // nz
        pidx = ((r // ny + 1) * (ny + 2) + r % ny + 1) * (nz + 2) + k + 1
        return list(zip(idx.split(cnt), pidx.split(cnt)))

    def padded(self, x):
        return torch.nn.functional.pad(x.reshape(self.d), (1,) * 6).reshape(-1)

    def inner(self, xp):
        nx, ny, nz = self.d
        return xp.reshape(nx + 2, ny + 2, nz + 2)[1:-1, 1:-1, 1:-1].contiguous()

    def factor_ilu0(self):
        ns, ec = len(self.off), self.ec
        LU = self.A.reshape(self.n, ns).clone()
        where = {o: e for e, o in enumerate(self.off)}
        nx, ny, nz = self.d
        lin = [(o[0] * ny + o[1]) * nz + o[2] for o in self.off]
        plan = []
        for e in range(ec):
            src, dst = [], []
            for f in range(ec + 1, ns):
                q = tuple(a + b for a, b in zip(self.off[e], self.off[f]))
                if q in where:
                    src.append(f)
                    dst.append(where[q])
            plan.append((torch.tensor(src, device="cuda"), torch.tensor(dst, device="cuda")))
        for idx, _ in self.fronts():
            W = LU[idx]
            for e in range(ec):
                # an off-grid neighbour has coefficient zero: any row in range may stand for it
                q = (idx + lin[e]).clamp_(0, self.n - 1)
                row = LU[q]
                l = W[:, e] / row[:, ec]
                W[:, e] = l
                if len(plan[e][0]):
                    W[:, plan[e][1]] -= l[:, None] * row[:, plan[e][0]]
            LU[idx] = W
        self.LU = LU

    def triangular(self, M, entries, dinv, b, up, reverse):
        """Solves with the given entries and 1/diagonal, updating the padded vector up in order."""
        sel = torch.tensor(entries, device="cuda")
        lin = self.lin[sel]
        fr = self.fronts()
        for idx, p in (reversed(fr) if reverse else fr):
            r = b[idx] - (M[idx][:, sel] * up[p[:, None] + lin]).sum(1)
            up[p] = r if dinv is None else r * dinv[idx]

    def smooth(self, kind, f, u, first):
        """One symmetric step on A u = f; first: from u = 0 (u is then ignored)."""
        ns, ec = len(self.off), self.ec
        others = [e for e in range(ns) if e != ec]
        if kind == "ilu0":
            r = f if first else f - self.apply(u)
            y = torch.zeros(self.n + 0, dtype=torch.float64, device="cuda")
            yp = self.padded(y)
            self.triangular(self.LU, list(range(ec)), None, r.reshape(-1), yp, False)
            y = self.inner(yp).reshape(-1)
            zp = torch.zeros_like(yp)
            self.triangular(self.LU, list(range(ec + 1, ns)), 1.0 / self.LU[:, ec], y, zp, True)
            z = self.inner(zp)
            return z if first else u + z
        if kind == "sgs":
            M = self.A.reshape(self.n, ns)
            dinv = 1.0 / M[:, ec]
            up = self.padded(torch.zeros_like(f) if first else u)
            self.triangular(M, others, dinv, f.reshape(-1), up, False)
            self.triangular(M, others, dinv, f.reshape(-1), up, True)
            return self.inner(up)
        return self.smooth_lines(f, torch.zeros_like(f) if first else u)

    def smooth_lines(self, f, u):
        nx, ny, nz = self.d
        if not hasattr(self, "Tinv"):
            cols = self.A.reshape(nx * ny, nz, -1)
            T = torch.diag_embed(cols[:, :, self.ec])
            T += torch.diag_embed(cols[:, 1:, self.off.index((0, 0, -1))], offset=-1)
            T += torch.diag_embed(cols[:, :-1, self.off.index((0, 0, 1))], offset=1)
            self.Tinv = torch.linalg.inv(T)
        ar = [torch.arange(t, device="cuda") for t in (nx, ny)]
        t = (2 * ar[0].view(-1, 1) + ar[1].view(1, -1)).reshape(-1)
        idx = torch.sort(t, stable=True)[1]
        fr = idx.split(torch.bincount(t).tolist())
        up = torch.nn.functional.pad(u.reshape(self.d), (1,) * 6).reshape(-1, nz + 2)
        A, b = self.A.reshape(nx * ny, nz, -1), f.reshape(nx * ny, nz)
        by_column = {}
        for e, o in enumerate(self.off):
            if o[:2] != (0, 0):
                by_column.setdefault(o[:2], []).append((e, o[2]))
        for order in (fr, reversed(fr)):
            for col in order:
                pc = (col // ny + 1) * (ny + 2) + col % ny + 1
                r, Ac = b[col], A[col]
                for (dx, dy), es in by_column.items():
                    x = up[pc + dx * (ny + 2) + dy]
                    for e, dz in es:
                        r = r - Ac[:, :, e] * x[:, 1 + dz:1 + dz + nz]
                up[pc, 1:-1] = torch.bmm(self.Tinv[col], r[:, :, None])[:, :, 0]
        return up.reshape(nx + 2, ny + 2, nz + 2)[1:-1, 1:-1, 1:-1].contiguous()


class _Reference:
    """The V-cycle of a scalar problem in 64 bits."""

    def __init__(self, c, off, A):
        self.c, self.axes = c, (0, 1) if c["transfer"] == "c16xy" else (0, 1, 2)
        dims = _level_dims(c)
        self.L = [_Level(dims[0], off, A)]
        for d in dims[1:]:
            self.L.append(self.galerkin(self.L[-1], d))
        if c["smoother"] == "ilu0":
            for lv in self.L[:-1]:
                lv.factor_ilu0()

    def prolong(self, x):
        for ax in self.axes:
            x = _prolong1(x.movedim(ax, 0), self.c["transfer"]).movedim(0, ax)
        return x.contiguous()

    def restrict(self, x):
        for ax in self.axes:
            x = _restrict1(x.movedim(ax, 0), self.c["transfer"]).movedim(0, ax)
        return x.contiguous()

    def galerkin(self, F, d):
        """R A P by probing with the 27 colour vectors of a 27-point coarse operator."""
        A = torch.zeros(*d, 27, dtype=torch.float64, device="cuda")
        g = [torch.arange(t, device="cuda").view([-1 if a == ax else 1 for a in range(3)]) for ax, t in enumerate(d)]
        for col in itertools.product(range(3), repeat=3):
            e = torch.zeros(d, dtype=torch.float64, device="cuda")
            e[col[0]::3, col[1]::3, col[2]::3] = 1.0
            w = self.restrict(F.apply(self.prolong(e)))
            for q, o in enumerate(I.OFF27):
                ok = [((g[a] + o[a]) % 3 == col[a]) & (g[a] + o[a] >= 0) & (g[a] + o[a] < d[a]) for a in range(3)]
                m = ok[0] & ok[1] & ok[2]
                A[..., q] += w * m
        return _Level(d, I.OFF27, A)

    def vcycle(self, f, l=0):
        lv = self.L[l]
        f = f.reshape(lv.d)
        if l + 1 == len(self.L):
            M = torch.zeros(lv.n, lv.n, dtype=torch.float64, device="cuda")
            nx, ny, nz = lv.d
            p = torch.arange(lv.n, device="cuda")
            i, j, k = p // (ny * nz), (p // nz) % ny, p % nz
            for e, o in enumerate(lv.off):
                ok = (i + o[0] >= 0) & (i + o[0] < nx) & (j + o[1] >= 0) & (j + o[1] < ny) & (k + o[2] >= 0) & (k + o[2] < nz)
                M[p[ok], p[ok] + (o[0] * ny + o[1]) * nz + o[2]] = lv.A.reshape(lv.n, -1)[ok, e]
            return torch.linalg.solve(M, f.reshape(-1)).reshape(lv.d)
        u = lv.smooth(self.c["smoother"], f, None, True)
        u = u + self.prolong(self.vcycle(self.restrict(f - lv.apply(u)), l + 1))
        return lv.smooth(self.c["smoother"], f, u, False)


def _poisson(d, b):
    """Solution of the 7-point Laplacian by sine transforms."""
    x, lam = b.reshape(d), 0.0
    Q = []
    for ax, n in enumerate(d):
        m = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
        Q.append(math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi / (n + 1) * m.view(-1, 1) * m.view(1, -1)))
        lam = lam + (2.0 - 2.0 * torch.cos(math.pi * m / (n + 1))).view([-1 if a == ax else 1 for a in range(3)])
    for ax in range(3):
        x = torch.tensordot(Q[ax], x, dims=([1], [ax])).movedim(0, ax)
    x = x / lam
    for ax in range(3):
        x = torch.tensordot(Q[ax], x, dims=([1], [ax])).movedim(0, ax)
    return x.reshape(-1)


def _layered(d, A, b):
    """Solution of the layered 3-unknown system: sine transforms in x and y
    (its coefficients depend on z alone), a dense solve in z per mode."""
    nx, ny, nz = d
    M = A.reshape(nx, ny, nz, 7, 3, 3)[1, 1]  # any interior column: entries in the order of OFF7
    T = -M[:, 1, 0, 0]  # the coupling to a neighbour in y (the same in x)
    base = torch.zeros(nz, 3, nz, 3, dtype=torch.float64, device="cuda")
    k = torch.arange(nz, device="cuda")
    base[k, :, k, :] = M[:, 3]
    base[k[1:], :, k[:-1], :] = M[1:, 2]
    base[k[:-1], :, k[1:], :] = M[:-1, 4]
    Q, mu = [], []
    for n in (nx, ny):
        m = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
        Q.append(math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi / (n + 1) * m.view(-1, 1) * m.view(1, -1)))
        mu.append(2.0 * torch.cos(math.pi * m / (n + 1)))
    f = torch.einsum("ia,jb,abkr->ijkr", Q[0], Q[1], b.reshape(nx, ny, nz, 3))
    x = torch.empty_like(f)
    off = torch.zeros(nz, 3, nz, 3, dtype=torch.float64, device="cuda")
    for r in range(3):
        off[k, r, k, r] = T
    m3 = 3 * nz
    for i in range(nx):
        sys = base.reshape(1, m3, m3) - (mu[0][i] + mu[1]).view(-1, 1, 1) * off.reshape(1, m3, m3)
        x[i] = torch.linalg.solve(sys, f[i].reshape(ny, m3, 1)).reshape(ny, nz, 3)
    return torch.einsum("ia,jb,abkr->ijkr", Q[0], Q[1], x).reshape(-1)


def _jacobi_cg(lv, b, tol=1e-13, maxit=6000):
    D = lv.A[..., lv.ec]
    b = b.reshape(lv.d)
    x = torch.zeros_like(b)
    r = b.clone()
    z = r / D
    p, rho = z.clone(), (r * z).sum()
    stop = tol * float(b.norm())
    for it in range(maxit):
        q = lv.apply(p)
        a = rho / (p * q).sum()
        x += a * p
        r -= a * q
        if it % 25 == 24 and float(r.norm()) < stop:
            break
        z = r / D
        new = (r * z).sum()
        p = z + (new / rho) * p
        rho = new
    return x.reshape(-1)


def _network(theta, in2, d):
    """The post-smoother's network in 64 bits; theta in PyTorch's conv3d order."""
    x, at = in2.reshape(1, 2, *d), 0
    for l, (ci, co) in enumerate(zip(I.CNN_CHANNELS[:-1], I.CNN_CHANNELS[1:])):
        W = theta[at:at + co * ci * 27].reshape(co, ci, 3, 3, 3)
        bias = theta[at + co * ci * 27:at + co * ci * 27 + co]
        at += co * ci * 27 + co
        xp = torch.nn.functional.pad(x, (1,) * 6)
        # the convolution tap by tap (27 small products)
        y = bias.view(1, co, 1, 1, 1)
        for a, b, c in itertools.product(range(3), repeat=3):
            y = y + torch.einsum("oi,nixyz->noxyz", W[:, :, a, b, c],
                                 xp[:, :, a:a + d[0], b:b + d[1], c:c + d[2]])
        x = torch.relu(y) if l < 2 else y
    return x.reshape(-1)


def _train_exact(c, seed):
    d = _dims(c)
    n = d[0] * d[1] * d[2]
    off, A, logk = _matrix(c, seed)
    ref = _Reference(c, off, A)
    lv = ref.L[0]
    D = lv.A[..., lv.ec].reshape(-1)
    e0 = _normal(n, seed, torch.float64)
    e1 = e0 - ref.vcycle(lv.apply(e0)).reshape(-1)
    r1 = lv.apply(e1).reshape(-1)
    rms = r1.norm() / math.sqrt(n)
    in2 = torch.cat([r1 / rms, logk])
    theta = I.cnn_theta(seed).cuda().double().requires_grad_(True)
    y = _network(theta, in2, d)
    nx, ny, nz = d
    xp = torch.nn.functional.pad((y / D).reshape(d), (1,) * 6)
    Ay = sum(lv.A[..., e] * xp[1 + o[0]:1 + o[0] + nx, 1 + o[1]:1 + o[1] + ny, 1 + o[2]:1 + o[2] + nz]
             for e, o in enumerate(lv.off))
    loss = (Ay.reshape(-1) - in2[:n]).square().sum() / n
    grad, = torch.autograd.grad(loss, theta)
    m, v = 0.1 * grad, 0.001 * grad * grad
    new = theta.detach() - 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return {"in2": in2, "target": D * e1 / rms, "loss": loss.detach().reshape(1), "grad": grad, "theta": new, "m": m,
            "v": v}


def exact(case, seed):
    c = case
    d = _dims(c)
    n = d[0] * d[1] * d[2]
    if c["do"] == "cnn":
        if n > 2 ** 22:
            return None  # 64-bit activations of 16 channels and their taps: too much memory traffic
        return _network(I.cnn_theta(seed).cuda().double(), _normal(2 * n, seed, torch.float32).double(), d).detach()
    if c["do"] == "train":
        return _train_exact(c, seed)
    off, A, _ = _matrix(c, seed)
    b = _vector(n * (3 if c["gen"] == "blk" else 1), seed)
    if c["do"] in ("solve", "tts"):
        # the true solution; the iteration count has no 64-bit value of its own
        if c["gen"] == "lap":
            return {"x": _poisson(d, b), "iterations": None}
        if c["gen"] == "blk":
            return {"x": _layered(d, A, b), "iterations": None}
        if n > 2 ** 21:
            return None  # unpreconditioned iterations on the full 27-point matrix take minutes
        return {"x": _jacobi_cg(_Level(d, off, A), b), "iterations": None}
    if c["gen"] == "blk":
        return None  # the block sweeps by wavefronts take over 20 s
    if c["smoother"] == "lgs" and d[0] * d[1] * d[2] * d[2] * 8 > 2 ** 33:
        return None  # the dense line inverses do not fit
    return _Reference(c, off, A).vcycle(b).reshape(-1)
