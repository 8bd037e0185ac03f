"""The work that users of the library have it do, as cases that can be timed and compared.

Every case goes through a public entry point of paper_1509_06865_gb300 (mgeig_*), with
the sizes of workloads.json, the benchmark and the tests or sizes between them.  Inputs
are made on the GPU from the seed alone: SU(3) links U = exp(i eps H) with Gaussian H,
Gaussian or Z2 spinors.  `exact` computes the same outputs in 64 bits with plain torch.

Kinds of cases
  stencil  Q - sigma or D - sigma gamma5 on device fields: one field (the outer FGMRES
           matvec and every residual: FP64; the smoothers' operator: FP32) or many
           right-hand sides in one launch (the Z2 noise sources of stochastic estimates)
  project  one classical Gram-Schmidt step of a new vector against k earlier ones on the
           device (FP64: Algorithm 1 and the FGMRES Arnoldi process; FP32: the fine-grid
           deflation of the shifted solves)
  coarse   (Q_c - sigma) on many coarse vectors, FP32 or 16-bit links
  cycle    one two-grid preconditioner application on device spinors
  solve    (Q - sigma) x = b from host spinors to host spinors, the whole FGMRES solve
  grads    forward and backward pass of the learned smoother: loss and all gradients
  eig      a whole eigensolve: gauge load, setup and Algorithm 1
"""
import math

import numpy as np
import torch

from paper_1509_06865_gb300 import (FP64, LINKS_BF16, LINKS_F16, LINKS_LEVEL, MIXED, OP_D, OP_Q, PREC_F32, PREC_F64,
                                    Context)

LINKS = {"level": LINKS_LEVEL, "bf16": LINKS_BF16, "f16": LINKS_F16}


def listed():
    return [
        # the smallest call: a smoother's operator on a small lattice (the size the learned smoother trains on)
        dict(name="stencil_f32_8x8x8x8", kind="stencil", dims="8x8x8x8", prec="f32", op="Q", nrhs=1, eps=0.2,
             m0=-0.05, csw=1.9, bct=1, sigma=0.01),
        # the outer FGMRES matvec and the residuals of the 16^3 x 32 workload
        dict(name="stencil_f64_16x16x16x32", kind="stencil", dims="16x16x16x32", prec="f64", op="Q", nrhs=1,
             eps=0.2, m0=-0.0428, csw=1.9, bct=1, sigma=0.01),
        # D on twelve noise or point sources (spin x colour) at once, antiperiodic in time, the largest lattice
        dict(name="stencil_f32_nrhs12_32x32x32x64", kind="stencil", dims="32x32x32x64", prec="f32", op="D", nrhs=12,
             eps=0.15, m0=-0.02, csw=1.9, bct=-1, sigma=0.0),
        # Algorithm 1's Gram-Schmidt against 20 vectors, FP64 storage in the mixed solver
        dict(name="project_f64_k20_16x16x16x32", kind="project", n=1572864, k=20, prec="f64", mixed=True),
        # the fine-grid deflation of a shifted solve: 32 iterated vectors in FP32
        dict(name="project_f32_k32_16x16x16x32", kind="project", n=1572864, k=32, prec="f32", mixed=True),
        # the default coarse operator on twelve right-hand sides, the benchmark's coarse grid
        dict(name="coarse_f32_nrhs12_16x16x16x32", kind="coarse", dims="16x16x16x32", agg="4x4x4x4",
             sap="4x4x4x4", ntv=20, links="level", nrhs=12, eps=0.2, m0=-0.0428, csw=1.9, sigma=0.01),
        # the 16-bit coarse operator on twelve right-hand sides, the largest coarse grid
        dict(name="coarse_bf16_nrhs12_32x32x32x64", kind="coarse", dims="32x32x32x64", agg="4x4x4x4",
             sap="4x4x4x4", ntv=20, links="bf16", nrhs=12, eps=0.15, m0=-0.02, csw=1.9, sigma=0.01),
        # the preconditioner of every outer step of the benchmark, mixed precision
        dict(name="cycle_mixed_16x16x16x32", kind="cycle", dims="16x16x16x32", agg="4x4x4x4", sap="4x4x4x4", ntv=20,
             mixed=True, links="level", eps=0.2, m0=0.0172, csw=1.9, sigma=0.01),
        # the all-FP64 path's preconditioner on the check field
        dict(name="cycle_fp64_8x8x8x16", kind="cycle", dims="8x8x8x16", agg="4x4x4x4", sap="4x4x4x4", ntv=20,
             mixed=False, links="level", eps=0.2, m0=0.0172, csw=1.9, sigma=0.01),
        # a propagator from a noise source on the middle lattice of the batched solves, to 1e-12
        dict(name="solve_mixed_12x12x12x24", kind="solve", dims="12x12x12x24", agg="4x4x4x4", sap="3x3x3x3", ntv=20,
             mixed=True, links="level", eps=0.2, m0=0.0172, csw=1.9, sigma=0.01, tol=1e-12),
        # one gradient evaluation of the learned smoother, four pairs
        dict(name="grads_8x8x8x16_b4", kind="grads", dims="8x8x8x16", batch=4),
        # a whole eigensolve: the four lowest modes of the dense check lattice
        dict(name="eig_4x4x4x4_n4", kind="eig", dims="4x4x4x4", agg="2x2x2x2", sap="2x2x2x2", ntv=8, mixed=True,
             eps=0.3, m0=-0.4, csw=1.0, neig=4, tol=1e-10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, vmax, unit, per_dir):
    """Extents unit * (one of per_dir) with a volume of at most vmax, its logarithm spread evenly."""
    target = rng.uniform(math.log(unit ** 4 * min(per_dir) ** 4), math.log(vmax))
    best = None
    for _ in range(40):
        d = [unit * rng.choice(per_dir) for _ in range(4)]
        v = math.log(d[0] * d[1] * d[2] * d[3])
        if v <= math.log(vmax) and (best is None or abs(v - target) < best[0]):
            best = (abs(v - target), d)
    return "x".join(str(x) for x in (best[1] if best else [unit * min(per_dir)] * 4))


def draw(rng):
    kind = rng.choice(["stencil", "stencil", "project", "project", "coarse", "cycle", "cycle", "solve", "grads"])
    eps = rng.choice([0.15, 0.2])
    sigma = round(rng.uniform(0.0, 0.03), 4)
    if kind == "stencil":
        nrhs = rng.choice([1, 1, 1, 2, 3, 5, 8, 12])
        prec = rng.choice(["f32", "f32", "f64"])
        # odd extents too: any extent >= 2 is taken
        dims = _dims(rng, 2097152 // nrhs, 1, [3, 4, 5, 6, 7, 8, 9, 12, 16, 20, 24, 32, 48])
        # the parameters are checked against even block counts, so odd lattices run with the library's defaults
        odd = any(int(x) % 2 for x in dims.split("x"))
        return dict(kind=kind, dims=dims, prec=prec, op=rng.choice(["Q", "D"]), nrhs=nrhs, eps=eps,
                    m0=0.0 if odd else -0.02, csw=1.0 if odd else 1.9, bct=1 if odd else rng.choice([1, -1]),
                    sigma=sigma)
    if kind == "project":
        prec = rng.choice(["f32", "f64"])
        k = rng.randint(1, 32)
        n = _log_int(rng, 3000, 25165824 if k <= 8 else 3000000)
        return dict(kind=kind, n=n, k=k, prec=prec, mixed=rng.random() < 0.75)
    if kind == "coarse":
        agg = rng.choice(["4x4x4x4", "4x4x4x4", "2x2x2x2"])
        vmax = 524288 if agg == "4x4x4x4" else 16384
        return dict(kind=kind, dims=_dims(rng, vmax, 8, [1, 1, 2, 3, 4]), agg=agg, sap="4x4x4x4",
                    ntv=rng.choice([8, 12, 20, 20, 24]), links=rng.choice(["level", "bf16", "f16"]),
                    nrhs=rng.randint(1, 16), eps=eps, m0=-0.02, csw=1.9, sigma=sigma)
    if kind == "cycle":
        mixed = rng.random() < 0.75
        return dict(kind=kind, dims=_dims(rng, 131072 if mixed else 32768, 8, [1, 1, 2, 3]), agg="4x4x4x4",
                    sap=rng.choice(["4x4x4x4", "4x4x4x4", "2x2x2x2"]), ntv=rng.choice([8, 16, 20]), mixed=mixed,
                    links="level" if not mixed else rng.choice(["level", "level", "bf16"]), eps=0.2, m0=0.0172,
                    csw=1.9, sigma=sigma)
    if kind == "solve":
        mixed = rng.random() < 0.75
        return dict(kind=kind, dims=_dims(rng, 65536 if mixed else 8192, 8, [1, 1, 2]), agg="4x4x4x4", sap="4x4x4x4",
                    ntv=rng.choice([12, 20]), mixed=mixed, links="level", eps=0.2, m0=0.0172, csw=1.9, sigma=sigma,
                    tol=1e-12)
    return dict(kind=kind, dims=_dims(rng, 32768, 4, [1, 2, 2, 3, 4]), batch=rng.randint(1, 4))


# ---------------------------------------------------------------------------
# inputs


def _four(text):
    return tuple(int(x) for x in text.split("x"))


def _volume(case):
    lx, ly, lz, lt = _four(case["dims"])
    return lx * ly * lz * lt


def _gen(seed, stream):
    return torch.Generator("cuda").manual_seed(int(seed) * 16 + stream)


def _randn(shape, seed, stream, dtype):
    return torch.randn(shape, generator=_gen(seed, stream), device="cuda", dtype=dtype)


def _mm(a, b):
    """Products of 3x3 matrices in the last two axes."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _gauge(dims, eps, seed):
    """SU(3) links exp(i eps H), H = sum_a h_a lambda_a / 2 with Gaussian h: [t][z][y][x][mu][3][3]."""
    lx, ly, lz, lt = dims
    lam = torch.zeros(8, 3, 3, dtype=torch.complex128)
    for a, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        lam[2 * a, i, j] = lam[2 * a, j, i] = 1
        lam[2 * a + 1, i, j], lam[2 * a + 1, j, i] = -1j, 1j
    lam[6, 0, 0], lam[6, 1, 1] = 1, -1
    lam[7, 0, 0] = lam[7, 1, 1] = 1 / math.sqrt(3)
    lam[7, 2, 2] = -2 / math.sqrt(3)
    n = lx * ly * lz * lt * 4
    h = _randn((n, 8), seed, 1, torch.float64)
    x = (h.to(torch.complex128) @ (0.5j * eps * lam).reshape(8, 9).cuda()).reshape(n, 3, 3)
    one = torch.eye(3, dtype=torch.complex128, device="cuda")
    u = one + x / 12
    for k in range(11, 0, -1):
        u = one + _mm(x, u) / k
    # back onto SU(3) to the last bit: two orthonormal rows and their conjugate cross product
    r0 = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=1, keepdim=True)
    r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=1).conj()
    return torch.stack([r0, r1, r2], 1).reshape(lt, lz, ly, lx, 4, 3, 3).contiguous()


def _spinors(case, seed, nrhs, dtype):
    """nrhs Gaussian fields in the library's device layout: FP64 [12][V], FP32 [6][V][2]."""
    shape = (nrhs, 12, _volume(case)) if dtype == torch.complex128 else (nrhs, 6, _volume(case), 2)
    return _randn(shape, seed, 2, dtype)


def _project_inputs(case, seed):
    n, k = case["n"], case["k"]
    dt = torch.complex128 if case["prec"] == "f64" else torch.complex64
    X = _randn((k, n + n % 2), seed, 3, dt)[:, :n] / math.sqrt(n)   # rows start on 16-byte boundaries
    c = _randn((k,), seed, 4, dt)
    y = _randn((n,), seed, 5, dt) / math.sqrt(n)
    for j in range(k):
        y += c[j] * X[j]
    return X, y


def _coarse_vectors(case, seed):
    nc = 1
    for d, a in zip(_four(case["dims"]), _four(case["agg"])):
        nc *= d // a
    return _randn((case["nrhs"], nc, 2 * case["ntv"]), seed, 6, torch.complex64)


def _z2(case, seed):
    lx, ly, lz, lt = _four(case["dims"])
    r = torch.randint(0, 2, (lt, lz, ly, lx, 4, 3, 2), generator=_gen(seed, 7), device="cuda")
    return torch.view_as_complex((2.0 * r.double() - 1) / math.sqrt(2.0))


def _net_inputs(case, seed):
    lx, ly, lz, lt = _four(case["dims"])
    x = _randn((case["batch"], lt, lz, ly, lx, 24), seed, 8, torch.float64)
    t = 0.3 * _randn(x.shape, seed, 9, torch.float64)
    W = torch.zeros(3, 81, 32, 32, dtype=torch.float32, device="cuda")
    for l, (ci, co) in enumerate(((24, 32), (32, 32), (32, 24))):
        W[l, :, :co, :ci] = 0.5 * math.sqrt(2 / (81 * ci)) * _randn((81, co, ci), seed, 10 + l, torch.float32)
    return x, t, W


def _context(case, seed, params):
    ctx = Context(_four(case["dims"]))
    if params is not None:
        ctx.set_params(**params)
    if "eps" in case:
        U = _gauge(_four(case["dims"]), case["eps"], seed)
        torch.cuda.synchronize()
        ctx.load_gauge_dev(U.data_ptr())
        return ctx, U
    return ctx, None


def _mg_params(case, **kw):
    return dict(m0=case["m0"], csw=case["csw"], agg=_four(case["agg"]), sap_block=_four(case["sap"]), n_tv=case["ntv"],
                precision=MIXED if case.get("mixed", True) else FP64, coarse_links=LINKS[case.get("links", "level")], **kw)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "stencil":
        odd = any(x % 2 for x in _four(case["dims"]))
        half = tuple(x // 2 for x in _four(case["dims"]))
        # a program that only applies the operator keeps no multigrid work space (few test vectors, no restart)
        small = tuple(next(b for b in (4, 3, 2, 1) if h % b == 0) for h in half)
        p = None if odd else dict(m0=case["m0"], csw=case["csw"], bc=(1, 1, 1, case["bct"]), agg=small,
                                  sap_block=small, n_tv=2, outer_restart=1)
        st["ctx"], U = _context(case, seed, p)
        st["x"] = _spinors(case, seed, case["nrhs"], torch.complex128 if case["prec"] == "f64" else torch.complex64)
        st["y"] = torch.empty_like(st["x"])
    elif kind == "project":
        st["ctx"] = Context((8, 8, 8, 8))
        st["ctx"].set_params(n_tv=2, outer_restart=1, precision=MIXED if case["mixed"] else FP64)
        st["X"], st["y0"] = _project_inputs(case, seed)
        st["y"] = torch.empty_like(st["y0"])
        st["ptrs"] = [x.data_ptr() for x in st["X"]]
        st["stream"] = torch.cuda.ExternalStream(st["ctx"].stream())
    elif kind == "coarse":
        st["ctx"], U = _context(case, seed, _mg_params(case, setup_smooth=1, setup_iters=0, sap_mr_iters=1,
                                                       outer_restart=1))
        st["ctx"].setup(seed)
        st["x"] = _coarse_vectors(case, seed)
        st["y"] = torch.empty_like(st["x"])
    elif kind == "cycle":
        st["ctx"], U = _context(case, seed, _mg_params(case, setup_iters=2))
        st["ctx"].setup(seed)
        st["x"] = _spinors(case, seed, 1, torch.complex64 if case["mixed"] else torch.complex128)
        st["y"] = torch.empty_like(st["x"])
    elif kind == "solve":
        st["ctx"], U = _context(case, seed, _mg_params(case, setup_iters=4, outer_maxiter=200))
        st["ctx"].setup(seed)
        st["b"] = _z2(case, seed).cpu().numpy()
    elif kind == "grads":
        x, t, W = _net_inputs(case, seed)
        st["ctx"] = Context(_four(case["dims"]))
        st["ctx"].net_set_weights(W.cpu().numpy())
        st["x"], st["t"] = x.cpu().numpy(), t.cpu().numpy()
    else:
        st["ctx"], st["U"] = _context(case, seed, _mg_params(case))
        st["seed"] = seed
    torch.cuda.synchronize()
    return st


def run(st):
    case, ctx, kind = st["case"], st["ctx"], st["case"]["kind"]
    if kind == "stencil":
        op = OP_Q if case["op"] == "Q" else OP_D
        prec = PREC_F64 if case["prec"] == "f64" else PREC_F32
        if case["nrhs"] == 1:
            ctx.apply_dev(st["x"].data_ptr(), st["y"].data_ptr(), case["sigma"], op, prec)
        else:
            ctx.apply_dev_nrhs(st["x"].data_ptr(), st["y"].data_ptr(), case["nrhs"], case["sigma"], op, prec)
        return st["y"]
    if kind == "project":
        prec = PREC_F64 if case["prec"] == "f64" else PREC_F32
        with torch.cuda.stream(st["stream"]):
            st["y"].copy_(st["y0"])   # the new vector, on the library's stream
        d = ctx.multidot_dev(st["ptrs"], st["y"].data_ptr(), case["n"], prec)
        ctx.multi_axpy_dev(st["ptrs"], -d, st["y"].data_ptr(), case["n"], prec)
        # FP32 vectors: the coefficients come from FP32 products and sums
        return [d if case["prec"] == "f64" else d.astype(np.complex64), st["y"]]
    if kind == "coarse":
        ctx.coarse_apply_dev_nrhs(st["x"].data_ptr(), st["y"].data_ptr(), case["nrhs"], case["sigma"])
        return st["y"]
    if kind == "cycle":
        ctx.mg_cycle_dev_noalloc(st["x"].data_ptr(), st["y"].data_ptr(), case["sigma"])
        return st["y"]
    if kind == "solve":
        return ctx.solve(st["b"], case["sigma"], case["tol"])[0]
    if kind == "grads":
        loss, G = ctx.net_loss_grads(st["x"], st["t"])
        return [np.float32(loss), G]   # the loss of an FP32 forward pass
    ctx.load_gauge_dev(st["U"].data_ptr())
    ctx.setup(st["seed"])
    return ctx.eigensolve(case["neig"], case["tol"], want_vectors=False)[0]


def work(case):
    kind = case["kind"]
    if kind == "project":
        n, k, b = case["n"], case["k"], 16 if case["prec"] == "f64" else 8
        return dict(bytes=float((k + 2) * n * b), flops=16.0 * k * n)
    V = _volume(case)
    if kind == "stencil":
        # x and y; links (two rows in FP32, full in FP64) and clover once for all fields
        per = case["nrhs"] * 384 + 1152 if case["prec"] == "f64" else case["nrhs"] * 192 + 480
        return dict(bytes=float(per * V), flops=1872.0 * V * case["nrhs"])
    if kind == "grads":
        flops = 2.0 * 81 * V * case["batch"] * ((24 * 32 + 32 * 32 + 32 * 24) * 2 + 32 * 32 + 32 * 24)
        return dict(bytes=V * case["batch"] * 48.0 * 8 + 2 * 3 * 81 * 1024 * 4.0, flops=flops)
    nc = V
    for a in _four(case["agg"]):
        nc //= a
    n2 = 2 * case["ntv"]
    if kind == "coarse":
        link = 8 if case["links"] == "level" else 4
        return dict(bytes=9.0 * nc * n2 * n2 * link + 16.0 * case["nrhs"] * nc * n2,
                    flops=8.0 * 9 * nc * n2 * n2 * case["nrhs"])
    # one two-grid cycle: P twice, the coarse operator once per step of a solve of 8 steps, 3 SAP cycles of
    # one residual and 4 minimal-residual steps; r, z, P, coarse operator, links and clover from memory once
    w = 4 if case["mixed"] else 8
    cyc_b = V * w * (24.0 * (case["ntv"] + 2) + 48 + 72) + 9.0 * nc * n2 * n2 * 2 * w
    cyc_f = 2 * 8.0 * 12 * V * case["ntv"] + 8 * 72.0 * nc * n2 * n2 + 3 * 5 * 1872.0 * V
    if kind == "cycle":
        return dict(bytes=cyc_b, flops=cyc_f)
    steps = 12 if kind == "solve" else 8 * (10 + 2 * case["neig"])   # outer steps a solve or an eigensolve takes at least
    return dict(bytes=cyc_b + V * 16.0 * (36 + 36 + 24), flops=steps * (cyc_f + 1872.0 * V))


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch

_AXIS = (-3, -4, -5, -6)   # x, y, z, t of a spinor [...][t][z][y][x][spin][colour]


def _gammas():
    s = [torch.tensor(m, dtype=torch.complex128) for m in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
    out = []
    for k in range(4):
        b = 1j * s[k] if k < 3 else torch.eye(2, dtype=torch.complex128)
        g = torch.zeros(4, 4, dtype=torch.complex128)
        g[:2, 2:], g[2:, :2] = b, b.conj().T
        out.append(g.cuda())
    return out


class _Wilson:
    """D = (4 + m0) - hops + clover of spinors [...][t][z][y][x][4][3], with an optional block grid for SAP."""

    def __init__(self, U, m0, csw, bct):
        self.g = _gammas()
        self.g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device="cuda")[:, None]
        self.U = [U[..., mu, :, :].contiguous() for mu in range(4)]
        self.m0, self.bct = m0, bct
        lt, lz, ly, lx = U.shape[:4]
        ext = (lx, ly, lz, lt)
        self.coord = [torch.arange(ext[mu], device="cuda").reshape([-1 if a == _AXIS[mu] else 1 for a in (-6, -5, -4, -3)] +
                                                                  [1, 1]) for mu in range(4)]
        self.ext = ext
        self.C = self._clover(csw)   # [t][z][y][x][chirality][6][6]

    def _up(self, f, mu, n=1):
        """f(x + n mu) of a matrix field [t][z][y][x][3][3]"""
        return torch.roll(f, -n, 3 - mu)

    def _clover(self, csw):
        U, C = self.U, None
        for mu in range(4):
            for nu in range(mu + 1, 4):
                um, un = U[mu], U[nu]
                umn, unm = self._up(um, nu), self._up(un, mu)             # U_mu(x + nu), U_nu(x + mu)
                q = _mm(_mm(um, unm), _mm(_dag(umn), _dag(un)))
                f = _dag(self._up(umn, mu, -1))                           # U_mu(x - mu + nu)^dag
                unb, umb = self._up(un, mu, -1), self._up(um, mu, -1)     # at x - mu
                q = q + _mm(_mm(un, f), _mm(_dag(unb), umb))
                unbb, umbb = self._up(unb, nu, -1), self._up(umb, nu, -1)  # at x - mu - nu
                und, umd = self._up(un, nu, -1), self._up(um, nu, -1)     # at x - nu
                q = q + _mm(_mm(_dag(umb), _dag(unbb)), _mm(umbb, und))
                q = q + _mm(_mm(_dag(und), umd), _mm(self._up(und, mu), _dag(um)))
                F = (q - _dag(q)) / 8
                sg = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                for ch in range(2):
                    s = 0.5j * csw * sg[2 * ch:2 * ch + 2, 2 * ch:2 * ch + 2]
                    t = (s[:, None, :, None] * F[..., None, :, None, :]).reshape(F.shape[:-2] + (6, 6))
                    if C is None:
                        C = torch.zeros(F.shape[:-2] + (2, 6, 6), dtype=torch.complex128, device="cuda")
                    C[..., ch, :, :] += t
        return C

    def D(self, psi, block=None):
        """D psi; with block extents only the hops that stay inside a block."""
        lead = psi.shape[:-2]
        out = (4 + self.m0) * psi + (self.C @ psi.reshape(lead + (2, 6, 1))).reshape(psi.shape)
        one = torch.eye(4, dtype=torch.complex128, device="cuda")
        for mu in range(4):
            L, c, u = self.ext[mu], self.coord[mu], self.U[mu]
            edge = float(self.bct) if mu == 3 else 1.0
            up = torch.where(c == L - 1, edge, 1.0).to(torch.float64)
            dn = torch.where(c == 0, edge, 1.0).to(torch.float64)
            if block is not None:
                up = torch.where(c % block[mu] == block[mu] - 1, 0.0, up)
                dn = torch.where(c % block[mu] == 0, 0.0, dn)
            f = torch.roll(psi, -1, _AXIS[mu]) @ u.transpose(-1, -2)
            out -= 0.5 * up * torch.einsum("ij,...jc->...ic", one - self.g[mu], f)
            b = torch.roll(psi @ u.conj(), 1, _AXIS[mu])
            out -= 0.5 * dn * torch.einsum("ij,...jc->...ic", one + self.g[mu], b)
        return out

    def Q(self, psi, sigma):
        return self.g5 * self.D(psi) - sigma * psi

    def Dsigma(self, psi, sigma):
        return self.D(psi) - sigma * self.g5 * psi


def _from_layout(x, dims):
    """One field of the library's layout -> [t][z][y][x][4][3] in complex128."""
    lx, ly, lz, lt = dims
    if x.dim() == 3:   # [6][V][2]
        x = x.permute(0, 2, 1).reshape(12, -1)
    return x.to(torch.complex128).reshape(4, 3, lt, lz, ly, lx).permute(2, 3, 4, 5, 0, 1)


def _to_layout(y, f32):
    y = y.permute(4, 5, 0, 1, 2, 3).reshape(12, -1)
    return y.reshape(6, 2, -1).permute(0, 2, 1).contiguous() if f32 else y.contiguous()


def _philox_uniform(V, j, seed, tag):
    """Components [V][12] of vector j of the setup: int32 words of Philox4x32-10 blocks (site, pair, j, tag) / 2^31."""
    m = 0xFFFFFFFF
    s = torch.arange(V, device="cuda", dtype=torch.int64)[:, None].expand(V, 6)
    q = torch.arange(6, device="cuda", dtype=torch.int64)[None, :].expand(V, 6)
    c = [s, q, torch.full_like(s, j), torch.full_like(s, tag)]
    k0, k1 = seed & m, (seed >> 32) & m

    def mul(a, b):   # 32 x 32 -> (high, low) words, by 16-bit halves
        ah, al = a >> 16, a & 0xFFFF
        lo = al * b
        hi = ah * b + (lo >> 16)
        return (hi >> 16) & m, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    w = [torch.where(x >= 2 ** 31, x - 2 ** 32, x).double() * 2.0 ** -31 for x in c]
    return torch.stack([torch.complex(w[0], w[1]), torch.complex(w[2], w[3])], 2).reshape(V, 12)


def _exact_coarse(case, seed):
    """(Q_c - sigma) x = P^dag (Q - sigma) P x with P from the setup's vectors: one SAP cycle of one
    minimal-residual step on Philox uniforms, orthonormalised per aggregate and chirality."""
    dims, blk, agg, ntv = _four(case["dims"]), _four(case["sap"]), _four(case["agg"]), case["ntv"]
    lx, ly, lz, lt = dims
    op = _Wilson(_gauge(dims, case["eps"], seed), case["m0"], case["csw"], 1)
    par = sum((op.coord[mu] // blk[mu]) for mu in range(4)) % 2

    def split(f, b):   # [t][z][y][x][4][3] -> [block][chirality][site in block][6], blocks with x fastest
        f = f.reshape(lt // b[3], b[3], lz // b[2], b[2], ly // b[1], b[1], lx // b[0], b[0], 2, 6)
        return f.permute(0, 2, 4, 6, 8, 1, 3, 5, 7, 9).reshape(-1, 2, b[0] * b[1] * b[2] * b[3] * 6)

    def join(f, b):
        f = f.reshape(lt // b[3], lz // b[2], ly // b[1], lx // b[0], 2, b[3], b[2], b[1], b[0], 6)
        return f.permute(0, 5, 1, 6, 2, 7, 3, 8, 4, 9).reshape(lt, lz, ly, lx, 4, 3)

    A = None
    for j in range(ntv):
        w = _philox_uniform(op.C.shape[0] * lz * ly * lx, j, int(seed), 0x5EED0001).to(torch.complex64).to(torch.complex128)
        rhs, z = op.g5 * w.reshape(lt, lz, ly, lx, 4, 3), torch.zeros(lt, lz, ly, lx, 4, 3, dtype=torch.complex128,
                                                                       device="cuda")
        for colour in range(2):
            rho = (rhs - op.D(z)) * (par == colour)
            q = op.D(rho, blk)
            qb, rb = split(q, blk).flatten(1), split(rho, blk).flatten(1)
            qq = (qb.abs() ** 2).sum(1, keepdim=True)
            alpha = torch.where(qq > 0, (qb.conj() * rb).sum(1, keepdim=True) / qq.clamp_min(1e-300), 0)
            z = z + join((alpha * rb).reshape(rb.shape[0], 2, -1), blk)
        a = split(z, agg)
        if A is None:
            A = torch.empty(a.shape + (ntv,), dtype=torch.complex128, device="cuda")
        A[..., j] = a
    for _ in range(2):   # Gram-Schmidt through the Cholesky factor, twice
        Lc = torch.linalg.cholesky(A.mH @ A)
        A = A @ torch.linalg.inv(Lc.mH)
    x = _coarse_vectors(case, seed).to(torch.complex128)
    out = torch.empty_like(x)
    for r in range(case["nrhs"]):
        v = join((A @ x[r].reshape(-1, 2, ntv, 1))[..., 0], agg)
        v = split(op.Q(v, case["sigma"]), agg)
        out[r] = (A.mH @ v[..., None])[..., 0].reshape(-1, 2 * ntv)
    return out


def _exact_solve(case, seed):
    op = _Wilson(_gauge(_four(case["dims"]), case["eps"], seed), case["m0"], case["csw"], 1)
    b = _z2(case, seed)
    x = torch.zeros_like(b)
    for _ in range(2):   # conjugate gradients on (Q - sigma)^2 and one refinement
        r = op.Q(b - op.Q(x, case["sigma"]), case["sigma"])
        p, d = r.clone(), torch.zeros_like(r)
        rr = torch.linalg.vector_norm(r) ** 2
        stop, its = float(rr) * 1e-24, 0
        while its < 4000 and (its % 20 or float(rr) > stop):
            q = op.Q(op.Q(p, case["sigma"]), case["sigma"])
            al = rr / (p.conj() * q).sum().real
            d, r = d + al * p, r - al * q
            new = torch.linalg.vector_norm(r) ** 2
            p, rr, its = r + (new / rr) * p, new, its + 1
        x = x + d
    return x


def _exact_grads(case, seed):
    x, t, W = _net_inputs(case, seed)
    W = [W[l, :, :co, :ci].double().requires_grad_() for l, (ci, co) in enumerate(((24, 32), (32, 32), (32, 24)))]

    def conv(f, w):
        out = 0
        for tap in range(81):
            d = (tap % 3 - 1, (tap // 3) % 3 - 1, (tap // 9) % 3 - 1, tap // 27 - 1)
            out = out + torch.roll(f, [-v for v in d], (4, 3, 2, 1)) @ w[tap].T
        return out

    y = conv(torch.nn.functional.gelu(conv(torch.nn.functional.gelu(conv(x, W[0]), approximate="tanh"), W[1]),
                                      approximate="tanh"), W[2])
    loss = 0.5 * ((y - t) ** 2).sum() / case["batch"]
    G = torch.zeros(3, 81, 32, 32, dtype=torch.float64, device="cuda")
    for l, g in enumerate(torch.autograd.grad(loss, W)):
        G[l, :, :g.shape[1], :g.shape[2]] = g
    return [loss.detach(), G]


def _exact_eig(case, seed):
    dims = _four(case["dims"])
    op = _Wilson(_gauge(dims, case["eps"], seed), case["m0"], case["csw"], 1)
    n = 12 * _volume(case)
    lx, ly, lz, lt = dims
    M = op.Q(torch.eye(n, dtype=torch.complex128, device="cuda").reshape(n, lt, lz, ly, lx, 4, 3), 0.0).reshape(n, n).T
    w = torch.linalg.eigvalsh(M).cpu().numpy()
    w = w[np.argsort(np.abs(w), kind="stable")][:case["neig"]]
    return w


def exact(case, seed):
    kind = case["kind"]
    if kind == "stencil":
        dims, f32 = _four(case["dims"]), case["prec"] == "f32"
        op = _Wilson(_gauge(dims, case["eps"], seed), case["m0"], case["csw"], case["bct"])
        x = _spinors(case, seed, case["nrhs"], torch.complex64 if f32 else torch.complex128)
        y = torch.empty(x.shape, dtype=torch.complex128, device="cuda")
        for r in range(case["nrhs"]):
            v = _from_layout(x[r], dims)
            y[r] = _to_layout(op.Q(v, case["sigma"]) if case["op"] == "Q" else op.Dsigma(v, case["sigma"]), f32)
        return y
    if kind == "project":
        X, y = _project_inputs(case, seed)
        y = y.to(torch.complex128)
        d = torch.stack([(x.to(torch.complex128).conj() * y).sum() for x in X])
        for j in range(case["k"]):
            y = y - d[j] * X[j].to(torch.complex128)
        return [d, y]
    if kind == "coarse":
        return _exact_coarse(case, seed)
    if kind == "solve":
        return _exact_solve(case, seed)
    if kind == "grads":
        return _exact_grads(case, seed)
    if kind == "eig":
        return _exact_eig(case, seed)
    return None   # a two-grid cycle is a truncated iteration: its output has no value apart from the method's own steps
