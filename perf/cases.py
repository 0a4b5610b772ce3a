"""The framework's work as measurable cases: the calls that a program solving the clover Wilson-Dirac equation makes.

Kinds of case
  solve      X = D_W^-1 B for a block of right-hand sides, in FP64 (the paper's methods) or in mixed precision on the
             even-odd system (the benchmark's configuration), as one or several block systems
  grad       a differentiable solve, forward and backward (gradients of B, kappa and the gauge field)
  op         one multi-RHS operator application: device-layout blocks in FP32 / FP16 storage (a solver's inner call),
             canonical blocks in FP64 (a user's own call)
  project    block algebra on device-layout blocks: Y = B - A (A^H B)
  setup      a new gauge configuration: upload, clover term, first operator application

Every input is made on the GPU from the seed alone.  Links are random SU(3), U = exp(i eps H); sources are the twelve
point sources or Z4 noise; operator inputs are complex Gaussian, as the iterates of a solve are.
"""
import math

import torch

EPS, CSW = 0.5, 1.0  # link spread and clover coefficient of the repository's benchmark and tests

C128, C64, F64, F32 = torch.complex128, torch.complex64, torch.float64, torch.float32
DEV = "cuda"


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # smallest call: the paper's block BiCGGR in FP64 on 4^4, one block of the 12 point sources (one propagator)
        dict(name="solve_fp64_4x4x4x4_L12", kind="solve", dims="4,4,4,4", L=12, source="point", split=12,
             kappas="0.12", method="bicggr", prec="fp64", eo=False),
        # a small lattice in mixed precision: launches and readbacks against little work
        dict(name="solve_mixed_8x8x8x16_L12", kind="solve", dims="8,8,8,16", L=12, source="point", split=6,
             kappas="0.125", method="bicgstab", prec="fp32", eo=True),
        # the paper's own experiment, 12 point sources in one FP64 block, on a lattice between its size and the tests'
        dict(name="solve_fp64_12x12x12x24_L12", kind="solve", dims="12,12,12,24", L=12, source="point", split=12,
             kappas="0.125", method="bicggr", prec="fp64", eo=False),
        # many noise sources at three quark masses, batched (uneven block systems of 6 and 2 columns)
        dict(name="solve_mixed_16x16x16x32_L60", kind="solve", dims="16,16,16,32", L=60, source="z4", split=6,
             kappas="0.12,0.125,0.13", method="bicgstab", prec="fp32", eo=True),
        # the largest lattice of the benchmark
        dict(name="solve_mixed_24x24x24x48_L28", kind="solve", dims="24,24,24,48", L=28, source="z4", split=6,
             kappas="0.12,0.124", method="bicgstab", prec="fp32", eo=True),
        # forward and backward through a solve: the noise estimate Re <B, D^-1 B> of the propagator's trace, with its
        # gradients in the sources (through X), kappa and every link
        dict(name="grad_8x8x8x16_L12", kind="grad", dims="8,8,8,16", L=12, kappa=0.125),
        # the operator inside a solver: the operator benchmark's default, and the largest block
        dict(name="op_fp32_16x16x16x32_L30", kind="op", dims="16,16,16,32", L=30, prec="fp32", kappa=0.125),
        dict(name="op_fp32_24x24x24x48_L96", kind="op", dims="24,24,24,48", L=96, prec="fp32", kappa=0.13),
        # half-precision storage, odd column count, extents that are no power of two
        dict(name="op_fp16_12x10x14x18_L13", kind="op", dims="12,10,14,18", L=13, prec="fp16", kappa=0.122),
        # a user's own application in FP64 on canonical blocks (a residual check)
        dict(name="op_fp64_16x16x16x32_L12", kind="op", dims="16,16,16,32", L=12, prec="fp64", kappa=0.125),
        # a wide block projected against another one
        dict(name="project_fp32_16x16x16x32_L48", kind="project", dims="16,16,16,32", L=48, prec="fp32"),
        # a new configuration of the paper's size
        dict(name="setup_16x16x16x32", kind="setup", dims="16,16,16,32", kappa=0.125),
    ]


def _dims_of(rng, lo, hi, even=False):
    """Four extents of 3 to 48 whose product lies in [lo, hi], spread over its logarithm (even: all of them even)."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = v ** 0.25
        d = [max(3, min(24, round(side * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(3)]
        if even:
            d = [x + (x & 1) for x in d]
        d.append(max(4, min(48, round(v / math.prod(d)))))
        if even:
            d[3] += d[3] & 1
        if lo <= math.prod(d) <= hi:
            return d


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "grad", "op", "op", "op", "project", "setup"])
    text = lambda d: ",".join(map(str, d))  # noqa: E731
    if kind == "solve" and rng.random() < 0.35:
        d = _dims_of(rng, 256, 41000)
        L = rng.randint(1, 12)
        return dict(kind="solve", dims=text(d), L=L, source="z4", split=12, kappas="%.4f" % rng.uniform(0.118, 0.128),
                    method=rng.choice(["bicggr", "bicgstab"]), prec="fp64", eo=False)
    if kind == "solve":
        eo = rng.random() < 0.8  # the even-odd form wants even extents
        d = _dims_of(rng, 256, 131072, even=eo)
        L = max(2, round(math.exp(rng.uniform(math.log(2), math.log(60)))))
        n = rng.randint(1, min(3, max(1, L // 2)))
        ks = ",".join("%.4f" % k for k in sorted(rng.uniform(0.118, 0.13) for _ in range(n)))
        return dict(kind="solve", dims=text(d), L=L, source="z4", split=rng.choice([4, 5, 6, 6, 6]), kappas=ks,
                    method="bicgstab", prec="fp32", eo=eo)
    if kind == "grad":
        return dict(kind="grad", dims=text(_dims_of(rng, 256, 8192)), L=rng.randint(1, 12),
                    kappa=round(rng.uniform(0.118, 0.128), 4))
    if kind == "op":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp16", "fp64"])
        d = _dims_of(rng, 256, 663552 if prec != "fp64" else 131072)
        cap = min(96 if prec != "fp64" else 24, (663552 * 60 if prec != "fp64" else 131072 * 24) // math.prod(d))
        L = max(1, round(math.exp(rng.uniform(0.0, math.log(max(1, cap))))))
        return dict(kind="op", dims=text(d), L=L, prec=prec, kappa=round(rng.uniform(0.118, 0.13), 4))
    if kind == "project":
        d = _dims_of(rng, 256, 131072)
        prec = rng.choice(["fp32", "fp32", "fp64"])
        L = max(1, round(math.exp(rng.uniform(0.0, math.log(60 if prec == "fp32" else 16)))))
        return dict(kind="project", dims=text(d), L=L, prec=prec)
    return dict(kind="setup", dims=text(_dims_of(rng, 256, 500000)), kappa=round(rng.uniform(0.118, 0.13), 4))


def _dims(case):
    return tuple(int(x) for x in case["dims"].split(","))


def _systems(case):
    """Block systems of a solve: the columns go to the kappas as evenly as they can, each kappa's in systems of at
    most `split` columns."""
    ks = [float(k) for k in case["kappas"].split(",")]
    n, kappas, Ls = len(ks), [], []
    for i, k in enumerate(ks):
        left = case["L"] * (i + 1) // n - case["L"] * i // n
        while left > 0:
            Ls.append(min(case["split"], left))
            kappas.append(k)
            left -= Ls[-1]
    return kappas, Ls


# ------------------------------------------------------------------ inputs

def _gen(seed, k):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 16 + k) & 0x7FFFFFFFFFFF)
    return g


def _gell_mann():
    g = torch.zeros(8, 3, 3, dtype=C128)
    g[0][0, 1] = g[0][1, 0] = 1
    g[1][0, 1], g[1][1, 0] = -1j, 1j
    g[2][0, 0], g[2][1, 1] = 1, -1
    g[3][0, 2] = g[3][2, 0] = 1
    g[4][0, 2], g[4][2, 0] = -1j, 1j
    g[5][1, 2] = g[5][2, 1] = 1
    g[6][1, 2], g[6][2, 1] = -1j, 1j
    g[7][0, 0] = g[7][1, 1] = 1 / math.sqrt(3)
    g[7][2, 2] = -2 / math.sqrt(3)
    return g


def _links(dims, seed):
    """U[mu, t, z, y, x, 3, 3] = exp(i eps sum_a c_a lambda_a / 2), c_a ~ N(0, 1)."""
    shape = (4, dims[3], dims[2], dims[1], dims[0])
    c = torch.randn(shape + (8,), dtype=F64, device=DEV, generator=_gen(seed, 1))
    A = (c.to(C128) @ (1j * EPS / 2 / 8 * _gell_mann()).to(DEV).reshape(8, 9)).reshape(shape + (3, 3))
    one = torch.eye(3, dtype=C128, device=DEV)
    E = one + A / 11
    for k in range(10, 0, -1):  # exp(A / 8) by its series, then squared three times
        E = one + (A @ E) / k
    for _ in range(3):
        E = E @ E
    return E.contiguous()


def _block(dims, L):
    return (L, dims[3], dims[2], dims[1], dims[0], 4, 3)


def _point(dims):
    B = torch.zeros(_block(dims, 12), dtype=C128, device=DEV)
    for i in range(12):
        B[i, 0, 0, 0, 0, i // 3, i % 3] = 1
    return B


def _z4(dims, L, seed, k=2):
    n = torch.randint(0, 4, _block(dims, L), device=DEV, generator=_gen(seed, k), dtype=torch.int64)
    return torch.tensor([1, 1j, -1, -1j], dtype=C128, device=DEV)[n]


def _gauss(dims, L, seed, k, prec):
    """Complex Gaussian block whose values the storage precision holds."""
    out = torch.empty(_block(dims, L), dtype=C128, device=DEV)
    g = _gen(seed, k)
    for j in range(L):
        x = torch.randn(out.shape[1:] + (2,), dtype=F64, device=DEV, generator=g) * math.sqrt(0.5)
        if prec != "fp64":
            x = x.to(F32)
        if prec == "fp16":  # per site and column: FP16 values times the largest component
            s = x.abs().amax(dim=(-3, -2, -1), keepdim=True)
            x = (x * (1 / s)).to(torch.float16).to(F32) * s
        out[j] = torch.view_as_complex(x.to(F64).contiguous())
    return out


def _sources(case, seed):
    dims = _dims(case)
    return _point(dims) if case.get("source") == "point" else _z4(dims, case["L"], seed)


def _project_inputs(case, seed):
    """A (columns of unit norm) and B, which has parts inside and outside the span of A."""
    dims, L, prec = _dims(case), case["L"], case["prec"]
    A = _gauss(dims, L, seed, 3, prec) / 2.0 ** round(math.log2(math.sqrt(12 * math.prod(dims))))
    B = _gauss(dims, L, seed, 4, prec)
    M = torch.randn((L, L), dtype=C128, device=DEV, generator=_gen(seed, 5))
    B = B / 64 + (M @ A.reshape(L, -1)).reshape(A.shape)
    return A, (B.to(C64).to(C128) if prec == "fp32" else B)


# ------------------------------------------------------------------ what a program has in hand, and a pass

def _lattice(dims, seed):
    import paper_0903_4936_gb300 as bk
    lat = bk.Lattice(dims)
    lat.upload_gauge(_links(dims, seed))
    lat.build_clover(CSW)
    return lat


def prepare(case, seed):
    kind, dims = case["kind"], _dims(case)
    st = dict(case=case, kind=kind)
    if kind == "solve":
        st["kappas"], st["Ls"] = _systems(case)
        st["B"] = _sources(case, seed)
        st["lat"] = _lattice(dims, seed)
    elif kind == "grad":
        import paper_0903_4936_gb300 as bk
        st["lat"] = bk.Lattice(dims)
        st["U"] = _links(dims, seed).requires_grad_()
        st["B"] = _z4(dims, case["L"], seed).requires_grad_()
        st["kappa"] = torch.tensor(case["kappa"], dtype=F64, device=DEV, requires_grad=True)
        st["eta"] = st["B"].detach().clone()
    elif kind == "op":
        st["lat"] = _lattice(dims, seed)
        X = _gauss(dims, case["L"], seed, 3, case["prec"])
        if case["prec"] == "fp64":
            st["X"] = X
        else:
            st["X"] = st["lat"].pack(X, case["prec"])
            st["Y"] = torch.zeros_like(st["X"])
    elif kind == "project":
        import paper_0903_4936_gb300 as bk
        lat = st["lat"] = bk.Lattice(dims)
        A, B = _project_inputs(case, seed)
        st["A"], st["B"] = lat.pack(A, case["prec"]), lat.pack(B, case["prec"])
    else:
        import paper_0903_4936_gb300 as bk
        st["lat"] = bk.Lattice(dims)
        st["U"] = _links(dims, seed)
        st["X"] = _gauss(dims, 1, seed, 3, "fp64")
    return st


def _values(field, case, prec):
    """The numbers of a device-layout block: (values, FP16 scales)."""
    V, np = math.prod(_dims(case)), (case["L"] + 1) // 2
    n = V * 12 * np * {"fp64": 32, "fp32": 16, "fp16": 8}[prec]
    if prec == "fp16":
        return field[:n].view(torch.float16), field[n:n + 8 * V * np].view(F32)
    return field[:n].view(F64 if prec == "fp64" else F32)


def run(st):
    case, kind, lat = st["case"], st["kind"], st["lat"]
    if kind == "solve":
        opts = dict(method=case["method"], prec=case["prec"], tol=1e-12, maxiter=2000)
        if case["prec"] != "fp64":
            opts.update(delta=0.003, anchor=1e-4, eo=case["eo"])
        if len(st["Ls"]) == 1:
            X, _ = lat.block_solve(st["B"], st["kappas"][0], **opts)
        else:
            X, _ = lat.block_solve_batched(st["B"], st["kappas"], st["Ls"], **opts)
        return X
    if kind == "grad":
        import paper_0903_4936_gb300 as bk
        X = bk.block_solve_autograd(lat, st["B"], st["kappa"], st["U"], CSW)
        return (X.detach(),) + torch.autograd.grad(X, (st["B"], st["kappa"], st["U"]), st["eta"])
    if kind == "op":
        if case["prec"] == "fp64":
            return lat.dslash(st["X"], case["kappa"], "fp64")
        lat.dslash_dev(st["X"], case["L"], case["kappa"], case["prec"], out=st["Y"])
        return _values(st["Y"], case, case["prec"])
    if kind == "project":
        G = lat.gram(st["A"], st["B"], case["L"], case["prec"])
        Y = lat.xmy(st["A"], G, case["L"], c=-1.0, Z=st["B"], prec=case["prec"])
        return _values(Y, case, case["prec"])
    lat.upload_gauge(st["U"])
    lat.build_clover(CSW)
    return lat.dslash(st["X"], case["kappa"], "fp64")


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """A solve: links and sources in, solution out, and the operator applied twice in each of at least 20 iterations
    (1872 flops per site and column); the iterates themselves could stay on the chip.  One operator application: links
    (72 reals) and site term (72 reals) once per site, each column in and out once."""
    kind, V, L = case["kind"], math.prod(_dims(case)), case.get("L", 1)
    links, cols = V * 72 * 8, V * L * 24 * 8
    if kind == "solve":
        return dict(bytes=links + 2 * cols, flops=1872.0 * V * L * 40)
    if kind == "grad":
        return dict(bytes=2 * links + 4 * cols, flops=1872.0 * V * L * 80)
    if kind == "op":
        size = {"fp64": 8, "fp32": 4, "fp16": 2}[case["prec"]]
        extra = V * L * 8 if case["prec"] == "fp16" else 0
        return dict(bytes=V * 144 * max(4, size) + 2 * V * L * 24 * size + extra, flops=1872.0 * V * L)
    if kind == "project":
        size = 8 if case["prec"] == "fp64" else 4
        return dict(bytes=3 * V * L * 24 * size, flops=2.0 * 8 * 12 * V * L * L)
    # clover: 6 planes x 4 leaves x 3 products of 3 x 3 matrices (198 flops each)
    return dict(bytes=links + 2 * cols, flops=V * (72 * 198 + 1872.0))


# ------------------------------------------------------------------ the same in 64 bits, plain torch
#
# Blocks here are [V, 3 colours, 4 spins, L]; a gamma matrix permutes the spins with a phase.

GAMMA = [([3, 2, 1, 0], [-1j, -1j, 1j, 1j]), ([3, 2, 1, 0], [-1, 1, 1, -1]),
         ([2, 3, 0, 1], [-1j, 1j, 1j, -1j]), ([0, 1, 2, 3], [1, 1, -1, -1])]


def _gamma(mu):
    m = torch.zeros(4, 4, dtype=C128)
    for a, (p, f) in enumerate(zip(*GAMMA[mu])):
        m[a, p] = f
    return m


def _times_gamma(mu, q):
    p, f = GAMMA[mu]
    return q[:, :, p] * torch.tensor(f, dtype=C128, device=q.device).reshape(1, 1, 4, 1)


def _dag(m):
    return m.conj().transpose(-1, -2)


class _Plain:
    def __init__(self, dims, U):
        self.V = math.prod(dims)
        n = torch.arange(self.V, device=DEV).reshape(dims[3], dims[2], dims[1], dims[0])
        self.up = [torch.roll(n, -1, 3 - mu).reshape(-1) for mu in range(4)]
        self.dn = [torch.roll(n, 1, 3 - mu).reshape(-1) for mu in range(4)]
        self.U = U.reshape(4, self.V, 3, 3)
        self.Ud = [_dag(self.U[mu][self.dn[mu]]) for mu in range(4)]
        self.F = {(m, n): self.field(m, n) for m in range(4) for n in range(m)}

    def field(self, m, n):
        """F_mn from the four closed leaves around each site."""
        Um, Un, up, dn = self.U[m], self.U[n], self.up, self.dn
        s1, s2 = dn[m], dn[n]
        s3, s4, s5 = up[n][dn[m]], dn[n][dn[m]], dn[n][up[m]]
        Q = Um @ Un[up[m]] @ _dag(Um[up[n]]) @ _dag(Un)
        Q = Q + Un @ _dag(Um[s3]) @ _dag(Un[s1]) @ Um[s1]
        Q = Q + _dag(Um[s1]) @ _dag(Un[s4]) @ Um[s4] @ Un[s2]
        Q = Q + _dag(Un[s2]) @ Um[s2] @ Un[s5] @ _dag(Um)
        return (Q - _dag(Q)) / 8j

    def mul(self, m, q):
        return (m @ q.reshape(self.V, 3, -1)).reshape(q.shape)

    def apply(self, q, kappa):
        """D q; kappa: one value or one per column."""
        h = torch.zeros_like(q)
        for mu in range(4):
            w = self.mul(self.U[mu], q[self.up[mu]])
            h = h + (w - _times_gamma(mu, w))
            w = self.mul(self.Ud[mu], q[self.dn[mu]])
            h = h + (w + _times_gamma(mu, w))
        for (m, n), F in self.F.items():
            # both orders of (m, n) give the same term: 2 (i / 2) sigma_mn F_mn, sigma_mn = gamma_m gamma_n
            h = h + CSW * 1j * _times_gamma(m, _times_gamma(n, self.mul(F, q)))
        return q - kappa * h

    def solve(self, b, kappa):
        """D x = b column by column with BiCGSTAB, started again from the true residual until it stops falling."""
        dot = lambda x, y: (x.conj() * y).sum(dim=(0, 1, 2))  # noqa: E731
        nb = dot(b, b).real.sqrt()
        x = torch.zeros_like(b)
        best = None
        for _ in range(8):
            r = b - self.apply(x, kappa)
            res = float((dot(r, r).real.sqrt() / nb).max())
            if best is not None and res > 0.3 * best[0]:
                break
            best = (res, x)
            if res < 2e-15:
                break
            rt, p, rho = r, r, dot(r, r)
            goal, d = 1e-9 * float(dot(r, r).real.sqrt().max()), torch.zeros_like(b)
            for _ in range(400):
                v = self.apply(p, kappa)
                alpha = rho / dot(rt, v)
                s = r - alpha * v
                t = self.apply(s, kappa)
                om = dot(t, s) / dot(t, t)
                d = d + alpha * p + om * s
                r = s - om * t
                if float(dot(r, r).real.sqrt().max()) < goal:
                    break
                new = dot(rt, r)
                p = r + (new / rho) * (alpha / om) * (p - om * v)
                rho = new
            x = x + d
        return best[1]


def _from_canonical(X):  # [L, t, z, y, x, 4, 3] -> [V, 3, 4, L]
    return X.reshape(X.shape[0], -1, 4, 3).permute(1, 3, 2, 0).contiguous()


def _to_canonical(q, dims):
    return q.permute(3, 0, 2, 1).reshape(_block(dims, q.shape[3])).contiguous()


def _to_device_layout(q, case):
    """[V, 3, 4, L] -> what _values() gives, in 64 bits."""
    V, L = q.shape[0], q.shape[3]
    np = (L + 1) // 2
    y = torch.zeros(V, 12, np, 2, 2, dtype=F64, device=DEV)  # site, component, pair, {re, im}, column of the pair
    z = q.permute(0, 2, 1, 3).reshape(V, 12, L)
    for h in (0, 1):
        k = (L + 1 - h) // 2
        y[:, :, :k, 0, h] = z[:, :, h::2].real
        y[:, :, :k, 1, h] = z[:, :, h::2].imag
    if case["prec"] != "fp16":
        return y.reshape(-1)
    s = y.abs().amax(dim=(1, 3))  # per site, pair and column
    inv = torch.where(s > 0, 1 / s, torch.zeros_like(s))
    return (y * inv[:, None, :, None, :]).reshape(-1), s.reshape(-1)


def exact(case, seed):
    kind, dims = case["kind"], _dims(case)
    V, L = math.prod(dims), case.get("L", 1)
    if kind == "project":
        A, B = _project_inputs(case, seed)
        A, B = A.reshape(L, -1), B.reshape(L, -1)
        Y = B - (A.conj() @ B.T).T @ A
        return _to_device_layout(_from_canonical(Y.reshape(_block(dims, L))), case)
    if kind == "solve" and V * L > 131072 * 24:
        return None  # over 20 seconds
    plain = _Plain(dims, _links(dims, seed))
    if kind == "solve":
        ks, Ls = _systems(case)
        kappa = torch.tensor([k for k, n in zip(ks, Ls) for _ in range(n)], dtype=F64, device=DEV)
        return _to_canonical(plain.solve(_from_canonical(_sources(case, seed)), kappa), dims)
    if kind == "grad":
        k = case["kappa"]
        x = plain.solve(_from_canonical(_z4(dims, L, seed)), k)
        g5 = lambda q: q[:, :, [2, 3, 0, 1]]  # noqa: E731
        # lam = D^-H B = gamma_5 D^-1 gamma_5 B; a change of D changes the loss by -Re <lam, dD x>
        lam = g5(plain.solve(g5(_from_canonical(_z4(dims, L, seed))), k))
        U = _links(dims, seed).requires_grad_()
        kk = torch.tensor(k, dtype=F64, device=DEV, requires_grad=True)
        f = -(lam.conj() * _Plain(dims, U).apply(x, kk)).real.sum()
        gk, gU = torch.autograd.grad(f, (kk, U))
        return _to_canonical(x, dims), _to_canonical(lam, dims), gk, gU
    k = case["kappa"]
    if kind == "setup":
        return _to_canonical(plain.apply(_from_canonical(_gauss(dims, 1, seed, 3, "fp64")), k), dims)
    X = _gauss(dims, L, seed, 3, case["prec"])
    y = torch.empty((V, 3, 4, L), dtype=C128, device=DEV)
    for c in range(0, L, 8):
        y[..., c:c + 8] = plain.apply(_from_canonical(X[c:c + 8]), k)
    return _to_canonical(y, dims) if case["prec"] == "fp64" else _to_device_layout(y, case)
