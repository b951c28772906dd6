"""The work that users have this library do, as cases that can be timed.

A case names an operation of the public interface (``op``), a lattice and its
Schwarz blocks, the precision, the number of right-hand sides and, where there
is a coarse space, the number of test vectors:

* ``D``         the Wilson-clover operator on device fields (a program's own
                Krylov solver, the mass scan, the check of a residual);
* ``sap``       the Schwarz smoother;
* ``restrict``, ``prolong``   to and from the coarse lattice;
* ``solve``     the sources one after the other on a kept setup;
* ``batch``     the sources in one lockstep batch on a kept setup;
* ``setup_solve``, ``setup_batch``   the adaptive setup and then the solves: what
                one gauge configuration costs.

Links are near-unit SU(3) matrices exp(i eps H), drawn on the GPU from the seed.
Solves return the whole solutions, to a true residual of 1e-10.  The single
steps return the field they compute; a step taken in FP32 is kept in complex64,
the precision it has (the interface hands out complex128 for every precision).
"""
import math

import torch

import paper_1811_00355_gb300 as P

PREC = {"fp64": P.FP64, "fp32": P.FP32, "bf16": P.BF16, "fp16": P.FP16}
TOL = 1e-10
C128 = torch.complex128


def _case(name, op, L, block="4x4x4x4", prec="fp32", nrhs=1, n_v=1, eps=0.25, m0=-0.3, csw=1.2):
    return {"name": name, "op": op, "L": L, "block": block, "prec": prec, "nrhs": nrhs, "n_v": n_v,
            "eps": eps, "m0": m0, "csw": csw}


def listed():
    return [
        # the smallest call: one operator application on the smallest serving lattice, bound by latency
        _case("D_8x8x8x8_fp64", "D", "8x8x8x8", prec="fp64"),
        # the true residual of a solve on a mid-size serving lattice
        _case("D_24x24x24x48_fp64", "D", "24x24x24x48", prec="fp64", eps=0.2, csw=1.5),
        # CG on the normal equations in the mass scan of the large lattice
        _case("D_32x32x32x64_fp32", "D", "32x32x32x64", eps=0.2, m0=-0.125, csw=1.5),
        # the smoother on the 16^4 workload, one right-hand side
        _case("sap_16x16x16x16_fp32", "sap", "16x16x16x16"),
        # extents and blocks that are no powers of two
        _case("sap_8x12x16x24_fp32", "sap", "8x12x16x24", block="4x6x4x2", nrhs=3, m0=-0.2),
        # the smoother inside a batched solve
        _case("sap_24x24x24x48_fp32", "sap", "24x24x24x48", nrhs=4, eps=0.2, csw=1.5),
        # the projections: the twelve sources of a batch, and one field
        _case("restrict_16x16x16x16_fp32", "restrict", "16x16x16x16", nrhs=12, n_v=20),
        _case("prolong_24x24x24x48_fp32", "prolong", "24x24x24x48", n_v=24, eps=0.2, csw=1.5),
        # a small request on a resident configuration: launches and round trips count
        _case("solve_8x8x8x8_fp32", "solve", "8x8x8x8", nrhs=2, n_v=20),
        # the headline workload: setup and the 12 point sources one at a time
        _case("setup_solve_16x16x16x16_fp32", "setup_solve", "16x16x16x16", nrhs=12, n_v=20),
        # a new configuration in half storage, its sources in one batch
        _case("setup_batch_16x16x16x32_fp16", "setup_batch", "16x16x16x32", prec="fp16", nrhs=12, n_v=24,
              eps=0.2, m0=-0.125, csw=1.5),
        # the batched solves of a large lattice on a kept setup
        _case("batch_24x24x24x48_fp32", "batch", "24x24x24x48", nrhs=12, n_v=24, eps=0.2, m0=-0.125, csw=1.5),
    ]


# the extents that even blocks leave an even number of blocks for, and those blocks
_BLOCKS = {8: (2, 4), 12: (2, 6), 16: (2, 4, 8), 24: (2, 4, 6), 32: (4, 8), 48: (4, 6, 8), 64: (4, 8)}


def _draw_lattice(rng, low, high, square):
    """A lattice of roughly log-uniform volume in [low, high] and its blocks (64 to 256 sites; 4^4 half the time)."""
    target = math.exp(rng.uniform(math.log(low), math.log(high)))
    while True:
        L = [rng.choice(sorted(_BLOCKS)) for _ in range(4)]
        if not (max(low, target / 1.5) <= math.prod(L) <= min(high, target * 1.5)):
            continue
        if square and rng.random() < 0.5:
            if any(4 not in _BLOCKS[v] for v in L):
                continue
            b = [4, 4, 4, 4]
        else:
            b = [rng.choice(_BLOCKS[v]) for v in L]
        if 64 <= math.prod(b) <= 256:
            return "x".join(map(str, L)), "x".join(map(str, b))


def draw(rng):
    op = rng.choice(["D", "sap", "restrict", "prolong", "solve", "batch", "setup_solve", "setup_batch"])
    c = {"op": op, "eps": round(rng.uniform(0.15, 0.25), 3), "m0": round(rng.uniform(-0.2, 0.1), 3),
         "csw": round(rng.uniform(1.0, 1.6), 2), "nrhs": 1, "n_v": 1, "prec": "fp32"}
    if op == "D":
        c["L"], c["block"] = _draw_lattice(rng, 2 ** 12, 2 ** 21, True)
        c["prec"] = rng.choice(["fp32", "fp64"])
    elif op == "sap":
        c["L"], c["block"] = _draw_lattice(rng, 2 ** 12, 2 ** 19, True)
        c["nrhs"] = rng.choice([1, 2, 3, 4])
    elif op in ("restrict", "prolong"):
        c["L"], c["block"] = _draw_lattice(rng, 2 ** 13, 2 ** 19, True)
        c["nrhs"] = rng.choice([1, 1, 3, 12])
        c["n_v"] = rng.randint(8, 32)
    else:
        c["L"], c["block"] = _draw_lattice(rng, 2 ** 12, 2 ** 17, True)
        c["prec"] = rng.choice(["fp32", "fp32", "bf16", "fp16"])
        c["nrhs"] = rng.choice([1, 2, 4, 12]) if "batch" in op else rng.choice([1, 2, 4])
        c["n_v"] = rng.randint(12, 24)
    return c


# ---- inputs ------------------------------------------------------------------------------
def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def _volume(c):
    return math.prod(_ints(c["L"]))


def _gaussian(shape, gen):
    """Iid N(0, 1) real and imaginary parts."""
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device="cuda", dtype=torch.float64))


def _links(c, gen):
    """exp(i eps H), H Gaussian, traceless and Hermitian: the series of a sixteenth (its norm is below 0.2), squared."""
    def mul(X, Y):
        return X[:, :, 0:1] * Y[:, 0:1] + X[:, :, 1:2] * Y[:, 1:2] + X[:, :, 2:3] * Y[:, 2:3]

    V = _volume(c)
    U = torch.empty((V * 4, 3, 3), dtype=C128, device="cuda")
    one = torch.eye(3, dtype=C128, device="cuda")
    for part in U.split(1 << 21):
        A = _gaussian(part.shape, gen)
        H = 0.5 * (A + A.mH)
        H -= (H.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3.0)[:, None, None] * one
        X = (1j / 16.0 * c["eps"]) * H
        E = one + X / 12.0
        for k in range(11, 0, -1):
            E = one + mul(X, E) / k
        for _ in range(4):
            E = mul(E, E)
        part.copy_(E)
    return U.view(V, 4, 3, 3)


def _fields(c, gen):
    V = _volume(c)
    if c["op"] in ("D", "sap", "restrict"):
        return _gaussian((c["nrhs"], V, 4, 3), gen)
    # point sources, the spin and colour running first, at a site of the seed's
    site = int(torch.randint(V, (1,), generator=gen, device="cuda"))
    b = torch.zeros((c["nrhs"], V, 4, 3), dtype=C128, device="cuda")
    for k in range(c["nrhs"]):
        b[k, (site + 97 * (k // 12)) % V, k % 12 // 3, k % 3] = 1.0
    return b


def _order(c):
    """Lexicographic sites in the order (aggregate, site in it), and the aggregates' count."""
    L, b = _ints(c["L"]), _ints(c["block"])
    g = [L[m] // b[m] for m in range(4)]
    i = torch.arange(math.prod(L), device="cuda").view(g[3], b[3], g[2], b[2], g[1], b[1], g[0], b[0])
    return i.permute(0, 2, 4, 6, 1, 3, 5, 7).reshape(math.prod(g), math.prod(b))


def _test_vectors(c, gen):
    """Gaussian vectors, orthonormal in every aggregate and chirality, as [n_v][V][4][3] and as [X][chirality][6 |X|][n_v]."""
    sites, V, n = _order(c), _volume(c), c["n_v"]
    X, Vb = sites.shape
    A = _gaussian((X, 2, 6 * Vb, n), gen)
    for _ in range(2):                           # A R^-1 with A^H A = R^H R
        R = torch.linalg.cholesky(A.mH @ A).mH
        A = torch.linalg.solve_triangular(R, A, upper=True, left=False)
    v = torch.empty((n, V, 4, 3), dtype=C128, device="cuda")
    v[:, sites.view(-1)] = A.view(X, 2, Vb, 2, 3, n).permute(5, 0, 2, 1, 3, 4).reshape(n, V, 4, 3)
    return v, A


def _inputs(c, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    d = {"links": _links(c, gen)}
    if c["op"] == "prolong":
        d["x"] = _gaussian((c["nrhs"], _order(c).shape[0], 2 * c["n_v"]), gen)
    else:
        d["x"] = _fields(c, gen)
    if c["op"] in ("restrict", "prolong"):
        d["vectors"], d["basis"] = _test_vectors(c, gen)
    return d


# ---- the calls -----------------------------------------------------------------------------
def prepare(case, seed):
    c, d = case, _inputs(case, seed)
    step = c["op"] in ("D", "sap", "restrict", "prolong")
    p = P.default_params(L=_ints(c["L"]), sap_block=_ints(c["block"]), n_v=c["n_v"], m0=c["m0"], csw=c["csw"],
                         precision=PREC["fp32" if step else c["prec"]], outer_restart=12, seed=1 + seed % 1000)
    s = P.DDAMG(p, d["links"], stream=torch.cuda.current_stream().cuda_stream)
    if "vectors" in d:
        s.set_test_vectors(d["vectors"])
    if c["op"] in ("solve", "batch"):
        s.run_setup()
    return {"op": c["op"], "solver": s, "x": d["x"], "prec": PREC[c["prec"]], "single": c["prec"] != "fp64"}


def run(state):
    s, x, op = state["solver"], state["x"], state["op"]
    if op == "setup_solve" or op == "setup_batch":
        s.run_setup()
    if op == "solve" or op == "setup_solve":
        return s.solve(x, TOL)[0]
    if op == "batch" or op == "setup_batch":
        return s.solve_batched(x, TOL)[0]
    call = {"D": s.apply_D, "sap": s.sap, "restrict": s.restrict, "prolong": s.prolong}[op]
    y = call(x, state["prec"])
    return y.to(torch.complex64) if state["single"] else y


def work(case):
    """Each input read and each output written once, in the storage that the precision needs (links as two rows, the
    clover blocks packed); the arithmetic of the method, for solves at the iteration counts of the 16^4 workload."""
    c, V, n, op = case, _volume(case), case["nrhs"], case["op"]
    r = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}[c["prec"]]
    field = 24 * 8 * V * n                       # a field of the interface
    links, clover = 48 * r * V, 72 * r * V
    if op == "D":
        return {"bytes": 2 * field + links + clover, "flops": 1920.0 * V * n}
    if op == "sap":
        # 4 cycles of two half-lattice sweeps, each a residual and a block solve of 4 iterations
        sweep = V / 2 * 1968 + V / 4 * (2 * 1900 + 4 * 4128)
        return {"bytes": 2 * field + links + 2 * clover, "flops": 8.0 * sweep * n}
    if op in ("restrict", "prolong"):
        coarse = V // math.prod(_ints(c["block"])) * 2 * c["n_v"] * 16 * n
        return {"bytes": field + coarse + 24 * r * V * c["n_v"], "flops": 96.0 * V * c["n_v"] * n}
    per_site = 1.46e6 * n + (7.27e6 if "setup" in op else 0.0)
    return {"bytes": 2 * field + 576 * V, "flops": per_site * V}


# ---- the single steps in 64 bits, in plain torch ---------------------------------------------
def _gammas():
    s = [[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]]
    g = torch.zeros((4, 4, 4), dtype=C128, device="cuda")
    for k in range(3):
        m = torch.tensor(s[k], dtype=C128, device="cuda")
        g[k, :2, 2:], g[k, 2:, :2] = -1j * m, 1j * m
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2, dtype=C128, device="cuda")
    return g


class _Wilson:
    """D of one gauge field: site-diagonal 6x6 blocks of the clover term and the eight hops."""

    def __init__(self, c, U):
        L = _ints(c["L"])
        V = math.prod(L)
        i = torch.arange(V, device="cuda").view(L[::-1])
        self.U, self.g = U, _gammas()
        self.fwd = [i.roll(-1, 3 - m).reshape(-1) for m in range(4)]
        self.bwd = [i.roll(1, 3 - m).reshape(-1) for m in range(4)]
        sign = torch.ones(L[::-1], dtype=torch.float64, device="cuda")
        last, first = sign.clone(), sign.clone()
        last[-1], first[0] = -1.0, -1.0
        self.edge = {3: (last.view(-1, 1, 1), first.view(-1, 1, 1))}
        self.A = torch.zeros((V, 2, 6, 6), dtype=C128, device="cuda")
        for m in range(4):
            for n in range(m):
                F = self._leaves(m, n)
                F = F - F.mH
                gg = self.g[m] @ self.g[n]
                for ch in range(2):
                    b = gg[2 * ch:2 * ch + 2, 2 * ch:2 * ch + 2]
                    for s in range(2):
                        for t in range(2):
                            self.A[:, ch, 3 * s:3 * s + 3, 3 * t:3 * t + 3] -= (c["csw"] / 16.0) * b[s, t] * F
        self.A.diagonal(dim1=-2, dim2=-1).add_(4.0 + c["m0"])

    def _leaves(self, m, n):
        """The four plaquettes of the m-n plane that start and end at a site."""
        U, f, b = self.U, self.fwd, self.bwd
        M, N = U[:, m], U[:, n]
        q = M @ N[f[m]] @ M[f[n]].mH @ N.mH
        q += N @ M[f[n][b[m]]].mH @ N[b[m]].mH @ M[b[m]]
        q += M[b[m]].mH @ N[b[n][b[m]]].mH @ M[b[n][b[m]]] @ N[b[n]]
        q += N[b[n]].mH @ M[b[n]] @ N[f[m][b[n]]] @ M.mH
        return q

    def hops(self, x):
        out = torch.zeros_like(x)
        for m in range(4):
            up = x[self.fwd[m]] @ self.U[:, m].mT
            dn = x[self.bwd[m]] @ self.U[self.bwd[m], m].conj()
            if m in self.edge:
                up, dn = up * self.edge[m][0], dn * self.edge[m][1]
            out += up + dn
            out -= self.g[m] @ (up - dn)
        return out

    def site(self, A, x):
        return (A @ x.reshape(-1, 2, 6, 1)).reshape(x.shape)

    def apply(self, x):
        return self.site(self.A, x) - 0.5 * self.hops(x)


def _smooth(c, D, b):
    """4 cycles over the two colours of blocks, each block solved by 4 minimal-residual steps on its even sites."""
    L, sites = _ints(c["L"]), _order(c)
    V, blk = math.prod(L), _ints(c["block"])
    i = torch.arange(V, device="cuda")
    x = [i % L[0], i // L[0] % L[1], i // (L[0] * L[1]) % L[2], i // (L[0] * L[1] * L[2])]
    odd = (x[0] + x[1] + x[2] + x[3]) % 2
    colour = sum(x[m] // blk[m] for m in range(4)) % 2
    owner = torch.empty(V, dtype=torch.int64, device="cuda")
    owner[sites] = torch.arange(sites.shape[0], device="cuda")[:, None]
    Ainv = torch.linalg.inv(D.A)

    def inner(u, v):
        return (u.conj() * v).sum((-1, -2))[sites].sum(-1)[owner][:, None, None]

    y = torch.zeros_like(b)
    for _ in range(4):
        for k in (0, 1):
            mask = (colour == k).to(torch.float64)[:, None, None]
            even = mask * (odd == 0).to(torch.float64)[:, None, None]
            uneven = mask - even
            # hops that stay in a block: blocks of one colour never touch
            to_even = lambda v: -0.5 * even * D.hops(v)        # noqa: E731
            to_odd = lambda v: -0.5 * uneven * D.hops(v)       # noqa: E731
            r = mask * (b - D.apply(y))
            res = even * r - to_even(D.site(Ainv, uneven * r))
            e = torch.zeros_like(b)
            for _ in range(4):
                p = even * D.site(D.A, res) - to_even(D.site(Ainv, to_odd(res)))
                pp = inner(p, p).real
                a = torch.where(pp > 0, inner(p, res) / torch.where(pp > 0, pp, 1.0), 0.0)
                e, res = e + a * res, res - a * p
            y = y + e + D.site(Ainv, uneven * r - to_odd(e))
    return y


def exact(case, seed):
    c, op = case, case["op"]
    if op not in ("D", "sap", "restrict", "prolong"):
        return None                              # a Krylov solver run in plain torch takes minutes
    d = _inputs(c, seed)
    if op in ("D", "sap"):
        D = _Wilson(c, d["links"])
        return torch.stack([D.apply(v) if op == "D" else _smooth(c, D, v) for v in d["x"]])
    A, n, V = d["basis"], c["nrhs"], _volume(c)
    sites = _order(c)
    X, Vb = sites.shape
    if op == "restrict":
        x = d["x"][:, sites.view(-1)].view(n, X, Vb, 2, 6).permute(1, 3, 2, 4, 0).reshape(X, 2, 6 * Vb, n)
        return (A.mH @ x).permute(3, 0, 1, 2).reshape(n, X, 2 * c["n_v"]).contiguous()
    y = A @ d["x"].view(n, X, 2, c["n_v"]).permute(1, 2, 3, 0)
    out = torch.empty((n, V, 4, 3), dtype=C128, device="cuda")
    out[:, sites.view(-1)] = y.view(X, 2, Vb, 2, 3, n).permute(5, 0, 2, 1, 3, 4).reshape(n, V, 4, 3)
    return out
