"""The work this library is measured on.

Each case is one call (or the pair of calls a solver makes) through the Python
binding, on the lattices, boxes and right-hand sides of the repository's own
workloads, or on drawn ones of the same ranges:

  dslash     M_{p,1-p}: one checkerboard block of D (dslash_eo)
  normal     M_pc, then M_pc^+ of its result: what a CG iteration applies
  apply_d    D (whole lattice) or D_Omega (boxes), both checkerboards
  solve      D x = b by even-odd CGNE, FP64 or mixed FP32/FP64: a whole call
  filter     the Chebyshev filter of the multigrid set-up
  force      the link force of Re <X, D Y>: the backward direction
  nn_apply   the learned preconditioner K on one residual
  nn_train   one Adam step of K on a batch of residuals

Links are SU(3): "exp" exp(i 0.3 H) with Gaussian H (the weak-coupling
ensembles of the workloads), or "haar" random.  Fields are Gaussian.
"""

import math

import numpy as np
import torch

from paper_2203_17119_gb300 import dwf as G

PREC = {"f64": G.FP64, "f32": G.FP32, "bf16": G.BF16}
REAL = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
WORD = {"f64": 8, "f32": 4, "bf16": 2}
M5 = 1.8
MOBIUS, SHAMIR = (1.5, 0.5), (1.0, 0.0)
# the batched workload's six Dirichlet blocks of uneven extents
SIX = "8x8x8x8 8x8x12x12 12x12x12x12 12x12x16x16 16x16x16x12 16x16x16x16"


def _case(op, dims, Ls, prec, *, nrhs=1, action=MOBIUS, mf=0.01, boxes="", links="exp", dagger=False, order=0,
          tol=0.0, tuned=False, name=None):
    c = {"op": op, "Lx": dims[0], "Ly": dims[1], "Lz": dims[2], "Lt": dims[3], "Ls": Ls, "prec": prec, "nrhs": nrhs,
         "b5": action[0], "c5": action[1], "mf": mf, "boxes": boxes, "links": links, "dagger": dagger,
         "order": order, "tol": tol, "tuned": tuned}
    return dict(c, name=name) if name else c


def _cube(L):
    return (L, L, L, L)


def listed():
    return [
        # the smallest call: one block of Shamir D on 4^4 x 8 (the check-out lattice), launch and latency
        _case("dslash", _cube(4), 8, "f64", action=SHAMIR, links="haar", name="dslash_f64_4x8"),
        # the same lattice solved in FP64: a few hundred dependent small kernels
        _case("solve", _cube(4), 8, "f64", action=SHAMIR, links="haar", tol=1e-12, name="solve_f64_4x8"),
        # the mid-size Moebius lattice of the mixed-precision workload: one FP32 block of D
        _case("dslash", _cube(16), 12, "f32", name="dslash_f32_16x12"),
        # its mixed-precision solve, tuned first as the README does it; 1e-12 is what a molecular-dynamics
        # trajectory asks for so that it is reversible
        _case("solve", _cube(16), 12, "f32", tol=1e-12, tuned=True, name="solve_f32_16x12"),
        # six uneven Dirichlet blocks, 16 right-hand sides at once (domain-decomposed HMC's local operators)
        _case("apply_d", _cube(24), 16, "f32", nrhs=16, boxes=SIX, name="dirichlet_f32_six_r16"),
        # the paper's per-GPU volume: the normal Schur operator of one FP32 CG iteration
        _case("normal", _cube(32), 16, "f32", mf=0.005, name="normal_f32_32x16"),
        # the same operator with BF16 operands
        _case("normal", _cube(24), 16, "bf16", mf=0.005, name="normal_bf16_24x16"),
        # FP64 D: the true residuals and reliable updates of every solve
        _case("apply_d", _cube(24), 16, "f64", mf=0.005, name="apply_d_f64_24x16"),
        # the filter of the multigrid set-up on the interior box of a width-2 band, 8 vectors: a ragged box
        _case("filter", _cube(16), 12, "f32", nrhs=8, action=SHAMIR, boxes="14x14x14x14@1,1,1,1", order=10,
              name="filter_f32_box14x12_r8"),
        # the force of a DD-HMC step: FP64, one pair of solved fields
        _case("force", _cube(16), 12, "f64", name="force_f64_16x12"),
        # the learned preconditioner inside flexible GCR
        _case("nn_apply", _cube(24), 16, "f32", mf=0.005, name="nn_apply_24x16"),
        # one training step of it on a batch of four residuals
        _case("nn_train", _cube(16), 12, "f32", nrhs=4, mf=0.005, name="nn_train_16x12_r4"),
    ]


def _even(rng, lo, hi):
    return 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)


def draw(rng):
    op = rng.choice(["dslash", "dslash", "normal", "normal", "apply_d", "apply_d", "solve", "filter", "force",
                     "nn_apply", "nn_train"])
    top = {"solve": 8, "nn_train": 12, "filter": 16, "force": 20}.get(op, 28)
    dims = [_even(rng, 4, top) for _ in range(4)]
    Ls = rng.choice([8, 10, 12, 14, 16, 16])
    prec = {"solve": ["f64", "f32"], "force": ["f64", "f64", "f32"], "filter": ["f32", "f32", "f64"],
            "nn_apply": ["f32"], "nn_train": ["f32"]}.get(op, ["f32", "f32", "f64", "bf16"])
    prec = rng.choice(prec)
    most = max(1, min({"nn_train": 4, "solve": 2, "force": 2, "nn_apply": 2, "filter": 8}.get(op, 16), 256 // Ls))
    nrhs = rng.choice([1, 1, 1, min(2, most), min(3, most), most])
    # no more work than the largest listed cases: FP64 counts for its slower arithmetic
    cost = {"nn_apply": 4, "nn_train": 24, "filter": 8}.get(op, 1) * (4 if prec == "f64" else 1) * Ls * nrhs
    while dims[0] * dims[1] * dims[2] * dims[3] * cost > 32 ** 4 * 16:
        k = max(range(4), key=lambda m: dims[m])
        dims[k] -= 2
    boxes = ""
    if op in ("normal", "apply_d", "filter", "solve") and rng.random() < 0.4:
        boxes = " ".join("x".join(str(rng.randint(min(3, L), L)) for L in dims) + "@"
                         + ",".join(str(rng.randrange(L)) for L in dims) for _ in range(rng.choice([1, 1, 2, 3])))
    return _case(op, dims, Ls, prec, nrhs=nrhs, action=rng.choice([MOBIUS, MOBIUS, SHAMIR]),
                 mf=rng.choice([0.005, 0.01, 0.02]) if op != "solve" else rng.choice([0.01, 0.02]), boxes=boxes,
                 links=rng.choice(["exp", "exp", "haar"]), dagger=rng.random() < 0.3,
                 order=rng.randint(4, 12) if op == "filter" else 0, tol=1e-12 if op == "solve" else 0.0)


# ---------------------------------------------------------------- inputs


def _dims(c):
    return (c["Lx"], c["Ly"], c["Lz"], c["Lt"])


def _boxes(c):
    got = []
    for text in c["boxes"].split():
        ext, _, org = text.partition("@")
        got.append((tuple(int(v) for v in org.split(",")) if org else (0, 0, 0, 0),
                    tuple(int(v) for v in ext.split("x"))))
    return got


def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(1009 * int(seed) + k)


def _links(c, seed):
    """[site lex][mu][3][3] complex128 SU(3) on the GPU."""
    n = 4 * c["Lx"] * c["Ly"] * c["Lz"] * c["Lt"]
    g = _gen(seed, 1)
    z = torch.view_as_complex(torch.randn((n, 3, 3, 2), dtype=torch.float64, device="cuda", generator=g))
    if c["links"] == "exp":   # exp(i eps H), H traceless Hermitian of unit-variance Gell-Mann coefficients
        H = (z + z.mH) / (2 * math.sqrt(2))
        H = H - torch.diagonal(H, dim1=1, dim2=2).mean(-1)[:, None, None] * torch.eye(3, device="cuda")
        A = 0.3j * H
        one = torch.eye(3, dtype=A.dtype, device="cuda").expand_as(A)
        z = one + A
        P = A
        for k in range(2, 6):
            P = (P[:, :, :, None] * A[:, None, :, :]).sum(2) / k
            z = z + P
    r0 = z[:, 0] / torch.linalg.vector_norm(z[:, 0], dim=1, keepdim=True)
    r1 = z[:, 1] - (r0.conj() * z[:, 1]).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=1).conj()
    return torch.stack((r0, r1, r2), 1).reshape(-1, 4, 3, 3)


def _gauss(shape, prec, seed, k):
    return torch.randn(shape, dtype=REAL[prec] if prec != "bf16" else torch.float32, device="cuda",
                       generator=_gen(seed, k)).to(REAL[prec])


def _shapes(c):
    """(sites of parity 0, of parity 1) of the case's domain."""
    n = [0, 0]
    for org, ext in _boxes(c) or [((0, 0, 0, 0), _dims(c))]:
        v = ext[0] * ext[1] * ext[2] * ext[3]
        p = sum(org) % 2   # the origin's parity has the odd site, if the volume is odd
        n[p] += (v + 1) // 2
        n[1 - p] += v // 2
    return n


def _weights(seed):
    """(W1, W2) of the 1 -> 16 -> 1 network: 1/d^2 on the identity transport and small Gaussian rest."""
    r = np.random.default_rng(int(seed) + 17)

    def z(*s):
        return 0.02 * (r.standard_normal(s) + 1j * r.standard_normal(s))

    W1, W2 = z(11, 16, 1, 4, 4), z(11, 1, 16, 4, 4)
    W1[0, 0, 0] += np.eye(4) / (MOBIUS[0] * (4 - M5) + 1) ** 2
    W2[0, 0, 0] += np.eye(4)
    return W1, W2


def _inputs(c, seed):
    """The input fields of a case, in the library's layouts."""
    n0, n1 = _shapes(c)
    tail = (12, c["nrhs"], c["Ls"], 2)
    op = c["op"]
    if op in ("dslash", "normal", "filter", "nn_apply"):
        return [_gauss((n1,) + tail, c["prec"], seed, 2)]
    if op == "apply_d":
        return [_gauss((n0 + n1,) + tail, c["prec"], seed, 2)]
    if op == "solve":
        return [_gauss((n0 + n1,) + tail, "f64", seed, 2)]
    if op == "force":
        return [_gauss((n0 + n1,) + tail, c["prec"], seed, k) for k in (2, 3)]
    return [_gauss((n1,) + tail, "f32", seed, k) for k in (2, 3)]   # nn_train: r, e


def _top(c):
    """Just above the top of the spectrum of M_pc^+ M_pc."""
    return 110.0 if c["c5"] else 30.0


def prepare(case, seed):
    c = case
    h = G.Handle(_dims(c), c["Ls"], G.Action(M5, c["mf"], c["b5"], c["c5"]), boxes=_boxes(c) or None,
                 nrhs_max=c["nrhs"])
    h.set_gauge(_links(c, seed).reshape(-1))
    s = {"c": c, "h": h, "in": _inputs(c, seed), "prec": PREC[c["prec"]]}
    if c["tuned"]:
        h.autotune(c["nrhs"], s["prec"])
    op, n = c["op"], c["nrhs"]
    if op == "dslash":
        s["out"] = [h.empty_cb(0, n, s["prec"])]
    elif op == "normal":
        s["out"] = [h.empty_cb(1, n, s["prec"]) for _ in range(2)]
    elif op == "filter":
        s["out"] = [h.empty_cb(1, n, s["prec"])]
    elif op == "apply_d":
        s["out"] = [h.empty_full(n, s["prec"])]
    elif op == "solve":
        s["out"] = [h.empty_full(n, G.FP64)]
    elif op == "force":
        V = c["Lx"] * c["Ly"] * c["Lz"] * c["Lt"]
        s["out"] = [torch.empty((V, 4, 3, 3, 2), dtype=torch.float64, device="cuda")]
    else:
        s["K"] = G.NN()
        s["K"].set_weights(*_weights(seed))
        s["out"] = [h.empty_cb(1, n, G.FP32)]
    return s


def run(state):
    s, c, h = state, state["c"], state["h"]
    op, n, p, dag = c["op"], c["nrhs"], s["prec"], c["dagger"]
    x, out = s["in"], s["out"]
    if op == "dslash":
        h.dslash_eo(out[0], x[0], 0, dagger=dag, prec=p, nrhs=n)
    elif op == "normal":
        h.mpc(out[0], x[0], dagger=dag, prec=p, nrhs=n)
        h.mpc(out[1], out[0], dagger=not dag, prec=p, nrhs=n)
    elif op == "apply_d":
        (h.dirichlet_block if h.boxes else h.apply_d)(out[0], x[0], dagger=dag, prec=p, nrhs=n)
    elif op == "solve":
        h.cgne_solve(out[0], x[0], nrhs=n, tol=c["tol"], inner=p)
    elif op == "filter":
        h.chebyshev_filter(out[0], x[0], c["order"], _top(c) / 50, _top(c), prec=p, nrhs=n)
    elif op == "force":
        h.force(out[0], x[0], x[1], prec=p, nrhs=n)
    elif op == "nn_apply":
        s["K"].apply(h, out[0], x[0], nrhs=n)
    else:
        loss = s["K"].train_step(h, x[0], x[1], nrhs=n, loss_kind="a2")
        g1, g2 = s["K"].last_grad(h)
        # the step's arithmetic is FP32; the binding widens what it returns
        return {"loss": torch.tensor(loss, dtype=torch.float32), "g1": g1.astype(np.complex64),
                "g2": g2.astype(np.complex64)}
    return out


# ------------------------------------------------------------ cost model


def work(case):
    """Bytes read and written once, and operations: 1320 per site and lane for the hop, 24 / 48 / 120 for the
    fifth-dimension factors S5 / B / (M^-1)."""
    c = case
    n0, n1 = _shapes(c)
    N5, w = c["Ls"] * c["nrhs"], WORD[c["prec"]]
    half, link = 24 * N5 * w, 72 * w     # a site's spinor; its four links
    V = n0 + n1
    hop = 1320 * N5
    op = c["op"]
    if op == "dslash":
        return {"bytes": V * half + V * link, "flops": n0 * (hop + (48 * N5 if c["c5"] else 0))}
    if op == "normal":
        return {"bytes": 3 * n1 * half + V * link, "flops": 2 * V * hop + 2 * n1 * N5 * 384}
    if op == "apply_d":
        return {"bytes": 2 * V * half + V * link, "flops": V * (hop + 96 * N5)}
    if op == "filter":
        return {"bytes": 2 * n1 * half + V * link, "flops": c["order"] * (2 * V * hop + 2 * n1 * N5 * 400)}
    if op == "solve":   # at least some tens of CG iterations; a floor of the fields alone is meaningless
        return {"bytes": 2 * V * 24 * N5 * 8 + V * 72 * 8, "flops": 100 * (2 * V * hop + 2 * n1 * N5 * 400)}
    if op == "force":
        return {"bytes": 2 * V * half + V * link + V * 72 * 8, "flops": V * 4 * 336 * N5}
    if op == "nn_apply":
        return {"bytes": 2 * n1 * half + V * link, "flops": N5 * 8 * (8 * n0 * 36 * 2 + 3 * (n0 * 1024 + n1 * 144))}
    A = 2 * (2 * V * hop + 2 * n1 * N5 * 384)
    mix = N5 * 8 * 3 * (16 * 16 * 8 * n0 + 16 * 16 * 3 * n1)
    return {"bytes": n1 * half + V * link + 2 * 11 * 16 * 16 * 8 * 3, "flops": 2 * A + 5 * mix}


# --------------------------------------------------- 64-bit plain values


class _Lattice:
    """One box (or the whole lattice) of a case in plain torch: fields [t, z, y, x, colour, spin, rhs, s]."""

    def __init__(self, c, U, box):
        self.c, self.L = c, _dims(c)
        org, ext = box
        self.ext = ext
        self.shape = (ext[3], ext[2], ext[1], ext[0])
        ax = [torch.arange(e, device="cuda") for e in ext]
        t, z, y, x = torch.meshgrid(ax[3], ax[2], ax[1], ax[0], indexing="ij")
        par = ((x + y + z + t + sum(org)) % 2).reshape(-1)
        self.idx = [torch.nonzero(par == p).reshape(-1) for p in range(2)]
        g = [(v + o) % L for v, o, L in zip((x, y, z, t), org, self.L)]
        lex = (g[0] + self.L[0] * (g[1] + self.L[1] * (g[2] + self.L[2] * g[3]))).reshape(-1)
        self.U = []
        for mu, v in enumerate((x, y, z, t)):
            u = U[lex, mu].clone()
            if ext[mu] < self.L[mu]:
                u[(v == ext[mu] - 1).reshape(-1)] = 0   # the link leaves the block
            self.U.append(u)
        s = [[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]]
        self.gam = []
        for k in range(4):
            m = torch.zeros((4, 4), dtype=torch.complex128)
            if k < 3:
                a = torch.tensor(s[k], dtype=torch.complex128)
                m[:2, 2:], m[2:, :2] = -1j * a, 1j * a
            else:
                m[:2, 2:] = m[2:, :2] = torch.eye(2)
            self.gam.append(m.cuda())

    def low(self):
        """The same lattice in 32 bits, to precondition a 64-bit refinement."""
        o = object.__new__(_Lattice)
        o.__dict__ = dict(self.__dict__, U=[u.to(torch.complex64) for u in self.U],
                          gam=[g.to(torch.complex64) for g in self.gam])
        return o

    def zeros(self, like):
        return torch.zeros(self.shape + tuple(like), dtype=self.U[0].dtype, device="cuda")

    def put(self, cb, p, f=None):
        """cb [site, 12, r, s] complex -> field."""
        f = self.zeros((3, 4) + cb.shape[2:]) if f is None else f
        f.view((-1,) + f.shape[4:])[self.idx[p]] = cb.unflatten(1, (4, 3)).transpose(1, 2)
        return f

    def get(self, f, p):
        return f.reshape((-1,) + f.shape[4:])[self.idx[p]].transpose(1, 2).flatten(1, 2)

    def mul(self, u, f):
        return torch.matmul(u, f.reshape(u.shape[0], 3, -1)).reshape(f.shape)

    def spin(self, m, f):
        return torch.matmul(m, f.flatten(-2)).reshape(f.shape)

    def roll(self, f, n, mu):
        return torch.roll(f, n, 3 - mu)

    def hop(self, f, dag=False):
        out = torch.zeros_like(f)
        one = torch.eye(4, dtype=f.dtype, device="cuda")
        for mu in range(4):
            sg = -1 if dag else 1
            out += self.spin(one - sg * self.gam[mu], self.mul(self.U[mu], self.roll(f, -1, mu)))
            out += self.spin(one + sg * self.gam[mu], self.roll(self.mul(self.U[mu].mH, f), 1, mu))
        return out

    def s5(self, f, dag=False):
        dn, up = torch.roll(f, 1, -1), torch.roll(f, -1, -1)
        dn[..., 0] *= -self.c["mf"]
        up[..., -1] *= -self.c["mf"]
        if dag:
            dn, up = up, dn
        return torch.cat((dn[..., :2, :, :], up[..., 2:, :, :]), dim=-3)

    def B(self, f, dag=False):
        return self.c["b5"] * f + self.c["c5"] * self.s5(f, dag)

    def M(self, f, dag=False):
        return (self.c["b5"] * (4 - M5) + 1) * f + (self.c["c5"] * (4 - M5) - 1) * self.s5(f, dag)

    def Minv(self, f, dag=False):
        Ls = self.c["Ls"]
        e = torch.eye(Ls, dtype=torch.float64)
        S = torch.roll(e, 1, 0)          # (S x)_s = x_{s-1}
        S[0] *= -self.c["mf"]
        d, k = self.c["b5"] * (4 - M5) + 1, self.c["c5"] * (4 - M5) - 1
        R = torch.roll(e, -1, 0)         # (R x)_s = x_{s+1}
        R[-1] *= -self.c["mf"]
        m = [torch.linalg.inv(d * e + k * s).T.to(f.dtype).cuda() for s in (S, R)]
        if dag:
            m = m[::-1]
        return torch.cat((f[..., :2, :, :] @ m[0], f[..., 2:, :, :] @ m[1]), dim=-3)

    def D(self, f, dag=False):
        if not dag:
            b = self.B(f)
            return (4 - M5) * b - 0.5 * self.hop(b) + f - self.s5(f)
        return self.B((4 - M5) * f - 0.5 * self.hop(f, True), True) + f - self.s5(f, True)

    def mpc(self, f, dag=False):
        if not dag:
            return self.M(f) - 0.25 * self.hop(self.B(self.Minv(self.hop(self.B(f)))))
        return self.M(f, True) - 0.25 * self.B(self.hop(self.Minv(self.B(self.hop(f, True), True), True), True), True)

    def normal(self, f):
        return self.mpc(self.mpc(f), True)

    def solve(self, b):
        """D x = b: 32-bit CGNE inside 64-bit residual refinement; 1e-13 of |b|."""
        lo, bn = self.low(), float(torch.linalg.vector_norm(b))
        x = torch.zeros_like(b)
        for _ in range(8):
            res = b - self.D(x)
            rn = float(torch.linalg.vector_norm(res))
            if rn < 1e-13 * bn:
                break
            r = lo.D((res / rn).to(torch.complex64), True)
            e, p, rr = torch.zeros_like(r), r.clone(), float(torch.linalg.vector_norm(r)) ** 2
            end = rr * 1e-10
            for _ in range(3000):
                q = lo.D(p)
                a = rr / float(torch.linalg.vector_norm(q)) ** 2
                e += a * p
                r -= a * lo.D(q, True)
                new = float(torch.linalg.vector_norm(r)) ** 2
                if new < end:
                    break
                p = r + (new / rr) * p
                rr = new
            x += rn * e.to(torch.complex128)
        return x

    def force(self, X, Y):
        Z, out = self.B(Y), []
        one = torch.eye(4, dtype=X.dtype, device="cuda")
        V = self.U[0].shape[0]

        def dot(a, b):   # sum over spin and lanes of a_i conj(b_j)
            return torch.matmul(a.reshape(V, 3, -1), b.reshape(V, 3, -1).mH)

        for mu in range(4):
            m = dot(self.roll(Z, -1, mu), self.spin(one - self.gam[mu], X))
            m = m + dot(Z, self.spin(one + self.gam[mu], self.roll(X, -1, mu))).mH
            f = torch.matmul(self.U[mu], m)
            f = 0.5 * (f - f.mH)
            f = f - torch.diagonal(f, dim1=1, dim2=2).mean(-1)[:, None, None] * torch.eye(3, device="cuda")
            out.append(-0.5 * f)
        return torch.stack(out, 1)

    def transport(self, f, d):
        if d == 0:
            return f
        if d <= 4:
            return self.mul(self.U[d - 1], self.roll(f, -1, d - 1))
        if d <= 8:
            return self.roll(self.mul(self.U[d - 5].mH, f), 1, d - 5)
        z = torch.zeros_like(f[..., :1])
        return torch.cat((f[..., 1:], z), -1) if d == 9 else torch.cat((z, f[..., :-1]), -1)

    def network(self, f, W1, W2):
        T = [self.transport(f, d) for d in range(11)]
        phi = [sum(self.spin(W1[d, a, 0], T[d]) for d in range(11)) for a in range(16)]
        return sum(self.transport(sum(self.spin(W2[d, 0, a], phi[a]) for a in range(16)), d) for d in range(11))


def _bf16(w):
    t = torch.view_as_real(torch.from_numpy(w).to(torch.complex64)).to(torch.bfloat16).to(torch.float64)
    return torch.view_as_complex(t.contiguous()).cuda()


def _complex(x):
    return torch.view_as_complex(x.to(torch.float64).contiguous())


def exact(case, seed):
    c, op, dag = case, case["op"], case["dagger"]
    V = sum(_shapes(c))
    if op == "solve" and V * c["Ls"] * c["nrhs"] > 16 ** 4 * 12:
        return None
    U = _links(c, seed)
    x = [_complex(v) for v in _inputs(c, seed)]
    doms = [_Lattice(c, U, b) for b in _boxes(c) or [((0, 0, 0, 0), _dims(c))]]
    n0 = _shapes(c)[0]
    if op == "force":
        D = doms[0]
        f = [D.put(v[n0:], 1, D.put(v[:n0], 0)) for v in x]
        return [torch.view_as_real(D.force(*f))]
    if op == "nn_apply":
        W = [_bf16(w) for w in _weights(seed)]
        D = doms[0]
        return [torch.view_as_real(D.get(D.network(D.put(x[0], 1), *W), 1))]
    if op == "nn_train":
        W = [_bf16(w).requires_grad_(True) for w in _weights(seed)]
        D = doms[0]
        r = D.put(x[0], 1)
        z = D.network(r, *W)
        z = D.put(D.get(z, 1), 1)
        diff = (D.normal(z) - r).abs().square().sum((0, 1, 2, 3, 4, 5, 7))
        loss = (diff / r.abs().square().sum((0, 1, 2, 3, 4, 5, 7))).mean()
        loss.backward()
        return {"loss": loss.detach().cpu(), "g1": W[0].grad.cpu().numpy(), "g2": W[1].grad.cpu().numpy()}
    res = [[], []]
    at = [0, 0]
    for D in doms:
        n = [len(i) for i in D.idx]
        cut = [slice(at[p], at[p] + n[p]) for p in range(2)]
        at = [at[p] + n[p] for p in range(2)]
        if op in ("dslash", "normal", "filter"):
            f = D.put(x[0][cut[1]], 1)
            if op == "dslash":
                g = D.B(D.hop(f, True), True) if dag else D.hop(D.B(f))
                res[0].append(D.get(-0.5 * g, 0))
            elif op == "normal":
                g = D.mpc(f, dag)
                res[0].append(D.get(g, 1))
                # the second call's input is the first one's output as stored
                g = D.put(_complex(torch.view_as_real(D.get(g, 1)).to(REAL[c["prec"]])), 1)
                res[1].append(D.get(D.mpc(g, not dag), 1))
            else:
                lo, hi = _top(c) / 50, _top(c)

                def zA(w):
                    return ((hi + lo) * w - 2 * D.normal(w)) / (hi - lo)

                prev, w = f, zA(f)
                for _ in range(c["order"] - 1):
                    prev, w = w, 2 * zA(w) - prev
                res[0].append(D.get(w, 1))
        else:
            f = D.put(x[0][:n0][cut[0]], 0)
            f = D.put(x[0][n0:][cut[1]], 1, f)
            g = D.solve(f) if op == "solve" else D.D(f, dag)
            res[0].append(D.get(g, 0))
            res[1].append(D.get(g, 1))
    if op in ("apply_d", "solve"):
        return [torch.view_as_real(torch.cat(res[0] + res[1]))]
    return [torch.view_as_real(torch.cat(v)) for v in res if v]
