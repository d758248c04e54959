"""The work this library does for its users, as cases that can be timed and checked.

A case is one call (or the two or three calls that always go together) of the public binding on
inputs of the kind the paper's method meets: smeared random SU(3) links close to the critical mass,
Gaussian or point sources, block subspaces of smooth fields.  The functions of the second half
restate every path in plain torch, in 64 bits, from the definitions alone.
"""
import math

import torch

from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

PREC = {"f64": dw.DW_F64, "f32": dw.DW_F32, "f64x": dw.DW_F64X}
CSW = 1.0


def _case(name, kind, L, **more):
    c = dict(kind=kind, L0=L[0], L1=L[1], L2=L[2], L3=L[3], m0=0.0, sap="4444", dfl="4444", antiperiodic=True,
             prec="f32", nrhs=1, Ns=0, ncy=4, nmr=4, steps=0, tol=0.0)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one D on the lattice of the smoke test: a user's first call, launch latency
        _case("apply_f32_8x8c3", "apply", (8, 8, 8, 8), m0=-0.2),
        # one D in FP32 on the benchmark lattice: twice per GCR step of every mixed solve
        _case("apply_f32_48x24c3", "apply", (48, 24, 24, 24)),
        # D on the 12 spin-colour components of a propagator: twice per step of the batched solve
        _case("apply_f32_12rhs_32x16c3", "apply", (32, 16, 16, 16), nrhs=12),
        # D on FP64 fields in double-float arithmetic: every restart residual; unequal extents
        _case("apply_f64x_40x24x16x24", "apply", (40, 24, 16, 24), prec="f64x"),
        # even-odd operator in FP64: the whole work of EO+BiCGstab and the plain comparison path
        _case("schur_f64_32x16c3", "schur", (32, 16, 16, 16), prec="f64"),
        # the Schwarz preconditioner with the solver's parameters: once per GCR step
        _case("sap_f32_48x24c3", "sap", (48, 24, 24, 24)),
        # three steps of the inverse iteration on the 20 start fields: the subspace generation
        _case("invit_20_24x16c3", "invit", (24, 16, 16, 16), nrhs=20, steps=3),
        # restriction to and prolongation from the 20-field BF16 subspace: once each per GCR step
        _case("project_f32_40x24x16x24", "project", (40, 24, 16, 24), Ns=20),
        # one little solve as inside a GCR step
        _case("little_f32_32x24c3", "little", (32, 24, 24, 24), Ns=20, tol=1e-6),
        # the benchmark: one quark propagator component to 1e-10 by deflated SAP-GCR
        _case("solve_f32_48x24c3", "solve", (48, 24, 24, 24), Ns=20, steps=11, tol=1e-10),
        # a whole point-to-all propagator: the 12 point sources as one lockstep batch
        _case("solve12_f32_24x16c3", "solve", (24, 16, 16, 16), Ns=20, steps=11, nrhs=12, tol=1e-10),
        # one training step of the learned subspace generation: loss and gradient on 8 fields, Adam
        _case("ptnet_train_8_16x8c3", "train", (16, 8, 8, 8), nrhs=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, unit, lo, hi):
    """Extents (multiples of unit) whose volume is spread over [lo, hi] on a logarithmic scale."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = None
    for _ in range(200):
        L = tuple(u * rng.randint(1, max(1, 48 // u)) for u in unit)
        off = abs(math.log(synth.volume(L) / target)) + 0.3 * math.log(max(L) / min(L))
        if best is None or off < best[0]:
            best = (off, L)
    return best[1]


def draw(rng):
    kind = rng.choice(["apply", "apply", "schur", "sap", "invit", "project", "little", "solve", "solve", "train"])
    sap = rng.choice(["4444", "4444", "4444", "2244", "4422", "2444"])
    unit = [2 * int(b) for b in sap]
    hi = {"apply": 400000, "schur": 150000, "sap": 400000, "invit": 100000, "project": 300000, "little": 300000,
          "solve": 200000, "train": 10000}[kind]
    more = {"m0": round(rng.uniform(0.0, 0.1), 4), "antiperiodic": rng.random() < 0.8}
    if kind == "apply":
        more["prec"] = rng.choice(["f32", "f32", "f64", "f64x"])
        more["nrhs"] = _log_int(rng, 1, 16)
        hi //= more["nrhs"]
    elif kind == "schur":
        more["prec"] = rng.choice(["f32", "f64"])
    elif kind == "sap":
        more["nrhs"], more["ncy"], more["nmr"] = _log_int(rng, 1, 12), rng.randint(1, 6), rng.randint(3, 5)
        hi //= more["nrhs"]
    elif kind == "invit":
        more["nrhs"], more["steps"] = rng.randint(4, 24), rng.randint(1, 4)
        hi //= 4
    elif kind in ("project", "little", "solve"):
        sap = "4444"
        unit = [8, 8, 8, 8]
        more["Ns"] = rng.choice([8, 12, 16, 20, 20])
        more["prec"] = rng.choice(["f32", "f32", "f64x"]) if kind == "project" else "f32"
        more["tol"] = {"project": 0.0, "little": 1e-6, "solve": 1e-10}[kind]
        if kind == "solve":
            more["nrhs"], more["steps"] = rng.choice([1, 1, 3, 12]), rng.randint(4, 11)
            hi //= more["nrhs"]
    else:
        more["nrhs"] = rng.randint(2, 8)
    return _case(None, kind, _lattice(rng, unit, 4096, max(hi, 8192)), sap=sap, **more)


# ------------------------------------------------------------------------------------- inputs
def _L(c):
    return (c["L0"], c["L1"], c["L2"], c["L3"])


def _bs(c, key):
    return tuple(int(b) for b in c[key])


def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1) + tag)
    return g


def _links(c, seed):
    """exp(0.3 i X) with X Gaussian traceless Hermitian, five APE steps, reunitarised: complex128[V, 4, 3, 3]."""
    V = synth.volume(_L(c))
    G = torch.randn(V * 4, 3, 3, 2, generator=_gen(seed, 1), dtype=torch.float64, device="cuda")
    G = torch.view_as_complex(G) * math.sqrt(0.5)
    H = 0.15 * (G + G.conj().transpose(-1, -2))
    one = torch.eye(3, dtype=H.dtype, device="cuda")
    H = 1j * (H - torch.diagonal(H, dim1=-2, dim2=-1).sum(-1)[:, None, None] / 3.0 * one)
    U, term = one + H, H
    for k in range(2, 9):
        term = _mm(term, H) / k
        U = U + term
    W = synth.reunitarize(U).reshape(_L(c) + (4, 3, 3))
    for _ in range(5):
        new = []
        for mu in range(4):
            Um, st = W[..., mu, :, :], 0
            for nu in range(4):
                if nu == mu:
                    continue
                Un = W[..., nu, :, :]
                st = st + _mm(_mm(Un, _sh(Um, nu, 1)), _dag(_sh(Un, mu, 1)))
                st = st + _sh(_mm(_mm(_dag(Un), Um), _sh(Un, mu, 1)), nu, -1)
            new.append(synth.reunitarize(0.5 * Um + (0.5 / 6.0) * st))
        W = torch.stack(new, dim=4)
    return W.reshape(V, 4, 3, 3).contiguous()


def _noise(c, seed, tag, n):
    """n Gaussian fields, E|z|^2 = 1, complex64[n, V, 4, 3]."""
    x = torch.randn(n, synth.volume(_L(c)), 4, 3, 2, generator=_gen(seed, tag), dtype=torch.float32, device="cuda")
    return torch.view_as_complex(x * math.sqrt(0.5))


def _smooth(c, seed, n):
    """n fields of mostly low momenta (Gaussian noise over (p^2 + 0.05)^2, as a few steps of an inverse
    iteration leave it), complex128[n, V, 4, 3]: the start of a subspace that needs no more steps."""
    L = _L(c)
    p2 = torch.full((1, 1, 1, 1), 0.05, dtype=torch.float64, device="cuda")
    for mu in range(4):
        p = 2 * math.pi * torch.fft.fftfreq(L[mu], dtype=torch.float64, device="cuda")
        p2 = p2 + (2 * torch.sin(p / 2)).square().reshape([-1 if k == mu else 1 for k in range(4)])
    out = []
    for k in range(n):
        x = _noise(c, seed, 100 + k, 1)[0].to(torch.complex128).reshape(L + (4, 3))
        x = torch.fft.ifftn(torch.fft.fftn(x, dim=(0, 1, 2, 3)) / p2.square()[..., None, None], dim=(0, 1, 2, 3))
        out.append(x.reshape(-1, 4, 3) / x.abs().square().mean().sqrt())
    return torch.stack(out)


def _weights(seed, C=16):
    """Near-identity complex weights of the three network layers as one list of complex64[9, 4 cout, 4 cin]."""
    g, out = _gen(seed, 7), []
    for cin, cout in ((1, C), (C, C), (C, 1)):
        w = torch.randn(9, 4 * cout, 4 * cin, 2, generator=g, dtype=torch.float32, device="cuda")
        w = torch.view_as_complex(w) * (0.3 / math.sqrt(72 * cin))
        one = torch.eye(4, device="cuda").repeat(cout, cin) / math.sqrt(cin * cout)
        w[0] += one
        out.append(w)
    return out


def _eta(c, seed):
    """Sources of a solve, complex128[nrhs, V, 4, 3]: the 12 point sources of one site, or Gaussian noise."""
    if c["nrhs"] != 12:
        return _noise(c, seed, 2, c["nrhs"]).to(torch.complex128)
    V = synth.volume(_L(c))
    eta = torch.zeros(12, V, 12, dtype=torch.complex128, device="cuda")
    eta[torch.arange(12), (7919 * seed) % V, torch.arange(12)] = 1.0
    return eta.reshape(12, V, 4, 3)


def _fields(c, seed):
    return _noise(c, seed, 3, c["nrhs"])


def _little_vector(c, seed, prec):
    n = synth.volume(_L(c)) // synth.volume(_bs(c, "dfl")) * c["Ns"]
    x = torch.randn(n, 2, generator=_gen(seed, 5), dtype=torch.float32, device="cuda")
    return x if prec == "f32" else x.double()


def _packed_prec(c):
    return dw.DW_F32 if c["prec"] == "f32" else dw.DW_F64


def prepare(case, seed):
    c = case
    ctx = dw.dw_create(_L(c), c["m0"], CSW, _links(c, seed).cpu(), _bs(c, "sap"), c["antiperiodic"])
    s = {"c": c, "ctx": ctx}
    kind = c["kind"]
    P = _packed_prec(c)
    if kind in ("apply", "schur", "sap", "invit", "project", "train"):
        s["x"] = ctx.empty_field(P, c["nrhs"])
        dw.dw_pack(ctx, P, c["nrhs"], _fields(c, seed).to(torch.complex128), s["x"])
        s["y"] = torch.empty_like(s["x"])
    if kind in ("project", "little"):
        s["dfl"] = dw.deflation_build(ctx, _bs(c, "dfl"), c["Ns"], 0, 4, 4, _smooth(c, seed, c["Ns"]))
        s["w"] = _little_vector(c, seed, c["prec"])
        s["v"] = torch.empty_like(s["w"])
    if kind == "solve":
        start = _noise(c, seed, 4, c["Ns"]).to(torch.complex128)
        s["dfl"] = dw.deflation_build(ctx, _bs(c, "dfl"), c["Ns"], c["steps"], c["ncy"], c["nmr"], start)
        s["eta"] = _eta(c, seed)
        s["psi"] = torch.empty_like(s["eta"])
    if kind == "train":
        dw.dw_pack(ctx, P, c["nrhs"], _smooth(c, seed, c["nrhs"]), s["y"])
        s["W0"] = torch.view_as_real(torch.cat([w.reshape(-1) for w in _weights(seed)])).reshape(-1).contiguous()
        s["W"], s["m"], s["v"], s["grad"] = (torch.empty_like(s["W0"]) for _ in range(4))
    torch.cuda.synchronize()
    return s


def run(s):
    c, ctx = s["c"], s["ctx"]
    kind = c["kind"]
    if kind == "apply":
        dw.dw_apply(ctx, PREC[c["prec"]], dw.DW_OP_FULL, c["nrhs"], s["x"], s["y"])
        return s["y"]
    if kind == "schur":
        dw.dw_apply(ctx, PREC[c["prec"]], dw.DW_OP_SCHUR, c["nrhs"], s["x"], s["y"])
        return s["y"]
    if kind == "sap":
        dw.sap_precondition(ctx, PREC[c["prec"]], c["ncy"], c["nmr"], c["nrhs"], s["x"], s["y"])
        return s["y"]
    if kind == "invit":     # works in place; the start fields are kept
        s["y"].copy_(s["x"])
        dw.dfl_inverse_iteration(ctx, c["ncy"], c["nmr"], c["steps"], c["nrhs"], s["y"])
        return s["y"]
    if kind == "project":
        dw.dfl_restrict(s["dfl"], PREC[c["prec"]], s["x"], s["v"])
        dw.dfl_prolong(s["dfl"], PREC[c["prec"]], s["w"], s["y"])
        return s["v"], s["y"]
    if kind == "little":
        dw.little_dirac_solve(s["dfl"], dw.DW_F32, s["w"], s["v"], c["tol"], 2000)
        return s["v"]
    if kind == "solve":
        p = dw.sol_params(tol=c["tol"], nkv=16, ncy=c["ncy"], nmr=c["nmr"], mixed=1)
        dw.gcr_solve(ctx, s["dfl"], p, c["nrhs"], s["eta"], s["psi"])
        return s["psi"]
    # train: the first step of Adam from the same weights
    s["W"].copy_(s["W0"])
    s["m"].zero_()
    s["v"].zero_()
    loss = dw.ptnet_loss_grad(ctx, s["W"], c["nrhs"], s["x"], s["y"], s["grad"])
    dw.ptnet_adam(s["W"], s["grad"], s["m"], s["v"], 1, 3e-3)
    return loss, s["grad"], s["m"], s["v"]


def work(case):
    """Bytes: links (two rows), clover term and inverse where the path has them, fields in and out, the
    subspace and the little operator, each once.  Flops: 1320 a Wilson hop, 552 a clover term per site."""
    c = case
    V, n, kind = synth.volume(_L(c)), c["nrhs"], c["kind"]
    r = 4 if c["prec"] == "f32" else 8                       # bytes per real
    links, clover, field = 48 * r, 72 * r, 24 * r
    if kind == "apply":
        return {"bytes": V * (n * 2 * field + links + clover), "flops": V * n * 1872.0}
    if kind == "schur":
        return {"bytes": V * (n * 1.5 * field + links + clover), "flops": V * n * 1872.0}
    sap = c["ncy"] * (948 + c["nmr"] * 2052 + 948 + 1872)
    if kind == "sap":
        return {"bytes": V * (n * 2 * field + links + clover), "flops": float(V * n * sap)}
    if kind == "invit":
        return {"bytes": V * (n * 2 * field + links + clover), "flops": float(V * n * c["steps"] * sap)}
    Ns = c["Ns"]
    Nb = V // synth.volume(_bs(c, "dfl"))
    basis = Ns * 48
    if kind == "project":
        return {"bytes": V * (2 * field + basis) + Nb * Ns * 4 * r, "flops": V * 2.0 * Ns * 96}
    if kind == "little":
        return {"bytes": Nb * (8 * Ns * Ns * 8 + Ns * 16), "flops": Nb * 8.0 * Ns * Ns * 8}
    if kind == "solve":
        return {"bytes": V * (n * 384 + 192 + 384 + 576 + basis) + Nb * 8 * Ns * Ns * 24, "flops": float(V * n * sap)}
    return {"bytes": V * n * 192 + 2 * 9 * 16 * 288 * 8, "flops": V * n * 3.0 * 8 * 3 * 9 * 16 * 288}


# ------------------------------------------------------------------------------------- 64-bit restatement
def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _sh(f, mu, s, lead=0):
    """f(x + s mu), periodic; the lattice axes come after `lead` others."""
    return torch.roll(f, shifts=-s, dims=lead + mu)


class _Op:
    """The Wilson-clover operator, its Schwarz procedure and the network's transports on fields
    complex128[n, L0, L1, L2, L3, 4, 3], from their definitions."""

    def __init__(self, c, seed):
        self.c, self.L = c, _L(c)
        U = _links(c, seed).reshape(self.L + (4, 3, 3))
        dev = U.device
        x = torch.meshgrid(*[torch.arange(n, device=dev) for n in self.L], indexing="ij")
        self.x, self.odd = x, (sum(x) % 2 == 1)[None, ..., None, None]
        I2, Z2 = torch.eye(2, dtype=U.dtype, device=dev), torch.zeros(2, 2, dtype=U.dtype, device=dev)
        pauli = [torch.tensor(m, dtype=U.dtype, device=dev) for m in
                 ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
        gam = []
        for e in [-I2] + [-1j * p for p in pauli]:
            gam.append(torch.cat([torch.cat([Z2, e], 1), torch.cat([_dag(e), Z2], 1)], 0))
        self.gam = gam
        C = torch.zeros(self.L + (2, 6, 6), dtype=U.dtype, device=dev)      # chiral blocks, index 3 spin + colour
        for mu in range(4):
            for nu in range(mu + 1, 4):
                sig = 0.5j * (gam[mu] @ gam[nu] - gam[nu] @ gam[mu])
                a, b = U[..., mu, :, :], U[..., nu, :, :]
                am, bn = _sh(a, mu, -1), _sh(b, nu, -1)
                Q = _mm(_mm(a, _sh(b, mu, 1)), _mm(_dag(_sh(a, nu, 1)), _dag(b)))
                Q = Q + _mm(_mm(b, _dag(_sh(am, nu, 1))), _mm(_dag(_sh(b, mu, -1)), am))
                Q = Q + _mm(_mm(_dag(am), _dag(_sh(_sh(b, mu, -1), nu, -1))), _mm(_sh(am, nu, -1), bn))
                Q = Q + _mm(_mm(_dag(bn), _sh(a, nu, -1)), _mm(_sh(bn, mu, 1), _dag(a)))
                F = (Q - _dag(Q)) / 8
                for k in range(2):
                    sk = sig[2 * k:2 * k + 2, 2 * k:2 * k + 2]
                    C[..., k, :, :] += 0.5j * CSW * (sk[:, None, :, None] * F[..., None, :, None, :]).reshape(
                        self.L + (6, 6))
        C += (4.0 + c["m0"]) * torch.eye(6, dtype=U.dtype, device=dev)
        self.C, self._Ci = C, None
        if c["antiperiodic"]:
            U = U.clone()
            U[self.L[0] - 1, :, :, :, 0] *= -1.0
        self.U = [U[..., mu, :, :].contiguous() for mu in range(4)]

    @property
    def Ci(self):
        if self._Ci is None:
            flat = self.C.reshape(-1, 6, 6)
            self._Ci = torch.cat([torch.linalg.inv(b) for b in flat.split(1 << 17)]).reshape(self.C.shape)
        return self._Ci

    def clover(self, M, f):
        g = f.reshape(f.shape[:5] + (2, 6))
        return torch.stack([(M * one[..., None, :]).sum(-1) for one in g]).reshape(f.shape)

    def forward(self, mu, f):
        """U_mu(x) f(x + mu)"""
        f = _sh(f, mu, 1, 1)
        return sum(self.U[mu][..., None, :, b] * f[..., b, None] for b in range(3))

    def backward(self, mu, f):
        """U_mu(x - mu)^+ f(x - mu)"""
        f = sum(self.U[mu][..., None, b, :].conj() * f[..., b, None] for b in range(3))
        return _sh(f, mu, -1, 1)

    def spin(self, M, f):
        return torch.einsum("st,...tc->...sc", M, f)

    def hop(self, f):
        one, out = torch.eye(4, dtype=f.dtype, device=f.device), torch.zeros_like(f)
        for mu in range(4):
            out -= 0.5 * self.spin(one - self.gam[mu], self.forward(mu, f))
            out -= 0.5 * self.spin(one + self.gam[mu], self.backward(mu, f))
        return out

    def D(self, f):
        return self.clover(self.C, f) + self.hop(f)

    def schur(self, f):
        """A_ee - D_eo A_oo^-1 D_oe on the even part of f; zero on odd sites."""
        f = f * ~self.odd
        t = self.clover(self.Ci, self.hop(f) * self.odd)
        return self.clover(self.C, f) - self.hop(t) * ~self.odd

    def sap(self, rho):
        """Multiplicative Schwarz: per colour nmr minimal-residual steps of the blocks' even-odd operator."""
        c, bs = self.c, _bs(self.c, "sap")
        n = rho.shape[0]
        split = [n] + [v for L, b in zip(self.L, bs) for v in (L // b, b)] + [4, 3]

        def dot(a, b):
            s = (a.conj() * b).reshape(split).sum(dim=(2, 4, 6, 8, 9, 10), keepdim=True)
            return s.expand(split[:9] + [1, 1]).reshape([n] + list(self.L) + [1, 1])

        colour = (sum(x // b for x, b in zip(self.x, bs)) % 2)[None, ..., None, None]
        xi, r = torch.zeros_like(rho), rho
        for _ in range(c["ncy"]):
            for col in range(2):
                e, o = (colour == col) & ~self.odd, (colour == col) & self.odd
                bo = r * o
                re = r * e - self.hop(self.clover(self.Ci, bo)) * e
                x = torch.zeros_like(re)
                for _ in range(c["nmr"]):
                    p = self.clover(self.C, re) - self.hop(self.clover(self.Ci, self.hop(re) * o)) * e
                    pp = dot(p, p).real
                    a = torch.where(pp > 0, dot(p, re) / torch.where(pp > 0, pp, torch.ones_like(pp)), 0)
                    x, re = x + a * re, re - a * p
                delta = x + self.clover(self.Ci, bo - self.hop(x) * o)
                xi = xi + delta
                r = rho - self.D(xi)
        return xi

    def transport(self, d, h):
        return h if d == 0 else self.forward((d - 1) // 2, h) if d % 2 else self.backward((d - 1) // 2, h)

    def layer(self, w, h):
        """sum_d W_d T_d h on h[channel, L.., 4, 3]"""
        cout, cin = w.shape[1] // 4, w.shape[2] // 4
        out = 0
        for d in range(9):
            th = self.transport(d, h).movedim(-2, 1).reshape(cin * 4, -1)
            out = out + w[d] @ th
        return out.reshape((cout, 4) + self.L + (3,)).movedim(1, -2)


def _bicgstab(A, b, tol):
    """A x = b for a batch b[n, ...]; None if it does not converge."""
    def dot(u, v):
        return (u.conj() * v).flatten(1).sum(1).reshape([-1] + [1] * (b.dim() - 1))

    def ratio(p, q):
        return torch.where(q.abs() > 0, p / torch.where(q.abs() > 0, q, torch.ones_like(q)), torch.zeros_like(p))

    x, r = torch.zeros_like(b), b.clone()
    r0, p, rho, norm = r.clone(), r.clone(), dot(r, r), dot(b, b).real
    for k in range(2000):
        v = A(p)
        al = ratio(rho, dot(r0, v))
        s = r - al * v
        t = A(s)
        om = ratio(dot(t, s), dot(t, t))
        x = x + al * p + om * s
        r = s - om * t
        if k % 10 == 9 and bool((dot(r, r).real <= tol * tol * norm).all()):
            return x
        new = dot(r0, r)
        p = r + ratio(new, rho) * ratio(al, om) * (p - om * v)
        rho = new
    return None


def _order(op):
    """Canonical site of each place of the packed layout: blocks in order, even half before odd half."""
    bs, sub, key = _bs(op.c, "sap"), 0, 0
    for mu in range(4):
        key = key * (op.L[mu] // bs[mu]) + op.x[mu] // bs[mu]
        sub = sub * bs[mu] + op.x[mu] % bs[mu]
    vol = synth.volume(bs)
    return (key * vol + (sum(op.x) % 2) * (vol // 2) + sub // 2).reshape(-1).argsort()


def _pack(op, f):
    """Canonical fields -> the packed layout (16-byte units, plane by plane) as 64-bit reals."""
    n, per = f.shape[0], 2 if op.c["prec"] == "f32" else 1
    f = f.reshape(n, -1, 12)[:, _order(op)]
    f = f.reshape(n, -1, 12 // per, per).transpose(1, 2).contiguous()
    return torch.view_as_real(f).reshape(-1)


class _Subspace:
    """Block subspace (two passes of modified Gram-Schmidt per block, rounded to BF16)."""

    def __init__(self, op, fields):
        bs, Ns = _bs(op.c, "dfl"), fields.shape[0]
        key = 0
        for mu in range(4):
            key = key * (op.L[mu] // bs[mu]) + op.x[mu] // bs[mu]
        self.sites = key.reshape(-1).argsort(stable=True).reshape(-1, synth.volume(bs))
        self.V = self.sites.numel()
        v = self.cut(fields)                                    # [Nb, Ns, sites * 12]
        for k in range(Ns):
            for _ in range(2):
                for j in range(k):
                    v[:, k] -= (v[:, j].conj() * v[:, k]).sum(-1, keepdim=True) * v[:, j]
            v[:, k] /= v[:, k].abs().square().sum(-1, keepdim=True).sqrt()
        b = torch.view_as_real(v).to(torch.float32).to(torch.bfloat16).to(torch.float64)
        self.phi = torch.view_as_complex(b)

    def cut(self, f):
        n = f.shape[0]
        return f.reshape(n, self.V, 12)[:, self.sites].transpose(0, 1).reshape(len(self.sites), n, -1).contiguous()

    def restrict(self, f):
        """[n, ...] -> [n, Nb, Ns]"""
        return torch.einsum("bki,bni->nbk", self.phi.conj(), self.cut(f))

    def prolong(self, q):
        """[n, Nb, Ns] -> [n, V, 12]"""
        p = torch.einsum("bki,nbk->nbi", self.phi, q)
        out = torch.empty(q.shape[0], self.V, 12, dtype=q.dtype, device=q.device)
        out[:, self.sites] = p.reshape(q.shape[0], len(self.sites), -1, 12)
        return out


def exact(case, seed):
    c = case
    kind, V, n = c["kind"], synth.volume(_L(c)), c["nrhs"]
    # minutes of 64-bit work: solves of large systems
    if kind == "solve" and V * n > 100000 or kind == "little" and V > 150000:
        return None
    op = _Op(c, seed)
    grid = (-1,) + op.L + (4, 3)
    if kind == "solve":
        eta = _eta(c, seed).reshape(grid)
        bhat = eta - op.hop(op.clover(op.Ci, eta * op.odd))
        xe = _bicgstab(op.schur, bhat * ~op.odd, 1e-13)
        if xe is None:
            return None
        xo = op.clover(op.Ci, (eta - op.hop(xe)) * op.odd)
        return (xe + xo).reshape(n, V, 4, 3)
    if kind in ("project", "little"):
        sub = _Subspace(op, _smooth(c, seed, c["Ns"]).to(torch.complex64).to(torch.complex128))   # packed in FP32
        w = _little_vector(c, seed, c["prec"]).double()
        q = torch.view_as_complex(w).reshape(1, -1, c["Ns"])
        if kind == "project":
            x = _fields(c, seed).to(torch.complex128)
            return torch.view_as_real(sub.restrict(x).reshape(-1)), _pack(op, sub.prolong(q))
        v = _bicgstab(lambda u: sub.restrict(op.D(sub.prolong(u).reshape(grid))), q, 1e-11)
        return None if v is None else torch.view_as_real(v.reshape(-1))
    x = _fields(c, seed).to(torch.complex128).reshape(grid)
    if kind == "train":
        y = _smooth(c, seed, n).to(torch.complex64).to(torch.complex128).reshape(grid)
        W = [w.to(torch.complex128).requires_grad_() for w in _weights(seed)]
        den, total = y.abs().square().sum(), 0.0
        for one, want in zip(x, y):
            h = one[None]
            for w in W:
                h = op.layer(w, h)
            loss = (h[0] - want).abs().square().sum() / den
            loss.backward()
            total += float(loss.detach())
        g = torch.view_as_real(torch.cat([w.grad.reshape(-1) for w in W])).reshape(-1)
        return total, g, 0.1 * g, 0.001 * g * g
    out = []
    for one in x.split(1):
        if kind == "invit":
            for _ in range(c["steps"]):
                one = op.sap(one)
                one = one / one.abs().square().sum().sqrt()
            out.append(one)
        else:
            out.append({"apply": op.D, "schur": op.schur, "sap": op.sap}[kind](one))
    return _pack(op, torch.cat(out))
