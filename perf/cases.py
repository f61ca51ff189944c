"""The work that programs have this library do, as cases to time and to compare.

Every case goes through the public binding (``paper_2202_07388_gb300.oq``):
operator applications on packed fields, the solvers on canonical fields, the
Schwarz preconditioner, the learned preconditioner forward and backward, and
the set-up of a new gauge field.  Sizes are those of the library's own
workloads (8^4, 32x16^3, 48x24^3, 64x32^3 and ragged test lattices).

``exact`` restates each path in binary64 with plain torch: the Wilson-clover
operator in the chiral basis, its even-odd Schur form, conjugate gradients,
the multiplicative Schwarz procedure with minimal-residual block steps and
the parallel-transport layers.
"""
import numpy as np
import torch

from paper_2202_07388_gb300 import oq

PREC = {"f64": oq.F64, "f32": oq.F32, "bf16": oq.BF16, "f16": oq.F16, "df64": oq.DF64}
ROUND = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16,
         "df64": torch.float64}
VIEW = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16,
        "df64": torch.float32}
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2, "df64": 8}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest lattice of the library's own tests and batches: one
        # operator application, where launches and latency count
        dict(name="dhat_f32_8c", op="dhat", dims="8x8x8x8", prec="f32", nrhs=1, dagger=False, tuned=False,
             kappa=0.135, eps=0.5),
        # ragged extents in binary64, the adjoint, two right-hand sides: the
        # operator of the residual checks and of plain binary64 solvers
        dict(name="dw_f64_ragged_dag", op="dw", dims="24x12x10x14", prec="f64", nrhs=2, dagger=True, tuned=False,
             kappa=0.135, eps=0.5),
        # the double-float operator of the reset steps
        dict(name="dhat_df64_32x16c_4rhs", op="dhat", dims="32x16x16x16", prec="df64", nrhs=4, dagger=False,
             tuned=False, kappa=0.135, eps=0.5),
        # the largest operator application: 12 spin-colour sources on 64x32^3
        dict(name="dhat_f16_64x32c_12rhs", op="dhat", dims="64x32x32x32", prec="f16", nrhs=12, dagger=False,
             tuned=False, kappa=0.135, eps=0.6),
        # one propagator source, binary32 storage: the everyday solve
        dict(name="cgne_f32_32x16c", op="cgne", dims="32x16x16x16", prec="f32", nrhs=1, tuned=False,
             kappa=0.135, eps=0.5),
        # all 12 sources of a propagator, binary16 storage, launches chosen by
        # the autotuner once per handle: the production solve
        dict(name="cgne_f16_48x24c_12rhs", op="cgne", dims="48x24x24x24", prec="f16", nrhs=12, tuned=True,
             kappa=0.135, eps=0.5),
        # an uneven batch of charged QCD+QED systems solved together
        dict(name="batch_f16_uneven", op="batch", dims="32x16x16x16", small="8x8x8x8", prec="f16",
             kappa=0.135, eps=0.5),
        # Schwarz-preconditioned GCR on the full system, near the critical kappa
        dict(name="sap_gcr_48x24c", op="gcr", dims="48x24x24x24", ncy=4, nmr=5, nkv=16, bs="4x4x4x4", eo=False,
             kappa=0.1365, eps=0.5),
        # the Schwarz preconditioner alone, even-odd reduced blocks
        dict(name="sap_eo_24x16c", op="sap", dims="24x16x16x16", ncy=2, nmr=4, bs="4x4x4x4", eo=True,
             kappa=0.135, eps=0.5),
        # the learned preconditioner: forward
        dict(name="ptc_48x24c", op="ptc", dims="48x24x24x24", kappa=0.1365, eps=0.5),
        # and one training gradient over a mini-batch of pairs
        dict(name="ptc_grad_32x16c", op="ptcgrad", dims="32x16x16x16", pairs=4, kappa=0.1365, eps=0.5),
        # a new gauge field: upload, clover term, and a first application to
        # canonical fields with its norm (what follows every gauge update)
        dict(name="setup_32c", op="setup", dims="32x32x32x32", prec="f32", nrhs=2, kappa=0.135, eps=0.6),
    ]


def _draw_dims(rng, lo, hi, step=2, least=4):
    """Four extents, multiples of `step`, with a volume between lo and hi (spread over its logarithm)."""
    vol = lo * (hi / lo) ** rng.random()
    side = vol ** 0.25
    while True:
        d = []
        for _ in range(4):
            e = side * 2.0 ** rng.uniform(-0.7, 0.7)
            d.append(max(least, int(round(e / step)) * step))
        v = d[0] * d[1] * d[2] * d[3]
        if lo * 0.6 <= v <= hi:
            return "x".join(str(x) for x in d)


def draw(rng):
    op = rng.choice(["dhat", "dhat", "dw", "cgne", "cgne", "batch", "gcr", "sap", "ptc", "ptcgrad", "setup"])
    kappa = round(rng.uniform(0.125, 0.1355), 4)
    eps = round(rng.uniform(0.3, 0.6), 2)
    c = dict(op=op, kappa=kappa, eps=eps)
    if op in ("dhat", "dw"):
        c.update(prec=rng.choice(["f64", "f32", "bf16", "f16", "df64"]), nrhs=rng.choice([1, 1, 2, 3, 4, 5, 8, 12]),
                 dagger=rng.random() < 0.5, tuned=rng.random() < 0.25)
        cost = {"f64": 8, "df64": 4}.get(c["prec"], 1) * c["nrhs"]
        c["dims"] = _draw_dims(rng, 8 ** 4, min(64 * 32 ** 3, 16e6 / cost))
    elif op == "cgne":
        c.update(prec=rng.choice(["f64", "f32", "bf16", "f16", "f16"]), nrhs=rng.choice([1, 1, 2, 3, 6, 12]),
                 tuned=rng.random() < 0.25)
        c["dims"] = _draw_dims(rng, 8 ** 4, (2e6 if c["prec"] != "f64" else 3e5) / c["nrhs"])
    elif op == "batch":
        c.update(prec=rng.choice(["f32", "bf16", "f16"]), dims=_draw_dims(rng, 16 ** 4, 32 * 16 ** 3),
                 small=_draw_dims(rng, 4 ** 4 * 2, 10 ** 4))
    elif op in ("gcr", "sap"):
        bs = rng.choice([(4, 4, 4, 4), (4, 4, 4, 4), (2, 4, 4, 4), (2, 2, 4, 4), (4, 2, 4, 2)])
        big = 48 * 24 ** 3 if op == "sap" else 32 * 16 ** 3
        c.update(ncy=rng.choice([1, 2, 4]), nmr=rng.choice([2, 3, 4, 5]), eo=rng.random() < 0.3,
                 bs="x".join(str(b) for b in bs))
        if op == "gcr":
            c.update(nkv=rng.choice([8, 16, 24]), ncy=rng.choice([0, 2, 4]))
        c["dims"] = _draw_dims(rng, 8 ** 4, big, step=8, least=8)
    elif op == "ptc":
        c["dims"] = _draw_dims(rng, 8 ** 4, 48 * 24 ** 3)
    elif op == "ptcgrad":
        c.update(dims=_draw_dims(rng, 8 ** 4, 32 * 16 ** 3), pairs=rng.choice([1, 2, 3, 4]))
    else:
        c.update(prec=rng.choice(["f64", "f32", "f16"]), nrhs=rng.choice([1, 2, 3]),
                 dims=_draw_dims(rng, 8 ** 4, 32 ** 4))
    return c


# ---------------------------------------------------------------------------
# inputs (from the seed alone, made on the device)
# ---------------------------------------------------------------------------

def _dims(text):
    return tuple(int(x) for x in text.split("x"))


def _vol(text):
    d = _dims(text)
    return d[0] * d[1] * d[2] * d[3]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _gen(seed):
    return torch.Generator(device=_device()).manual_seed(1000003 * (int(seed) % 2000000011) + 17)


def _randn(gen, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=_device(), generator=gen)


def _gauge(gen, vol, eps):
    """SU(3) links (vol, 4, 3, 3): 1 + i eps H, H a traceless Hermitian Gaussian matrix, rows orthonormalised."""
    n = vol * 4
    z = torch.view_as_complex(_randn(gen, n, 3, 3, 2))
    h = 0.5 * (z + z.conj().transpose(1, 2))
    del z
    tr = (h[:, 0, 0] + h[:, 1, 1] + h[:, 2, 2]) / 3
    eye = torch.eye(3, dtype=torch.complex128, device=h.device)
    m = eye + 1j * eps * (h - tr[:, None, None] * eye)
    r0, r1 = m[:, 0], m[:, 1]
    r0 = r0 / r0.abs().square().sum(1, keepdim=True).sqrt()
    r1 = r1 - (r0.conj() * r1).sum(1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(1, keepdim=True).sqrt()
    r2 = torch.linalg.cross(r0, r1).conj()
    return torch.stack([r0, r1, r2], 1).reshape(vol, 4, 3, 3).contiguous()


def _spinors(gen, n, vol, prec="f64"):
    """n Gaussian spinor fields (n, vol, 24 reals), rounded to the storage type that they are packed in."""
    x = _randn(gen, n, vol, 24) * 0.5 ** 0.5
    return x.to(ROUND[prec]).to(torch.float64)


def _parity(dims):
    g = torch.meshgrid(*[torch.arange(d, device=_device()) for d in dims], indexing="ij")
    return ((g[0] + g[1] + g[2] + g[3]) & 1).reshape(-1)


def _batch_systems(case):
    """(dims, charge) of the systems of a batch: both lattices with both quark charges."""
    return [(case["small"], 2.0 / 3.0), (case["dims"], 2.0 / 3.0), (case["small"], -1.0 / 3.0),
            (case["dims"], -1.0 / 3.0)]


def _weights(gen):
    """Binary32 master weights of the two layers (9 paths, 2 hidden fields, complex 4x4 spin matrices)."""
    return (0.15 * _randn(gen, 2 * 2 * 9 * 2 * 16)).to(torch.float32)


def _params(case):
    if case["op"] in ("cgne", "batch"):
        return oq.SolverParams(res=1e-10, nmx=3000, sdtype=PREC[case["prec"]])
    return oq.SolverParams(res=1e-10, nmx=2000, nkv=case.get("nkv", 16), ncy=case["ncy"], nmr=case["nmr"],
                           bs=_dims(case["bs"]), sdtype=oq.F32, sap_eo=int(case["eo"]))


def _inputs(case, seed):
    """What prepare and exact share: links and canonical fields."""
    gen = _gen(seed)
    op = case["op"]
    if op == "batch":
        out = []
        for text, q in _batch_systems(case):
            vol = _vol(text)
            u = _gauge(gen, vol, case["eps"])
            a = 0.2 * _randn(gen, vol, 4)
            e = _spinors(gen, 1, vol)
            e[:, _parity(_dims(text)) == 1] = 0.0
            out.append((text, q, u, a, e))
        return out
    vol = _vol(case["dims"])
    u = _gauge(gen, vol, case["eps"])
    if op in ("dhat", "dw"):
        x = _spinors(gen, case["nrhs"], vol, case["prec"])
    elif op == "cgne":
        x = _spinors(gen, case["nrhs"], vol)[:, _parity(_dims(case["dims"])) == 0].contiguous()
    elif op == "gcr":
        x = _spinors(gen, 1, vol)
    elif op in ("sap", "ptc"):
        x = _spinors(gen, 1, vol, "f32")
    elif op == "ptcgrad":
        x = _spinors(gen, 2 * case["pairs"], vol, "f32")
    else:
        x = _spinors(gen, case["nrhs"], vol, case["prec"])
    w = _weights(gen) if op in ("ptc", "ptcgrad") else None
    return u, x, w


CSW = 1.0


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        sys = _inputs(case, seed)
        h = oq.Handle([_dims(t) for t, _, _, _, _ in sys])
        etas, psis = [], []
        for lat, (_, q, u, a, e) in enumerate(sys):
            h.gauge_upload_qed(u, a, q, lat=lat)
            h.clover_build(case["kappa"], CSW, lat=lat)
            etas.append(e)
            psis.append(torch.zeros_like(e))
        return dict(op=op, h=h, etas=etas, psis=psis, prm=_params(case))
    u, x, w = _inputs(case, seed)
    h = oq.Handle(_dims(case["dims"]))
    s = dict(op=op, h=h, kappa=case["kappa"])
    if op == "setup":
        n = case["nrhs"]
        s.update(u=u, x=x, n=n, prec=PREC[case["prec"]], a=h.new_packed(PREC[case["prec"]], nrhs=n),
                 b=h.new_packed(PREC[case["prec"]], nrhs=n), y=torch.zeros_like(x))
        return s
    h.gauge_upload(u, oq.LINK_12)
    h.clover_build(case["kappa"], CSW)
    if op in ("dhat", "dw"):
        p, sub, n = PREC[case["prec"]], oq.EVEN if op == "dhat" else oq.FULL, case["nrhs"]
        if case["tuned"]:
            h.autotune(p, nrhs=n)
        a = h.new_packed(p, sub, nrhs=n)
        h.pack(x, a, p, sub, nrhs=n)
        s.update(prec=p, n=n, dagger=case["dagger"], a=a, b=h.new_packed(p, sub, nrhs=n), view=VIEW[case["prec"]])
    elif op == "cgne":
        if case["tuned"]:
            h.autotune(PREC[case["prec"]], nrhs=case["nrhs"])
        s.update(n=case["nrhs"], eta=x, psi=torch.zeros_like(x), prm=_params(case))
    elif op == "gcr":
        s.update(eta=x, psi=torch.zeros_like(x), prm=_params(case))
    elif op == "sap":
        a = h.new_packed(oq.F32)
        h.pack(x, a, oq.F32)
        s.update(a=a, b=h.new_packed(oq.F32), prm=_params(case))
    elif op == "ptc":
        a = h.new_packed(oq.F32)
        h.pack(x, a, oq.F32)
        s.update(a=a, b=h.new_packed(oq.F32), w=w)
    else:
        k = case["pairs"]
        a, b = h.new_packed(oq.F32, nrhs=k), h.new_packed(oq.F32, nrhs=k)
        h.pack(x[:k].contiguous(), a, oq.F32, nrhs=k)
        h.pack(x[k:].contiguous(), b, oq.F32, nrhs=k)
        s.update(a=a, b=b, w=w, k=k, g=torch.zeros(w.numel(), dtype=torch.float64, device=w.device))
    return s


def run(s):
    op, h = s["op"], s["h"]
    if op == "dhat":
        h.dw_hat(s["a"], s["b"], s["prec"], nrhs=s["n"], dagger=s["dagger"])
        return s["b"].view(s["view"])
    if op == "dw":
        h.dw(s["a"], s["b"], s["prec"], nrhs=s["n"], dagger=s["dagger"])
        return s["b"].view(s["view"])
    if op == "cgne":
        h.cgne_even(s["eta"], s["psi"], s["prm"], nrhs=s["n"])
        return s["psi"]
    if op == "batch":
        h.cgne_batch(list(range(len(s["etas"]))), s["etas"], s["psis"], s["prm"])
        return s["psis"]
    if op == "gcr":
        h.sap_gcr(s["eta"], s["psi"], s["prm"])
        return s["psi"]
    if op == "sap":
        h.sap_apply(s["a"], s["b"], s["prm"])
        return s["b"].view(torch.float32)
    if op == "ptc":
        h.nnprec_apply(s["w"], s["a"], s["b"])
        return s["b"].view(torch.float32)
    if op == "ptcgrad":
        loss = h.nnprec_grad(s["w"], s["a"], s["b"], s["k"], s["g"])
        return dict(grad=s["g"], loss=loss)
    h.gauge_upload(s["u"], oq.LINK_12)
    h.clover_build(s["kappa"], CSW)
    h.pack(s["x"], s["a"], s["prec"], nrhs=s["n"])
    h.dw(s["a"], s["b"], s["prec"], nrhs=s["n"])
    norms = h.norm2(s["b"], s["prec"], nrhs=s["n"])
    h.unpack(s["b"], s["y"], s["prec"], nrhs=s["n"])
    return dict(y=s["y"], norms=norms)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _operator_work(vol, prec, nrhs, full):
    """One Dhat (full: one Dw): links (12 reals for the binary32-arithmetic types), clover and fields once."""
    wide = prec in ("f64", "df64")
    fixed = vol * ((4 * 18 + 72) * 8 if wide else (4 * 12 + 72) * 4)
    sites = vol if full else vol / 2
    byts = fixed + nrhs * sites * 48 * BYTES[prec]
    return byts, 1824.0 * vol * nrhs


def _cgne_work(vol, prec, nrhs, steps=40):
    """steps applications of Dhat^dag Dhat in the storage type with the vector updates, one binary64 residual."""
    b1, f1 = _operator_work(vol, prec, nrhs, False)
    b2, f2 = _operator_work(vol, "f64", nrhs, False)
    vec = nrhs * vol / 2 * 24 * (4 * BYTES[prec] + 2 * max(4, BYTES[prec] if prec == "f64" else 4))
    return steps * (2 * b1 + vec) + 2 * b2 + nrhs * vol / 2 * 24 * 8 * 2, steps * 2 * f1 + 2 * f2


def work(case):
    op = case["op"]
    vol = _vol(case["dims"])
    if op in ("dhat", "dw"):
        b, f = _operator_work(vol, case["prec"], case["nrhs"], op == "dw")
    elif op == "cgne":
        b, f = _cgne_work(vol, case["prec"], case["nrhs"])
    elif op == "batch":
        w = [_cgne_work(_vol(t), case["prec"], 1) for t, _ in _batch_systems(case)]
        b, f = sum(x[0] for x in w), sum(x[1] for x in w)
    elif op in ("gcr", "sap"):
        # a Schwarz cycle: rho and phi, links and clover once; a full and nmr block operators
        cb, cf = vol * (3 * 96 + 480), 1824.0 * vol * (1 + case["nmr"])
        if op == "sap":
            b, f = case["ncy"] * cb, case["ncy"] * cf
        else:
            steps = 18 if case["ncy"] else 67
            ob, of = _operator_work(vol, "f32", 1, True)
            b = steps * (case["ncy"] * cb + ob + vol * 96 * (case["nkv"] + 4)) + 2 * vol * 192
            f = steps * (case["ncy"] * cf + of + vol * 192 * case["nkv"])
    elif op == "ptc":
        b, f = vol * (2 * 96 + 192 + 2 * 192), vol * 2 * (8 * 264 * 1.5 + 9 * 2 * 384)
    elif op == "ptcgrad":
        k = case["pairs"]
        b, f = k * vol * (4 * 192 + 8 * 96), k * 2.5 * vol * 2 * (8 * 264 * 1.5 + 9 * 2 * 384)
    else:
        ob, of = _operator_work(vol, case["prec"], case["nrhs"], True)
        # links in (binary64) and out (binary64, binary32 of 12 and 18 reals); A and its inverse in both types
        b = vol * (576 * 2 + 192 + 288 + 2 * 72 * 12) + ob + case["nrhs"] * vol * 24 * (16 + 2 * BYTES[case["prec"]])
        f = of + vol * (6 * 10 * 216 + 2 * 1000)
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    op = case["op"]
    if op in ("dhat", "dw"):
        # sums in another order: one rounding of the arithmetic type per
        # value, and for the 16-bit types results that round the other way
        return {"rel": {"f64": 2e-15, "df64": 4e-13, "f32": 5e-7, "bf16": 3e-3, "f16": 4e-4}[case["prec"]],
                "max": {"f64": 1e-12, "df64": 1e-6, "f32": 1e-5, "bf16": 5e-2, "f16": 1e-2}[case["prec"]]}
    if op in ("cgne", "batch", "gcr"):
        # solutions of residual 1e-10: off by that times the condition number
        return {"rel": 1e-8, "max": 1e-6}
    if op == "sap":
        return {"rel": 1e-6, "max": 4e-5}
    if op == "ptc":
        return {"rel": 1.2e-6, "max": 4e-5}
    if op == "ptcgrad":
        return {"rel": 4e-7, "max": 1e-5}
    return {"rel": {"f64": 4e-15, "f32": 5e-7, "f16": 6e-4}[case["prec"]],
            "max": {"f64": 1e-11, "f32": 2e-5, "f16": 1e-2}[case["prec"]]}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------

def _gamma():
    s = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
    g = np.zeros((4, 4, 4), dtype=complex)
    g[0, :2, 2:] = g[0, 2:, :2] = -np.eye(2)
    for k in range(3):
        g[k + 1, :2, 2:] = -1j * s[k]
        g[k + 1, 2:, :2] = 1j * s[k]
    return g


GAMMA = _gamma()


class _Dirac:
    """The Wilson-clover operator on one lattice: fields (dims, 4, 3) complex128, antiperiodic time."""

    def __init__(self, dims, u, kappa, csw=CSW):
        self.dims = tuple(dims)
        self.u = u.reshape(self.dims + (4, 3, 3))
        self.dev = u.device
        self.even = (_parity(self.dims) == 0).reshape(self.dims + (1, 1))
        self.site = torch.meshgrid(*[torch.arange(d, device=self.dev) for d in self.dims], indexing="ij")
        self._clover(kappa, csw)

    def shift(self, f, mu, d):
        """f(x + d mu), periodic."""
        return torch.roll(f, -d, mu)

    def fshift(self, f, mu, d):
        """The same for fermion fields: antiperiodic in time."""
        f = torch.roll(f, -d, mu)
        if mu == 0:
            f = f.clone()
            f[-1 if d > 0 else 0] *= -1
        return f

    def _clover(self, kappa, csw):
        u = self.u
        blocks = [torch.zeros(self.dims + (6, 6), dtype=torch.complex128, device=self.dev) for _ in range(2)]
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a, b = u[..., mu, :, :], u[..., nu, :, :]
                dag = lambda m: m.conj().transpose(-1, -2)  # noqa: E731
                # the plaquette at x, carried to its other three corners
                lo = torch.matmul(a, self.shift(b, mu, 1))
                hi = torch.matmul(b, self.shift(a, nu, 1))
                p = torch.matmul(lo, dag(hi))
                q = p + self.shift(torch.matmul(dag(a), torch.matmul(p, a)), mu, -1)
                q = q + self.shift(torch.matmul(dag(b), torch.matmul(p, b)), nu, -1)
                q = q + self.shift(self.shift(torch.matmul(dag(hi), lo), mu, -1), nu, -1)
                f = 0.125 * (q - dag(q))
                sig = 0.5j * (GAMMA[mu] @ GAMMA[nu] - GAMMA[nu] @ GAMMA[mu])
                for c in range(2):
                    s = 0.5j * csw * torch.from_numpy(sig[2 * c:2 * c + 2, 2 * c:2 * c + 2]).to(self.dev)
                    blocks[c] += (s[:, None, :, None] * f[..., None, :, None, :]).reshape(self.dims + (6, 6))
        for m in blocks:
            m += torch.eye(6, dtype=torch.complex128, device=self.dev) / (2 * kappa)
        self.a = blocks
        self.ai = [torch.linalg.inv(m) for m in blocks]

    @staticmethod
    def _blocks(m, v):
        out = [torch.matmul(m[c], v[..., 2 * c:2 * c + 2, :].reshape(v.shape[:4] + (6, 1))) for c in range(2)]
        return torch.cat([o.reshape(v.shape[:4] + (2, 3)) for o in out], -2)

    def local(self, v):
        return self._blocks(self.a, v)

    def inverse_local(self, v):
        return self._blocks(self.ai, v)

    def hop(self, v, dag=False, bs=None):
        """-1/2 times the hopping sum (bs: hops that leave a block are dropped)."""
        out = torch.zeros_like(v)
        for mu in range(4):
            u = self.u[..., mu, :, :]
            g = GAMMA[mu]
            perm = [int(np.nonzero(g[s])[0][0]) for s in range(4)]
            ph = torch.tensor([g[s, perm[s]] for s in range(4)], dtype=torch.complex128, device=self.dev)[:, None]
            for d in (1, -1):
                sgn = (-1.0 if d > 0 else 1.0) * (-1.0 if dag else 1.0)  # 1 + sgn g_mu
                h = (v + sgn * ph * v[..., perm, :])[..., :2, :]  # the lower half follows from the upper one
                if d > 0:
                    h = self.fshift(h, mu, 1)
                    t = sum(u[..., None, :, b] * h[..., :, None, b] for b in range(3))
                else:
                    t = sum(u.conj()[..., None, b, :] * h[..., :, None, b] for b in range(3))
                    t = self.fshift(t, mu, -1)
                if bs is not None:
                    edge = self.site[mu] % bs[mu] != (bs[mu] - 1 if d > 0 else 0)
                    t = t * edge[..., None, None]
                # lower components: (1 + sgn g) h = h, so low = sgn g_low,up h_up
                low = torch.stack([sgn * ph[s] * t[..., perm[s], :] for s in (2, 3)], -2)
                out[..., :2, :] -= 0.5 * t
                out[..., 2:, :] -= 0.5 * low
        return out

    def dw(self, v, dag=False):
        return self.local(v) + self.hop(v, dag)

    def dhat(self, v, dag=False):
        t = torch.where(self.even, 0, self.inverse_local(self.hop(v, dag)))
        return torch.where(self.even, self.local(v) - self.hop(t, dag), 0)

    def field(self, x):
        """canonical reals (vol, 24) -> field"""
        return torch.view_as_complex(x.reshape(self.dims + (4, 3, 2)).contiguous())

    def solve_normal(self, eta, res=1e-13, nmx=3000):
        """x with Dhat^dag Dhat x = eta (even fields): conjugate gradients, residual recomputed at the end."""
        x = torch.zeros_like(eta)
        nb = float(eta.abs().square().sum())
        for _ in range(3):
            r = eta - self.dhat(self.dhat(x), True)
            p, rr = r, float(r.abs().square().sum())
            for _ in range(nmx):
                if rr <= res * res * nb:
                    break
                q = self.dhat(self.dhat(p), True)
                al = rr / float((p.conj() * q).sum().real)
                x = x + al * p
                r = r - al * q
                new = float(r.abs().square().sum())
                p, rr = r + (new / rr) * p, new
        return x

    def solve(self, eta):
        """D x = eta through the even-odd Schur complement."""
        e = torch.where(self.even, eta, 0)
        o = torch.where(self.even, 0, self.inverse_local(torch.where(self.even, 0, eta)))
        b = e - torch.where(self.even, self.hop(o), 0)
        x = self.solve_normal(self.dhat(b, True))
        return x + o - torch.where(self.even, 0, self.inverse_local(self.hop(x)))

    # the Schwarz procedure -------------------------------------------------
    def _block_sum(self, f, bs):
        n = [d // b for d, b in zip(self.dims, bs)]
        s = f.sum((-1, -2)).reshape(n[0], bs[0], n[1], bs[1], n[2], bs[2], n[3], bs[3]).sum((1, 3, 5, 7))
        for mu in range(4):
            s = s.repeat_interleave(bs[mu], mu)
        return s[..., None, None]

    def _mr(self, apply, r, bs, nmr):
        x = torch.zeros_like(r)
        for _ in range(nmr):
            p = apply(r)
            pp = self._block_sum(p.conj() * p, bs).real
            om = torch.where(pp > 0, self._block_sum(p.conj() * r, bs) / torch.where(pp > 0, pp, 1.0), 0)
            x = x + om * r
            r = r - om * p
        return x

    def sap(self, rho, bs, ncy, nmr, eo):
        colour = sum(self.site[mu] // bs[mu] for mu in range(4)) % 2
        phi = torch.zeros_like(rho)
        for _ in range(ncy):
            for c in range(2):
                sel = (colour == c)[..., None, None]
                r = torch.where(sel, rho - self.dw(phi), 0)
                if not eo:
                    d = self._mr(lambda v: self.local(v) + self.hop(v, bs=bs), r, bs, nmr)
                else:
                    ro = torch.where(self.even, 0, r)
                    re = torch.where(self.even, r - self.hop(self.inverse_local(ro), bs=bs), 0)

                    def schur(v):
                        t = torch.where(self.even, 0, self.inverse_local(self.hop(v, bs=bs)))
                        return torch.where(self.even, self.local(v) - self.hop(t, bs=bs), 0)

                    x = self._mr(schur, re, bs, nmr)
                    d = x + torch.where(self.even, 0, self.inverse_local(ro - self.hop(x, bs=bs)))
                phi = phi + torch.where(sel, d, 0)
        return phi

    # parallel-transport layers ---------------------------------------------
    def transport(self, v, q):
        if q == 0:
            return v
        mu, fwd = (q - 1) // 2, (q - 1) % 2 == 0
        u = self.u[..., mu, :, :]
        if fwd:
            h = self.fshift(v, mu, 1)
            return sum(u[..., None, :, b] * h[..., :, None, b] for b in range(3))
        t = sum(u.conj()[..., None, b, :] * v[..., :, None, b] for b in range(3))
        return self.fshift(t, mu, -1)

    def layer(self, w, fields):
        """w[path, out, in, s, t] on the transported fields (in, dims, 4, 3)."""
        out = [0] * w.shape[1]
        for q in range(9):
            for ci, f in enumerate(fields):
                t = self.transport(f, q)
                for co in range(w.shape[1]):
                    out[co] = out[co] + sum(w[q, co, ci, :, k, None] * t[..., k, None, :] for k in range(4))
        return out


def _real(field, vol):
    return torch.view_as_real(field.contiguous()).reshape(vol, 24)


def _packed(x, dims, prec, even_only):
    """canonical (n, vol, 24) reals -> the packed layout, in the type of its view, flat."""
    par = _parity(dims)
    per = 16 // BYTES[prec]
    halves = [x[:, par == p] for p in ((0,) if even_only else (0, 1))]
    out = torch.stack([h.reshape(h.shape[0], h.shape[1], 24 // per, per).permute(0, 2, 1, 3) for h in halves], 1)
    out = out.reshape(-1)
    if prec == "df64":
        hi = out.to(torch.float32)
        return torch.stack([hi, (out - hi.double()).to(torch.float32)], -1).reshape(-1)
    return out


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        out = []
        for text, q, u, a, e in _inputs(case, seed):
            u = u * torch.exp(1j * q * a)[..., None, None]
            d = _Dirac(_dims(text), u, case["kappa"])
            out.append(_real(d.solve_normal(d.field(e[0])), _vol(text))[None])
        return out
    dims, vol = _dims(case["dims"]), _vol(case["dims"])
    if op == "cgne" and vol * case["nrhs"] > 600000:
        return None  # over 20 seconds
    u, x, w = _inputs(case, seed)
    d = _Dirac(dims, u, case["kappa"])
    if op in ("dhat", "dw"):
        f = d.dhat if op == "dhat" else d.dw
        x = x if op == "dw" else x * (_parity(dims) == 0)[:, None]
        y = torch.stack([_real(f(d.field(v), case["dagger"]), vol) for v in x])
        return _packed(y, dims, case["prec"], op == "dhat")
    if op == "cgne":
        even = _parity(dims) == 0
        out = torch.empty_like(x)
        for k in range(x.shape[0]):
            full = torch.zeros(vol, 24, dtype=torch.float64, device=x.device)
            full[even] = x[k]
            out[k] = _real(d.solve_normal(d.field(full)), vol)[even]
        return out
    if op == "gcr":
        return _real(d.solve(d.field(x[0])), vol)[None]
    if op == "sap":
        y = d.sap(d.field(x[0]), _dims(case["bs"]), case["ncy"], case["nmr"], case["eo"])
        return _packed(_real(y, vol)[None], dims, "f32", False)
    if op in ("ptc", "ptcgrad"):
        wc = torch.view_as_complex(w.to(torch.bfloat16).to(torch.float64).reshape(-1, 2))
        n1 = wc.numel() // 2
        w1, w2 = wc[:n1].reshape(9, 2, 1, 4, 4), wc[n1:].reshape(9, 1, 2, 4, 4)
        if op == "ptc":
            y = d.layer(w2, d.layer(w1, [d.field(x[0])]))[0]
            return _packed(_real(y, vol)[None], dims, "f32", False)
        w1, w2 = w1.clone().requires_grad_(True), w2.clone().requires_grad_(True)
        k, loss = case["pairs"], 0.0
        for j in range(k):
            e = d.field(x[k + j])
            y = d.layer(w2, d.layer(w1, [d.field(x[j])]))[0]
            part = (y - e).abs().square().sum() / e.abs().square().sum() / k
            part.backward()
            loss += float(part.detach())
        g = torch.cat([w1.grad.reshape(-1), w2.grad.reshape(-1)])
        return dict(grad=torch.view_as_real(g).reshape(-1), loss=loss)
    y = torch.stack([_real(d.dw(d.field(v)), vol) for v in x])
    return dict(y=y, norms=y.square().sum((1, 2)).cpu().numpy())
