"""The launch chosen without the tuner: both sides of its rules (one and several
right-hand sides, problem sizes, storage types, link formats, odd counts)
against one thread per site and right-hand side, pinned."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs", [((4, 6, 2, 8), 3), ((8, 8, 16, 16), 5), ((16, 16, 16, 16), 9),
                                       ((2, 2, 2, 2), 1), ((4, 6, 10, 6), 1), ((16, 32, 32, 18), 1)])
@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("link_fmt", [0, 1])
def test_default_against_pinned(dims, nrhs, prec, link_fmt):
    import torch
    from paper_2202_07388_gb300 import oq, synth
    from tests.gpu_cases import to_dev
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(synth.make_gauge(dims, 0.5, 941)), link_fmt)
    h.clover_build(0.13, 1.0)
    g = torch.Generator(device="cuda").manual_seed(942)
    vol = dims[0] * dims[1] * dims[2] * dims[3]
    x = torch.randn(nrhs, vol, 24, dtype=torch.float64, device="cuda", generator=g)
    a, b, c = (h.new_packed(prec, nrhs=nrhs) for _ in range(3))
    h.pack(x, a, prec, nrhs=nrhs)
    view = {1: torch.float32, 2: torch.bfloat16, 3: torch.float16}[prec]
    eps = {1: 2.0 ** -24, 2: 2.0 ** -8, 3: 2.0 ** -11}[prec]
    prm = oq.SolverParams(res=1e-9, nmx=400, sdtype=prec)
    eta = torch.randn(nrhs, vol // 2, 24, dtype=torch.float64, device="cuda", generator=g)
    sol = []
    for pinned in (False, True):
        for mode in (0, 1, 2):
            if pinned:
                h.tune_set(prec, mode, nrhs, 128, 1, nr=1)
        h.dw(a, c if pinned else b, prec, nrhs=nrhs, dagger=True)
        psi = torch.zeros_like(eta)
        rc, st = h.cgne_even(eta, psi, prm, nrhs=nrhs)
        assert rc == oq.OK and all(s["converged"] for s in st)
        sol.append(psi)
    d = (b.view(view).double() - c.view(view).double()).norm() / c.view(view).double().norm()
    # binary32 sums in another order (~50 terms), then one rounding of the storage type
    assert d < 16 * 2.0 ** -24 + (eps if prec != 1 else 0.0)
    # two solutions of residual 1e-9, condition number of Dhat^dag Dhat below 1e3
    assert (sol[0] - sol[1]).norm() / sol[1].norm() < 2e-6
    h.close()


def _operator(prec, link_fmt, nrhs, dims, pins):
    """Dw, Dhat and a short CGNE solve with `pins` (bx, by) for every mode, "tuned" or None
    (the default launch)."""
    import torch
    from paper_2202_07388_gb300 import oq, synth
    from tests.gpu_cases import to_dev
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(synth.make_gauge(dims, 0.5, 943)), link_fmt)
    h.clover_build(0.13, 1.0)
    g = torch.Generator(device="cuda").manual_seed(944)
    vol = dims[0] * dims[1] * dims[2] * dims[3]
    x = torch.randn(nrhs, vol, 24, dtype=torch.float64, device="cuda", generator=g)
    eta = torch.randn(nrhs, vol // 2, 24, dtype=torch.float64, device="cuda", generator=g)
    a, b = h.new_packed(prec, nrhs=nrhs), h.new_packed(prec, nrhs=nrhs)
    e, f = h.new_packed(prec, oq.EVEN, nrhs=nrhs), h.new_packed(prec, oq.EVEN, nrhs=nrhs)
    h.pack(x, a, prec, nrhs=nrhs)
    h.pack(x, e, prec, oq.EVEN, nrhs=nrhs)
    if pins == "tuned":
        h.autotune(prec, nrhs)
    elif pins is not None:
        for mode in (0, 1, 2):
            h.tune_set(prec, mode, nrhs, *pins)
            assert h.tune_get(prec, mode, nrhs)[:2] == pins
    h.dw(a, b, prec, nrhs=nrhs)
    h.dw_hat(e, f, prec, nrhs=nrhs)
    psi = torch.zeros_like(eta)
    rc, st = h.cgne_even(eta, psi, oq.SolverParams(res=1e-9, nmx=400, sdtype=prec), nrhs=nrhs)
    assert rc == oq.OK and all(s["converged"] for s in st)
    return h, (a, b, e, f, eta, psi)


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("link_fmt", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_one_and_two_threads_per_site_have_names(prec, link_fmt, nrhs):
    """(64, 1) is one thread per site, the arithmetic of (128, 1) in other CTAs; (64, 0) is two
    threads per site, the default for one right-hand side (its reductions in CTAs of the same
    sites): the operators and a solve have the same bits."""
    import torch
    dims = (4, 6, 10, 6)
    r = {k: _operator(prec, link_fmt, nrhs, dims, k) for k in ((64, 1), (128, 1), (64, 0), None)}
    for k in (1, 3):   # Dw, Dhat
        assert torch.equal(r[(64, 1)][1][k], r[(128, 1)][1][k])
        if nrhs == 1:
            assert torch.equal(r[(64, 0)][1][k], r[None][1][k])
    if prec == 1:   # the hops are added in another order (a 16-bit type's rounding may hide it)
        assert not torch.equal(r[(64, 0)][1][1], r[(64, 1)][1][1])
    if nrhs == 1:
        assert torch.equal(r[(64, 0)][1][5], r[None][1][5])
    for h, _ in r.values():
        h.close()


@pytest.mark.parametrize("prec,link_fmt,nrhs,dw_pair,dhat_pair", [
    (1, 1, 15, True, True), (1, 1, 16, False, False),       # F32: 2^17 site-rhs of a parity
    (3, 1, 3, True, True), (3, 1, 4, False, True),          # 16 bits, 12-real: 3 * 2^14 launched
    (2, 1, 6, False, True), (2, 1, 7, False, False),
    (3, 0, 7, True, True), (2, 0, 8, False, True),          # 18-real: 2^17 launched
    (3, 0, 15, False, True), (3, 0, 16, False, False)])
def test_default_on_both_sides_of_its_limits(prec, link_fmt, nrhs, dw_pair, dhat_pair):
    """The launch without the tuner is two threads per site below the limits and two
    right-hand sides per thread above: the bits of that launch, pinned."""
    import torch
    from paper_2202_07388_gb300 import oq, synth
    from tests.gpu_cases import to_dev
    dims = (8, 8, 16, 16)
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(synth.make_gauge(dims, 0.5, 946)), link_fmt)
    h.clover_build(0.13, 1.0)
    x = torch.randn(nrhs, 8 * 8 * 16 * 16, 24, dtype=torch.float64, device="cuda")
    a, e = h.new_packed(prec, nrhs=nrhs), h.new_packed(prec, oq.EVEN, nrhs=nrhs)
    h.pack(x, a, prec, nrhs=nrhs)
    h.pack(x, e, prec, oq.EVEN, nrhs=nrhs)
    out = {}
    for pin in (None, (64, 0, 1, 0), (64, 1, 2, 3 if prec != 1 and link_fmt == 1 else 1)):
        if pin:
            for mode in (0, 1, 2):
                h.tune_set(prec, mode, nrhs, *pin[:2], nr=pin[2], regcap=pin[3])
        b, f = torch.empty_like(a), torch.empty_like(e)
        h.dw(a, b, prec, nrhs=nrhs)
        h.dw_hat(e, f, prec, nrhs=nrhs)
        out["default" if not pin else pin[1] == 0] = b, f
    for k, pair in enumerate((dw_pair, dhat_pair)):
        assert torch.equal(out["default"][k], out[pair][k])
        assert not torch.equal(out["default"][k], out[not pair][k])
    h.close()


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_reported_launch_comes_back(prec, nrhs):
    """oq_tune_set with what oq_tune_get reported gives the tuner's launches: the same bits."""
    import torch
    from paper_2202_07388_gb300 import oq
    h, (a, b, e, f, eta, psi) = _operator(prec, 1, nrhs, (4, 6, 10, 6), "tuned")
    c, d = torch.empty_like(b), torch.empty_like(f)
    for mode in (0, 1, 2):
        bx, by, _, fmt, nr, cap = h.tune_get(prec, mode, nrhs)
        h.tune_set(prec, mode, nrhs, bx, by, nr=nr, regcap=cap,
                   link_fmt=oq.LINK_12 if fmt == "12-real" else oq.LINK_18)
    h.dw(a, c, prec, nrhs=nrhs)
    h.dw_hat(e, d, prec, nrhs=nrhs)
    assert torch.equal(b, c) and torch.equal(f, d)
    h.close()


def test_two_threads_per_site_refused_elsewhere():
    from paper_2202_07388_gb300 import oq, synth
    from tests.gpu_cases import to_dev
    dims = (4, 6, 4, 6)
    u = synth.make_gauge(dims, 0.5, 945)
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(u), oq.LINK_12)
    for kw in (dict(bx=128, by=0), dict(bx=64, by=0, nr=2), dict(bx=64, by=0, regcap=1), dict(bx=64, by=-1)):
        assert h.tune_set(oq.F32, 0, 4, check=False, **kw) == oq.ERR_ARG, kw
    for prec in (oq.F64, oq.DF64):
        assert h.tune_set(prec, 0, 1, 64, 0, check=False) == oq.ERR_ARG
    h.close()
    s = oq.Handle((2,) + dims[1:], bc_t=oq.BC_HALO)
    s.gauge_upload_halo(to_dev(u), oq.LINK_12)   # 2 slices and one beyond each face
    assert s.tune_set(oq.F32, 0, 1, 64, 0, check=False) == oq.ERR_ARG
    assert s.tune_set(oq.F32, 0, 1, 64, 1, check=False) == oq.OK
    s.close()


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((4, 6, 10, 6), 3), ((16, 16, 16, 16), 1),
                                       ((16, 16, 16, 16), 2), ((16, 16, 16, 18), 2)])
def test_default_double_float_launch(dims, nrhs):
    """OQ_DF64 without the tuner: 168 registers, or 128 where that makes one wave of the
    launch (16^4: Dw with 1, the passes of Dhat with 2 right-hand sides); the caps do not
    change a bit of the uncapped kernel's result."""
    import torch
    from paper_2202_07388_gb300 import oq, synth
    from tests.gpu_cases import to_dev
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(synth.make_gauge(dims, 0.5, 947)), oq.LINK_18)
    h.clover_build(0.13, 1.0)
    x = torch.randn(nrhs, dims[0] * dims[1] * dims[2] * dims[3], 24, dtype=torch.float64, device="cuda")
    a, e = h.new_packed(oq.DF64, nrhs=nrhs), h.new_packed(oq.DF64, oq.EVEN, nrhs=nrhs)
    h.pack(x, a, oq.DF64, nrhs=nrhs)
    h.pack(x, e, oq.DF64, oq.EVEN, nrhs=nrhs)
    out = []
    for pinned in (False, True):
        if pinned:
            for mode in (0, 1, 2):
                h.tune_set(oq.DF64, mode, nrhs, 128, 1, regcap=0)
        b, f = torch.empty_like(a), torch.empty_like(e)
        h.dw(a, b, oq.DF64, nrhs=nrhs)
        h.dw_hat(e, f, oq.DF64, nrhs=nrhs)
        out.append((b, f))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    h.close()
