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


@pytest.mark.parametrize("prec", [1, 2, 3])
def test_reported_launch_comes_back(prec):
    """oq_tune_set with what oq_tune_get reported gives the tuner's launch: the same bits."""
    import torch
    from paper_2202_07388_gb300 import oq, synth
    from tests.gpu_cases import to_dev
    dims = (4, 6, 10, 6)
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(synth.make_gauge(dims, 0.5, 943)), 1)
    h.clover_build(0.13, 1.0)
    x = torch.randn(1, 4 * 6 * 10 * 6, 24, dtype=torch.float64, device="cuda")
    a, b, c = (h.new_packed(prec) for _ in range(3))
    h.pack(x, a, prec)
    h.autotune(prec, 1)
    h.dw(a, b, prec)
    bx, by, _, fmt, nr, cap = h.tune_get(prec, 0, 1)
    h.tune_set(prec, 0, 1, bx, by, nr=nr, regcap=cap, link_fmt=oq.LINK_12 if fmt == "12-real" else oq.LINK_18)
    h.dw(a, c, prec)
    assert torch.equal(b, c)
    h.close()
