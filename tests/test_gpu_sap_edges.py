"""The Schwarz block kernels (full and even-odd reduced) at the edges of its block sizes: blocks
smaller than a warp, not a multiple of a warp, extents of one site (neighbours
outside on both sides), the largest block; an output buffer that holds NaN
(the first cycle must not read it); no MR step at all."""
import numpy as np
import pytest

from oracle import solvers
from paper_2202_07388_gb300 import synth
from tests.gpu_cases import oracle_case, make_handle, to_dev, from_dev, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bs,ncy,nmr", [((4, 4, 6, 8), (1, 2, 3, 2), 2, 3),
                                             ((4, 2, 4, 8), (2, 1, 1, 4), 1, 4),
                                             ((4, 12, 4, 8), (2, 6, 2, 4), 2, 2),
                                             ((8, 8, 4, 16), (4, 4, 2, 8), 1, 3),
                                             ((8, 8, 8, 8), (4, 4, 4, 4), 1, 0)])
@pytest.mark.parametrize("link_fmt", [0, 1])
def test_block_shapes(dims, bs, ncy, nmr, link_fmt):
    import torch
    from paper_2202_07388_gb300 import oq
    u, a, _ = oracle_case(dims, 0.5, 931, 0.1365, 1.0)
    rho = synth.make_source(dims, 932)
    ref = solvers.sap(u, a, rho, bs, ncy, nmr)
    h = make_handle(dims, u, 0.1365, 1.0, link_fmt)
    prho, pphi = h.new_packed(oq.F32), h.new_packed(oq.F32)
    pphi.view(torch.float32).fill_(float("nan"))
    h.pack(to_dev(rho), prho, oq.F32)
    h.sap_apply(prho, pphi, oq.SolverParams(ncy=ncy, nmr=nmr, bs=bs))
    out = to_dev(np.zeros_like(rho))
    h.unpack(pphi, out, oq.F32)
    got = from_dev(out, rho.shape)
    if nmr == 0:
        assert not got.any()
    else:
        assert rel_err(got, ref) < 1e-5
    h.close()


@pytest.mark.parametrize("dims,bs,ncy,nmr", [((4, 4, 6, 8), (1, 2, 3, 2), 2, 3),
                                             ((4, 2, 4, 8), (2, 1, 1, 4), 1, 4),
                                             ((4, 12, 4, 8), (2, 6, 2, 4), 2, 2),
                                             ((8, 8, 4, 16), (4, 4, 2, 8), 1, 3),
                                             ((8, 8, 8, 8), (4, 4, 4, 4), 2, 0)])
@pytest.mark.parametrize("link_fmt", [0, 1])
def test_even_odd_block_shapes(dims, bs, ncy, nmr, link_fmt):
    import torch
    from paper_2202_07388_gb300 import oq
    u, a, ainv = oracle_case(dims, 0.5, 933, 0.1365, 1.0)
    rho = synth.make_source(dims, 934)
    ref = solvers.sap(u, a, rho, bs, ncy, nmr, eo=True, ainv=ainv)
    h = make_handle(dims, u, 0.1365, 1.0, link_fmt)
    prho, pphi = h.new_packed(oq.F32), h.new_packed(oq.F32)
    pphi.view(torch.float32).fill_(float("nan"))
    h.pack(to_dev(rho), prho, oq.F32)
    h.sap_apply(prho, pphi, oq.SolverParams(ncy=ncy, nmr=nmr, bs=bs, sap_eo=1))
    out = to_dev(np.zeros_like(rho))
    h.unpack(pphi, out, oq.F32)
    assert rel_err(from_dev(out, rho.shape), ref) < 1e-5
    h.close()


@pytest.mark.parametrize("dims,bs,ncy,nmr", [((4, 4, 6, 8), (1, 2, 3, 2), 2, 3),
                                             ((4, 12, 4, 8), (2, 6, 2, 4), 2, 2),
                                             ((8, 8, 8, 8), (4, 4, 4, 4), 1, 4)])
@pytest.mark.parametrize("link_fmt", [0, 1])
@pytest.mark.parametrize("eo", [0, 1])
def test_block_ordered_operands(dims, bs, ncy, nmr, link_fmt, eo):
    """The solver's SAP reads block-ordered links and clover.  One Krylov vector:
    psi = phi <D phi, eta> / <D phi, D phi> with phi = SAP eta.  The binary32
    errors of phi and D phi enter psi, the latter through the coefficient: the
    bound of the single application above, doubled.  A second solve with another
    right-hand side finds the same operands."""
    import torch
    from oracle import dirac
    from paper_2202_07388_gb300 import oq
    u, a, ainv = oracle_case(dims, 0.5, 935, 0.1365, 1.0)
    h = make_handle(dims, u, 0.1365, 1.0, link_fmt)
    for seed in (936, 937):
        eta = synth.make_source(dims, seed)
        phi = solvers.sap(u, a, eta, bs, ncy, nmr, eo=bool(eo), ainv=ainv)
        chi = dirac.dw(u, a, phi, -1.0)
        ref = phi * (np.vdot(chi, eta) / np.vdot(chi, chi))
        psi = to_dev(np.zeros_like(eta))
        h.sap_gcr(to_dev(eta), psi, oq.SolverParams(nkv=1, nmx=1, res=1e-12, ncy=ncy, nmr=nmr, bs=bs, sap_eo=eo,
                                                    sdtype=oq.F32))
        assert rel_err(from_dev(psi, eta.shape), ref) < 2e-5
    h.close()


def test_solution_update_from_zero_components():
    """A point source: phi is exactly zero away from it, and the update of the
    binary64 solution must leave those components zero."""
    from oracle import dirac
    from paper_2202_07388_gb300 import oq
    dims, bs = (8, 8, 8, 8), (4, 4, 4, 4)
    u, a, ainv = oracle_case(dims, 0.5, 938, 0.1365, 1.0)
    h = make_handle(dims, u, 0.1365, 1.0, 1)
    eta = np.zeros_like(synth.make_source(dims, 939))
    eta[0, 0, 0, 0, 0, 0] = 1.0
    phi = solvers.sap(u, a, eta, bs, 1, 1)
    chi = dirac.dw(u, a, phi, -1.0)
    ref = phi * (np.vdot(chi, eta) / np.vdot(chi, chi))
    psi = to_dev(np.zeros_like(eta))
    h.sap_gcr(to_dev(eta), psi, oq.SolverParams(nkv=1, nmx=1, res=1e-12, ncy=1, nmr=1, bs=bs, sdtype=oq.F32))
    got = from_dev(psi, eta.shape)
    far = ref == 0
    assert far.sum() > ref.size // 2 and not got[far].any()
    assert rel_err(got, ref) < 2e-5  # as test_block_ordered_operands
    h.close()
