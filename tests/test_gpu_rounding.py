"""The order in which the stencil adds the site's own term A in2 to the sum of its
hops: on unit links, a diagonal A (c_sw = 0) and spinors of few bits every hop and
every partial sum of hops is exact, so Dw may round only where A in2 comes in."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KAPPA = 0.135


def _field(dims, nrhs):
    """Multiples of 2^-8 in [-4, 4)."""
    g = np.random.default_rng(951)
    return g.integers(-1024, 1024, (nrhs,) + dims + (4, 3, 2)) / 256.0


def _hops(dims, psi, dagger):
    """-1/2 sum of the hops of Dw (Dw^dag) on unit links, antiperiodic in time: exact in binary64."""
    from oracle import dirac
    u = np.broadcast_to(np.eye(3), dims + (4, 3, 3)).astype(complex)
    op = dirac.dw_dagger if dagger else dirac.dw
    zero = np.zeros(dims + (12, 12), complex)
    return np.stack([op(u, zero, (p[..., 0] + 1j * p[..., 1])) for p in psi])


def _dw(dims, psi, prec, dagger, pin=None):
    from paper_2202_07388_gb300 import oq
    from tests.gpu_cases import to_dev, from_dev
    nrhs = len(psi)
    h = oq.Handle(dims)
    h.gauge_upload(to_dev(np.broadcast_to(np.eye(3), dims + (4, 3, 3)).astype(complex)), oq.LINK_12)
    h.clover_build(KAPPA, 0.0)
    if pin:
        h.tune_set(prec, 0, nrhs, *pin[:2], nr=pin[2], regcap=pin[3])
    c = psi[..., 0] + 1j * psi[..., 1]
    x, y = h.new_packed(prec, nrhs=nrhs), h.new_packed(prec, nrhs=nrhs)
    h.pack(to_dev(c), x, prec, nrhs=nrhs)
    h.dw(x, y, prec, nrhs=nrhs, dagger=dagger)
    out = to_dev(np.zeros_like(c))
    h.unpack(y, out, prec, nrhs=nrhs)
    h.close()
    return c, from_dev(out, c.shape)


@pytest.mark.parametrize("dims", [(4, 6, 2, 8), (2, 2, 2, 2)])
@pytest.mark.parametrize("dagger", [False, True])
def test_binary64_rounds_once(dims, dagger):
    """binary64: c0 x by an FMA onto the hops, one rounding."""
    psi = _field(dims, 1)
    c, got = _dw(dims, psi, 0, dagger)
    hop = _hops(dims, psi, dagger)
    c0 = Fraction(1.0 / (2.0 * KAPPA))
    for part in ("real", "imag"):
        x, s, g = (getattr(v, part).reshape(-1) for v in (c, hop, got))
        for k in range(0, x.size, 3):
            assert g[k] == float(c0 * Fraction(x[k]) + Fraction(s[k])), k


@pytest.mark.parametrize("nrhs,pin", [(2, (64, 1, 2, 1)), (3, (32, 1, 2, 0)), (4, (64, 1, 4, 1)), (12, (64, 1, 2, 1))])
@pytest.mark.parametrize("dagger", [False, True])
def test_binary32_several_rhs_round_once(nrhs, pin, dagger):
    """binary32, several right-hand sides per thread: c0 x by an FMA onto the hops, one
    rounding.  (One site per thread or per two threads: A in2 rounded, then added.)"""
    dims = (8, 8, 8, 16)
    psi = _field(dims, nrhs)
    c, got = _dw(dims, psi, 1, dagger, pin)
    want = np.float32(1.0 / (2.0 * KAPPA)).astype(np.float64) * c + _hops(dims, psi, dagger)   # exact: 34 bits
    assert np.array_equal(got.astype(np.complex64), want.astype(np.complex64))
    assert np.array_equal(got, got.astype(np.complex64))
