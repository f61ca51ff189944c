"""The clover build where its elimination needs pivoting: blocks far from
diagonally dominant (large c_sw), against the oracle's inverse."""
import numpy as np
import pytest

from oracle import dirac
from paper_2202_07388_gb300 import synth
from tests.gpu_cases import make_handle, to_dev, from_dev, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,csw", [((2, 4, 6, 2), 1.0), ((4, 2, 6, 4), 9.0), ((4, 4, 4, 6), 25.0)])
def test_inverse_blocks_of_any_sign(dims, csw):
    from paper_2202_07388_gb300 import oq
    kappa = 0.13
    u = synth.make_gauge(dims, 0.9, 901)
    a = dirac.clover_field(u, dirac.kappa_to_m0(kappa), csw)
    ainv = np.linalg.inv(a)
    cond = np.linalg.cond(a).max()
    if csw > 1.0:  # indefinite blocks: eliminations without pivoting meet small pivots
        assert np.linalg.eigvalsh(a.reshape(-1, 12, 12)).min() < -1.0
    psi = dirac.even_part(synth.make_source(dims, 902))
    h = make_handle(dims, u, kappa, csw, oq.LINK_12)
    pin, pout = h.new_packed(oq.F64, oq.EVEN), h.new_packed(oq.F64, oq.EVEN)
    h.pack(to_dev(psi), pin, oq.F64, oq.EVEN)
    h.dw_hat(pin, pout, oq.F64)
    out = to_dev(np.zeros_like(psi))
    h.unpack(pout, out, oq.F64, oq.EVEN)
    ref = dirac.dw_hat(u, a, ainv, psi)
    # both inverses err by a few eps times the condition number of a block
    assert rel_err(from_dev(out, psi.shape), ref) < 64 * 2.0 ** -53 * max(cond, 10.0)
    h.close()
