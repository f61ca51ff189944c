"""Gradients of the learned preconditioner at the edges of their kernels:
more pairs than one group of loss read-backs, lattices with fewer sites than
a block of the weight-gradient grid, and values beyond 2^100 (whose warp sums
are taken in binary64)."""
import numpy as np
import pytest

from oracle import ptc
from paper_2202_07388_gb300 import synth
from tests.gpu_cases import oracle_case, make_handle, rel_err
from tests.test_gpu_nnprec import _packed, _split, _wdev, _weights, NW1, NW2

pytestmark = pytest.mark.gpu


def _grad(h, w, rp, ep, n):
    import torch
    g = torch.zeros(2 * (NW1 + NW2), dtype=torch.float64, device="cuda")
    loss = h.nnprec_grad(_wdev(w), rp, ep, n, g)
    return g.cpu().numpy(), loss


def test_gradient_over_several_groups_of_pairs():
    from paper_2202_07388_gb300 import oq
    dims, n = (2, 4, 2, 4), 35
    u, _, _ = oracle_case(dims, 0.5, 911, 0.135, 1.0)
    h = make_handle(dims, u, 0.135, 1.0, oq.LINK_12)
    r, e = synth.make_source(dims, 912, nrhs=n), synth.make_source(dims, 913, nrhs=n)
    w = _weights(914)
    g, loss = _grad(h, w, _packed(h, oq, r), _packed(h, oq, e), n)
    one = [_grad(h, w, _packed(h, oq, r[k:k + 1]), _packed(h, oq, e[k:k + 1]), 1) for k in range(n)]
    # the same binary32 sums, scaled by 1/n in the loss gradient (one rounding)
    assert rel_err(g, sum(x[0] for x in one) / n) < 1e-6
    assert abs(loss - sum(x[1] for x in one) / n) < 1e-12 * loss
    h.close()


@pytest.mark.parametrize("scale", [1e17, 1.0])
def test_gradient_of_large_values(scale):
    from paper_2202_07388_gb300 import oq
    dims = (4, 2, 4, 6)
    u, _, _ = oracle_case(dims, 0.5, 921, 0.135, 1.0)
    h = make_handle(dims, u, 0.135, 1.0, oq.LINK_18)
    r, e = scale * synth.make_source(dims, 922), synth.make_source(dims, 923)
    w = _weights(924)
    w1, w2 = _split(w)
    g, _ = _grad(h, w, _packed(h, oq, r[None]), _packed(h, oq, e[None]), 1)
    ref = ptc.backward(u, w1, w2, r, e)
    g1, g2 = [x for x in ref if isinstance(x, np.ndarray) and x.ndim == 5][:2]
    refg = np.concatenate([g1.reshape(-1), g2.reshape(-1)])
    got = g[0::2] + 1j * g[1::2]
    if scale > 1.0:
        assert np.abs(refg).max() > 2.0 ** 100
    assert rel_err(got, refg) < 1e-5  # binary32 site sums
    h.close()
