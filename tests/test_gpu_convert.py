"""Packing and unpacking of fields bit for bit against the conversions of the host
(round to nearest even; binary64, binary32 and binary16): ties, values that round up to the next
exponent or to infinity, binary32 subnormals, zeros of both signs, infinities
and NaN, with scale 1 and a power of two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _specials():
    one = np.float64(1.0)
    ulp = 2.0 ** -23
    v = [0.0, -0.0, 1.0, -1.0, one + ulp / 2, one + 1.5 * ulp, one + ulp / 2 + 2.0 ** -50, one + ulp / 2 - 2.0 ** -50,
         2.0 - ulp / 2, 2.0 - ulp / 4, np.finfo(np.float32).max, 3.4028235677973366e38, 3.40282356e38, 1e39, -1e39,
         2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -25), 2.0 ** -127, 2.0 ** -149, 2.0 ** -150, 1e-46, -1e-310,
         np.inf, -np.inf, np.nan, 2.0 ** 127, 2.0 ** 128 * (1 - 2.0 ** -25), 1e-300]
    rng = np.random.default_rng(951)
    bits = rng.integers(0, 1 << 63, 4000, dtype=np.uint64).view(np.float64)
    near = (rng.standard_normal(4000).astype(np.float32).astype(np.float64) * (1 + rng.choice([0, 1, -1, 3], 4000) * 2.0 ** -24))
    return np.concatenate([v, bits, near, rng.standard_normal(4000) * 2.0 ** rng.integers(-160, 130, 4000)])


@pytest.mark.parametrize("scale", [1.0, 0.25])
@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("dims", [(4, 4, 6, 8), (2, 2, 2, 2), (2, 6, 10, 6)])   # 384, 8, 360 sites of a parity
def test_binary32_pack_and_unpack_bits(scale, half, dims):
    import torch
    from paper_2202_07388_gb300 import oq
    vol = int(np.prod(dims))
    x = np.resize(_specials(), (vol, 24))
    h = oq.Handle(dims)
    sub = oq.EVEN if half else oq.FULL
    packed = h.new_packed(oq.F32, sub)
    h.pack(torch.from_numpy(x).cuda(), packed, oq.F32, sub, scale=scale)
    with np.errstate(over="ignore", invalid="ignore"):
        ref = (x * scale).astype(np.float32)
    par = (np.indices(dims).sum(axis=0) % 2).reshape(-1)
    halves = [ref[par == p] for p in ((0,) if half else (0, 1))]
    want = np.concatenate([v.reshape(-1, 6, 4).transpose(1, 0, 2).reshape(-1) for v in halves])
    got = packed.view(torch.float32).cpu().numpy()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got.view(np.uint32)[~nan], want.view(np.uint32)[~nan])
    back = torch.zeros(vol, 24, dtype=torch.float64, device="cuda")
    h.unpack(packed, back, oq.F32, sub, scale=scale)
    exp = ref.astype(np.float64) / scale
    if half:
        exp[par == 1] = 0.0
    b = back.cpu().numpy()
    ok = ~np.isnan(exp)
    assert np.array_equal(b.view(np.uint64)[ok], exp.view(np.uint64)[ok]) and np.isnan(b[~ok]).all()
    h.close()


@pytest.mark.parametrize("scale", [1.0, 0.25])
@pytest.mark.parametrize("sub", [0, 1, 2])
@pytest.mark.parametrize("prec", [0, 3])
def test_pack_and_unpack_bits_of_two_fields(prec, sub, scale):
    """Subsets and two right-hand sides, a site count that fills no last CTA; the sites
    of the other parity stay as they were.  All-zero sites and fields included."""
    import torch
    from paper_2202_07388_gb300 import oq
    dims = (2, 6, 10, 6)
    vol = 720
    rng = np.random.default_rng(952)
    x = rng.standard_normal((2, vol, 24))
    x[0, ::7] = 0.0
    x[1, 100:400] = -0.0
    h = oq.Handle(dims)
    packed = h.new_packed(prec, sub, nrhs=2)
    h.pack(torch.from_numpy(x).cuda(), packed, prec, sub, scale=scale, nrhs=2)
    t = {0: np.float64, 3: np.float16}[prec]
    ref = (x * scale).astype(t)
    par = (np.indices(dims).sum(axis=0) % 2).reshape(-1)
    chunk = 16 // np.dtype(t).itemsize
    want = [ref[r][par == p].reshape(-1, 24 // chunk, chunk).transpose(1, 0, 2).reshape(-1)
            for r in (0, 1) for p in ((0, 1) if sub == oq.FULL else (sub,))]
    got = packed.cpu().numpy().view(np.uint8)
    assert np.array_equal(got, np.concatenate(want).view(np.uint8))
    back = torch.full((2, vol, 24), 7.0, dtype=torch.float64, device="cuda")
    h.unpack(packed, back, prec, sub, scale=scale, nrhs=2)
    exp = ref.astype(np.float64) / scale
    if sub != oq.FULL:
        exp[:, par != sub] = 7.0
    assert np.array_equal(back.cpu().numpy().view(np.uint64), exp.view(np.uint64))
    h.close()
