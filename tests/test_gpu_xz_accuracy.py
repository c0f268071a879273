"""FP64 decodes under independent X/Z noise at d >= 15 (pairs of FP32 numbers,
and FP64 where rates leave their range), against the sum over each part's
patterns by a column transfer on (d-1)/2 + 1 bits in extended precision: all
four classes, at every rate.

Tolerance: a column's (d-1)/2 gates are each off by 2^-46 (pairs: products and
sums of 2^-47, weights of 2^-49), so the 2 d (d-1)/2 of a decode are off by at
most 600 * 2^-46 = 8.5e-12 at d = 25, besides the rounding of ln Z itself."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mld():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_17230_gb300 as m
    m.load()
    return m


def _part(d, p, e, turned):
    """ln of a part's coset sums [B][2] relative to the errors e [B][n], without
    and with the string on the last column; the other part's plaquettes of
    the patch turned by a quarter are this part's."""
    B, n = e.shape
    grid = np.arange(n).reshape(d, d)
    order = (grid[::-1].T if turned else grid).reshape(-1)
    p, e = p[order].astype(np.longdouble), e[:, order]
    string = np.zeros(n, np.uint8)
    string[d - 1::d] = 1
    e2 = np.stack([e, e ^ string], 1).reshape(2 * B, n)
    w = np.stack([np.where(e2, p, 1 - p), np.where(e2, 1 - p, p)], 2)
    S = np.repeat((np.arange(1 << (d + 1) // 2) == 0).astype(np.longdouble)[None], 2 * B, 0)
    ln = np.zeros(2 * B, np.longdouble)
    pair = np.arange(2)[:, None] ^ np.arange(2)[None]
    for c in range(d):
        for r in range(d) if c % 2 == 0 else range(d - 1, -1, -1):
            q, k = w[:, r * d + c], r // 2
            if r % 2 == 0:
                S = S.reshape(2 * B, -1, 2, 1 << k)
                S = q[:, 0, None, None, None] * S + q[:, 1, None, None, None] * S[:, :, ::-1]
            else:
                S = S.reshape(2 * B, -1, 2, 2, 1 << k)
                S = S * q[:, pair][:, None, :, :, None]
        S = S.reshape(2 * B, -1)
        top = S.max(1, keepdims=True)
        S, ln = S / top, ln + np.log(top[:, 0])
    return (ln + np.log(S[:, 0])).reshape(B, 2)


def _reference(d, px, pz, syn):
    rep = oracle.representatives(d, syn)[:, 0]
    zx = _part(d, px, rep & 1, False)
    zz = _part(d, pz, rep >> 1, True)
    return np.stack([zx[:, l & 1] + zz[:, l >> 1] for l in range(4)], 1).astype(np.float64)


def _decode(mld, d, px, pz, syn):
    code = mld.Code(d)
    lp, am = code.decode_xz(torch.tensor(px, device="cuda"), torch.tensor(pz, device="cuda"),
                            torch.tensor(syn.view(np.int64), device="cuda"), mld.MLD_FP64)
    torch.cuda.synchronize()
    return lp.cpu().numpy(), am.cpu().numpy(), code.status()


def _syndromes(d, weights, rng):
    E = np.zeros((len(weights), d * d), np.uint8)
    for b, w in enumerate(weights):
        E[b] = (rng.random(d * d) < w) + 2 * (rng.random(d * d) < w)
    return synth.syndromes_of(d, E)


@pytest.mark.parametrize("d", [15, 17, 21, 25])
def test_uniform_rates(mld, d):
    """One rate for all qubits: a rounding of a gate's weights comes back in
    every gate. The odds are rounded to 2^-49, which the n p flips of a part
    carry; the gates' roundings add up at random, 3 sqrt(d^2) 2^-47."""
    p = np.full(d * d, 0.1, np.float32)
    syn = _syndromes(d, [0.0, 0.1, 0.1], np.random.default_rng(d))
    ref = _reference(d, p, p, syn)
    lp, am, status = _decode(mld, d, p, p, syn)
    assert status == 0
    np.testing.assert_allclose(lp, ref, rtol=0, atol=2 * 0.1 * d * d * 2.0 ** -49 + 3 * d * 2.0 ** -47)
    assert np.array_equal(am, np.argmax(lp, axis=1))


RATES = ["0.1", "0.01", "1e-4", "1e-6", "1e-8", "1e-12", "mixed", "mostly certain"]


@pytest.mark.parametrize("d", [15, 17, 21, 25])
@pytest.mark.parametrize("rates", RATES)
def test_every_rate(mld, d, rates):
    """From typical to dense errors, where entries of a column lie (p)^d below
    its largest, and with certain errors on half of the qubits."""
    rng = np.random.default_rng(d)
    n = d * d
    if rates == "mixed":
        px, pz = (10 ** rng.uniform(-8, -0.5, n) for _ in range(2))
    elif rates == "mostly certain":
        px, pz = (np.where(rng.random(n) < 0.5, 1e-6, 1 - 1e-6) for _ in range(2))
    else:
        px = pz = np.full(n, float(rates))
    px, pz = px.astype(np.float32), pz.astype(np.float32)
    syn = _syndromes(d, [0.0, 0.02, 0.1, 0.3, 0.5], rng)
    ref = _reference(d, px, pz, syn)
    lp, am, status = _decode(mld, d, px, pz, syn)
    assert status == 0
    np.testing.assert_allclose(lp, ref, rtol=1e-15, atol=1e-11)
    assert np.array_equal(am, np.argmax(lp, axis=1))


@pytest.mark.parametrize("d,B", [(15, 37), (17, 9), (25, 3)])
@pytest.mark.parametrize("bitflip", [False, True])
def test_marked_among_others(mld, d, B, bitflip):
    """Dense errors beside typical ones at p = 1e-4 in one batch: only some
    leave the pairs' range, and each gives the same bits alone."""
    rng = np.random.default_rng(B)
    p = np.full(d * d, 1e-4, np.float32)
    syn = _syndromes(d, rng.choice([0.0, 0.02, 0.5], B), rng)
    code = mld.Code(d)
    tp = torch.tensor(p, device="cuda")
    ts = torch.tensor(syn.view(np.int64), device="cuda")
    lp, am = code.decode_xz(tp, None if bitflip else tp, ts, mld.MLD_FP64)
    assert not torch.isnan(lp).any()
    for b in range(B):
        one, oam = code.decode_xz(tp, None if bitflip else tp, ts[b:b + 1], mld.MLD_FP64)
        assert torch.equal(lp[b:b + 1], one) and torch.equal(am[b:b + 1], oam)
    assert code.status() == 0
