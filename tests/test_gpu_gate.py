"""The column transfer (untruncated chi, d <= 13) at the sizes where its
launch shapes can go wrong: around a thread block's and a warp's share of a
batch, at the slots whose logarithms are taken together, and past one pass of
the resident blocks; both noise modes, against the FP64 oracle. Tolerance: at
most d^2 gates of three roundings each, relative 2^-24, random in sign:
3 sigma at d = 13 is 3 * sqrt(3 * 169) * 6e-8 = 4e-6, below the 1e-5 of the
untruncated path."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def mld():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_17230_gb300 as m
    m.load()
    return m


def _decode(mld, d, noise, syn, chi):
    code = mld.Code(d)
    lp, am = code.decode(torch.tensor(noise, device="cuda"), torch.tensor(syn.view(np.int64), device="cuda"), chi)
    torch.cuda.synchronize()
    assert code.status() == 0
    return lp.cpu().numpy(), am.cpu().numpy()


@pytest.mark.parametrize("d", [3, 5, 7, 9, 11, 13])
@pytest.mark.parametrize("B", [1, 2, 7, 8, 9, 17, 63, 65, 130])
def test_ragged_batches(mld, d, B):
    n, chi = d * d, 2 ** (d // 2)
    noise = synth.lognormal_biased(n, seed=d).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, B, seed=B))
    k = min(B, 24)                                        # oracle-checked: both ends of the batch
    at = np.unique(np.r_[0:k // 2, B - (k - k // 2):B])
    ref, _ = oracle.decode(d, noise.astype(np.float64), syn[at])
    lp, am = _decode(mld, d, noise, syn, chi)
    np.testing.assert_allclose(lp[at], ref, rtol=0, atol=TOL)
    assert np.array_equal(am, np.argmax(lp, axis=1))
    p = np.random.default_rng(B).uniform(0.02, 0.18, B).astype(np.float32)
    rows = [np.array([np.float32(1) - p[b]] + [p[b] * np.float32(1.0 / 3.0)] * 3, np.float64) for b in at]
    ref = np.concatenate([oracle.decode(d, np.tile(r, (n, 1)), syn[b:b + 1])[0] for r, b in zip(rows, at)])
    lp, am = _decode(mld, d, p, syn, chi)
    np.testing.assert_allclose(lp[at], ref, rtol=0, atol=TOL)
    assert np.array_equal(am, np.argmax(lp, axis=1))


@pytest.mark.parametrize("d,B", [(3, 90001), (5, 90001), (7, 70001), (9, 40003), (11, 12007), (13, 4111)])
def test_more_than_one_pass_of_the_resident_blocks(mld, d, B):
    """Every syndrome of a batch larger than the chip holds at once, against
    the same syndromes decoded in small batches (equal bits), and ties marked
    by uniform noise: decisions are classes, and argmax of the stored ln Z."""
    n, chi = d * d, 2 ** (d // 2)
    noise = synth.depolarizing(n, 0.15).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, 512, seed=1))
    syn = syn[np.random.default_rng(d).integers(0, 512, B)]
    lp, am = _decode(mld, d, noise, syn, chi)
    assert np.isfinite(lp).all() and np.array_equal(am, np.argmax(lp, axis=1))
    for b in (0, B // 2, B - 33):
        few, fam = _decode(mld, d, noise, syn[b:b + 33], chi)
        np.testing.assert_array_equal(lp[b:b + 33], few)
        np.testing.assert_array_equal(am[b:b + 33], fam)


@pytest.mark.parametrize("d", [3, 5, 7, 9, 11])
def test_extreme_rates(mld, d):
    """Arbitrary syndromes at p = 1e-5 (entries far apart, rescaled column by
    column), and certain errors (p = 1: no identity weight anywhere)."""
    n, chi = d * d, 2 ** (d // 2)
    rng = np.random.default_rng(d)
    syn = synth.pack_bits((rng.random((12, n - 1)) < 0.25).astype(np.uint8))
    for p in (1e-5, 1.0):
        noise = synth.depolarizing(n, p).astype(np.float32)
        ref, _ = oracle.decode(d, noise.astype(np.float64), syn)
        lp, _ = _decode(mld, d, noise, syn, chi)
        fin = np.isfinite(ref)
        assert np.array_equal(np.isfinite(lp), fin)
        np.testing.assert_allclose(lp[fin], ref[fin], rtol=0, atol=TOL)
