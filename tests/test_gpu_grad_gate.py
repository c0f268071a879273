"""The adjoint of the column transfer where its lanes and ranges can go wrong:
batches that leave a warp's units empty, and classes whose probabilities are so
far apart that they are swept back one at a time (or one of them is zero).
Tolerance: a gradient entry sums products that pass some 3 d^2 roundings of
2^-24 each way, 3 sqrt(6 d^2) 6e-8 = 4e-6 at d = 9 of the largest entry, and
cancels between classes by less than a factor of five here: 2e-5."""
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


def _grad(mld, d, noise, syn, up, chi):
    code = mld.Code(d)
    dn = torch.zeros((d * d, 4), dtype=torch.float64, device="cuda")
    lp = torch.zeros((len(syn), 4), dtype=torch.float64, device="cuda")
    mld.mld_decode_grad(code.handle, torch.tensor(noise, device="cuda"), torch.tensor(syn.view(np.int64), device="cuda"),
                        len(syn), chi, torch.tensor(up, device="cuda"), lp, dn)
    torch.cuda.synchronize()
    assert code.status() == 0
    return dn.cpu().numpy(), lp.cpu().numpy()


def _oracle(d, noise, syn, up):
    n = d * d
    lz, g = oracle.coset_dlogz(d, noise.astype(np.float64), oracle.representatives(d, syn).reshape(-1, n))
    return np.einsum("bl,blqp->qp", up, g.reshape(len(syn), 4, n, 4)), lz.reshape(-1, 4)


def _check(dn, ref):
    np.testing.assert_allclose(dn, ref, rtol=2e-5, atol=2e-5 * np.abs(ref).max())


@pytest.mark.parametrize("d", [3, 5, 7, 9])
@pytest.mark.parametrize("B", [1, 2, 3, 5, 9])
def test_ragged_batches(mld, d, B):
    noise = synth.lognormal_biased(d * d, seed=d).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, B, seed=B))
    up = np.random.default_rng(B).normal(size=(B, 4))
    dn, lp = _grad(mld, d, noise, syn, up, 2 ** (d // 2))
    ref, lz = _oracle(d, noise, syn, up)
    _check(dn, ref)
    np.testing.assert_allclose(lp, lz, rtol=0, atol=1e-5)


@pytest.mark.parametrize("d", [3, 5, 7, 9])
@pytest.mark.parametrize("only", [None, 0, 1, 2, 3])
def test_classes_far_apart(mld, d, only):
    """p = 1e-5: the less likely classes lie up to d ln(3e5) = 110 below the
    leading one; upstream gradients on all classes, or on one."""
    B = 6
    noise = synth.depolarizing(d * d, 1e-5).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, synth.depolarizing(d * d, 0.05), B, seed=d))
    up = np.random.default_rng(d).normal(size=(B, 4))
    if only is not None:
        up[:, [l for l in range(4) if l != only]] = 0.0
    dn, _ = _grad(mld, d, noise, syn, up, 2 ** (d // 2))
    ref, _ = _oracle(d, noise, syn, up)
    _check(dn, ref)


@pytest.mark.parametrize("d", [5, 7])
def test_impossible_classes(mld, d):
    """Bit-flip noise: half of the classes have probability zero and add
    nothing."""
    noise = np.zeros((d * d, 4), np.float32)
    noise[:, 0], noise[:, 1] = 0.9, 0.1
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, 7, seed=1))
    up = np.ones((7, 4))
    dn, lp = _grad(mld, d, noise, syn, up, 2 ** (d // 2))
    live = np.where(np.isfinite(lp), up, 0.0)
    assert (live == 0).sum() == 14
    n = d * d
    _, g = oracle.coset_dlogz(d, noise.astype(np.float64), oracle.representatives(d, syn).reshape(-1, n))
    g = g.reshape(7, 4, n, 4)
    ref = np.einsum("bl,blqp->qp", live, np.where(live[:, :, None, None] != 0, g, 0.0))
    _check(dn, ref)
