"""The adjoint over rare syndromes: a syndrome far less likely than its patch's
typical ones has states whose entries differ by hundreds of powers of two, and
gradients of the order 1/p. Every gradient is finite, whatever the rates and
the zeros of the table; where the span of a state stays above 2^-170 of the
2^-180 that the states keep, it is the oracle's: (p/3)^(3d/2) where every qubit
is noisy (the paths of a column and a half, between two rescalings, may cost a
rate for each qubit), (p/3)^(3d) where paths lead around perfect ones. Tolerance
as for the ragged batches: 2e-5 of the largest entry."""
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


def _tables(n, p, rng):
    """Depolarizing; without Y; dephasing; perfect qubits among noisy ones."""
    t = {"depolarizing": synth.depolarizing(n, p)}
    t["no Y"] = np.tile([1 - p, p / 2, 0.0, p / 2], (n, 1))
    t["dephasing"] = np.tile([1 - p, 0.0, 0.0, p], (n, 1))
    t["perfect qubits"] = synth.depolarizing(n, p)
    t["perfect qubits"][rng.random(n) < 0.3] = [1, 0, 0, 0]
    return {k: v.astype(np.float32) for k, v in t.items()}


def _errors(table, B, rng):
    """Errors of every weight among those that the table allows."""
    n = table.shape[0]
    code = np.array([0, 1, 3, 2], np.uint8)               # I, X, Y, Z -> x + 2z
    E = np.zeros((B, n), np.uint8)
    for b in range(B):
        for q in range(n):
            allowed = np.flatnonzero(table[q, 1:]) + 1
            if allowed.size and rng.random() < 0.75 * b / B:
                E[b, q] = code[rng.choice(allowed)]
    return E


def _grad(mld, d, noise, syn, up):
    code = mld.Code(d)
    dn = torch.zeros((d * d, 4), dtype=torch.float64, device="cuda")
    mld.mld_decode_grad(code.handle, torch.tensor(noise, device="cuda"), torch.tensor(syn.view(np.int64), device="cuda"),
                        len(syn), 2 ** (d // 2), torch.tensor(up, device="cuda"), None, dn)
    torch.cuda.synchronize()
    return dn.cpu().numpy(), code.status()


@pytest.mark.parametrize("d", [3, 5, 7, 9, 11])
@pytest.mark.parametrize("p", [1e-5, 1e-6, 1e-8, 1e-12, 1e-20])
def test_finite_at_any_rate(mld, d, p):
    rng = np.random.default_rng(d)
    for name, noise in _tables(d * d, p, rng).items():
        syn = synth.syndromes_of(d, _errors(noise, 40, rng))
        dn, _ = _grad(mld, d, noise, syn, rng.normal(size=(40, 4)))
        assert np.isfinite(dn).all(), name


@pytest.mark.parametrize("name,columns", [("depolarizing", 1.5), ("perfect qubits", 3)])
@pytest.mark.parametrize("d", [3, 5, 7, 9, 11])
def test_rare_syndromes(mld, d, name, columns):
    rng = np.random.default_rng(d)
    n, B, p = d * d, 12, 3 * 2.0 ** (-170 / (columns * d))
    noise = _tables(n, p, rng)[name]
    syn = synth.syndromes_of(d, _errors(noise, B, rng))
    up = rng.normal(size=(B, 4))
    lz, g = oracle.coset_dlogz(d, noise.astype(np.float64), oracle.representatives(d, syn).reshape(-1, n))
    possible = np.isfinite(lz).reshape(B, 4)
    up = np.where(possible, up, 0.0)
    g = np.where(possible[..., None, None], g.reshape(B, 4, n, 4), 0.0)
    for b in range(B):                                    # shot by shot: their scales differ by 1/p
        ref = np.einsum("l,lqp->qp", up[b], g[b])
        dn, status = _grad(mld, d, noise, syn[b:b + 1], up[b:b + 1])
        assert status == 0
        np.testing.assert_allclose(dn, ref, rtol=2e-5, atol=2e-5 * np.abs(ref).max(), err_msg=str(b))


@pytest.mark.parametrize("d", [3, 5, 7, 9])
def test_batch_gradient_against_64_bits(mld, d):
    """The marginal likelihood's gradient over a batch. A gate's sums are put
    on the overlap of the first gate on its side of the column, so at most
    (d+1)/2 gates of two roundings each separate them, on either state:
    sqrt(2 (d+1)) 2^-25 / sqrt(3) = 8e-8 a shot at d = 9, in part averaged over
    the batch: half an ulp, 2^-24, of the gradient's norm."""
    n, B = d * d, 512
    noise = synth.lognormal_biased(n, seed=d).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, B, seed=1))
    lz, g = oracle.coset_dlogz(d, noise.astype(np.float64), oracle.representatives(d, syn).reshape(-1, n))
    lz = lz.reshape(B, 4)
    post = np.exp(lz - lz.max(axis=1, keepdims=True))
    up = -post / post.sum(axis=1, keepdims=True) / B
    ref = np.einsum("bl,blqp->qp", up, g.reshape(B, 4, n, 4))
    dn, status = _grad(mld, d, noise, syn, up)
    assert status == 0
    assert np.linalg.norm(dn - ref) <= 2.0 ** -24 * np.linalg.norm(ref)


@pytest.mark.parametrize("d", [3, 5, 7, 9])
@pytest.mark.parametrize("up", [(1, -1, 0, 0), (1, -0.3, 0, 0), (0, 0, 1, -0.6), (1, 0.5, 0.2, 0.1)])
def test_opposing_classes(mld, d, up):
    """Single shots whose two l_X classes pull apart: the sums of each class are
    put on its own overlap, so that between two gates of a column's side lie at
    most (d+1)/2 of them, two roundings of 2^-25 / sqrt(3) each on either state:
    sqrt(2 (d+1)) 1.7e-8 of a class's terms, 7.7e-8 at d = 9, besides the sums'
    own and the weights', below 2e-8 d + 6e-8 over both classes. (Without,
    d^2 gates lie between: 3.1e-7 at d = 9.)"""
    n, B = d * d, 64
    noise = synth.lognormal_biased(n, seed=d).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, B, seed=5))
    _, g = oracle.coset_dlogz(d, noise.astype(np.float64), oracle.representatives(d, syn).reshape(-1, n))
    terms = np.array(up, np.float64)[None, :, None, None] * g.reshape(B, 4, n, 4)
    off = []
    for b in range(B):
        dn, status = _grad(mld, d, noise, syn[b:b + 1], np.array([up], np.float64))
        assert status == 0
        off.append(np.linalg.norm(dn - terms[b].sum(0)) / np.linalg.norm(terms[b]))
    assert np.sqrt(np.mean(np.square(off))) <= 2e-8 * d + 6e-8
