"""The column transfer behind FP64 decodes under independent X/Z noise at the
distances where its lane layout changes (one thread a unit up to d = 13, 2 to
64 lanes above), and at batches that do not fill a block. Tolerance: some
2 d^2 operations of relative error 2^-46 on ln Z, random in sign, stay below
1e-12; the Kac-Ward oracle's dense determinant carries 1e-8 at these rates."""
import numpy as np
import pytest

import oracle.kac_ward as okw
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


def _inputs(d, B, seed):
    n = d * d
    rng = np.random.default_rng(seed)
    px = rng.uniform(0.05, 0.12, n).astype(np.float32)
    pz = rng.uniform(0.05, 0.12, n).astype(np.float32)
    tab = okw.xz_table(px.astype(np.float64), pz.astype(np.float64))
    return px, pz, synth.syndromes_of(d, synth.sample_errors(d, tab, B, seed=seed + 1))


def _decode(mld, d, px, pz, syn):
    code = mld.Code(d)
    lp, am = code.decode_xz(torch.tensor(px, device="cuda"), None if pz is None else torch.tensor(pz, device="cuda"),
                            torch.tensor(syn.view(np.int64), device="cuda"), mld.MLD_FP64)
    torch.cuda.synchronize()
    assert code.status() == 0
    return lp.cpu().numpy(), am.cpu().numpy()


@pytest.mark.parametrize("d", [3, 7, 13, 15, 19, 21, 23, 25])
def test_every_lane_layout(mld, d):
    px, pz, syn = _inputs(d, 3, d)
    ref, _ = okw.decode_xz(d, px.astype(np.float64), pz.astype(np.float64), syn)
    lp, am = _decode(mld, d, px, pz, syn)
    near = ref >= ref.max(axis=1, keepdims=True) - 12.0
    np.testing.assert_allclose(lp[near], ref[near], rtol=0, atol=1e-7)
    assert np.array_equal(am, np.argmax(lp, axis=1))


@pytest.mark.parametrize("d", [5, 13, 15, 17, 19, 21, 23, 25])
@pytest.mark.parametrize("bitflip", [False, True])
def test_ragged_batches(mld, d, bitflip):
    """Every syndrome of a batch that leaves a block partly empty, equal bits
    to the same syndromes one by one."""
    px, pz, syn = _inputs(d, 67 if d <= 17 else 11, 3 * d)
    pz = None if bitflip else pz
    lp, am = _decode(mld, d, px, pz, syn)
    for b in (0, 1, len(syn) // 2, len(syn) - 1):
        one, oam = _decode(mld, d, px, pz, syn[b:b + 1])
        np.testing.assert_array_equal(lp[b:b + 1], one)
        np.testing.assert_array_equal(am[b:b + 1], oam)


@pytest.mark.parametrize("d", [9, 15, 21])
def test_more_than_the_resident_blocks(mld, d):
    px, pz, syn = _inputs(d, 64, d)
    at = np.random.default_rng(d).integers(0, 64, {9: 20011, 15: 9001, 21: 1501}[d])
    few, fam = _decode(mld, d, px, pz, syn)
    lp, am = _decode(mld, d, px, pz, syn[at])
    np.testing.assert_array_equal(lp, few[at])
    np.testing.assert_array_equal(am, fam[at])
