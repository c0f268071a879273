"""The column transfer at rates where the classes lie far apart: l_X = 1 of a
light syndrome pays a rate in every row of one column (of any: its strings lie
(p/3)^d below a state's largest entry), l_Z = 1 one in every column. While
(p/3)^d stays above 2^-220 (FP32's range below 2^100, less the accuracy asked
for) ln Z of all four classes is the FP64 oracle's, tolerance as for the ragged
batches. Below, the last column's own strings still hold: its (d+1)/2 first
rows are paid before the classes are rescaled, (p/3)^((d+1)/2) >= 2^-249, and
no possible class is lost."""
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


def _decode(mld, d, p, mode):
    n, rng = d * d, np.random.default_rng(d)
    E = np.zeros((4, n), np.uint8)
    for b in range(1, 4):                                  # one, two, three single-qubit errors
        E[b, rng.choice(n, b, replace=False)] = rng.integers(1, 4, b)
    syn = synth.syndromes_of(d, E)
    code, sy = mld.Code(d), torch.tensor(syn.view(np.int64), device="cuda")
    if mode == "detector picture":
        q, c = np.repeat(np.arange(n), 3).astype(np.int32), np.tile([1, 2, 3], n).astype(np.int32)
        lp, _ = code.decode_dem(q, c, np.full(3 * n, p / 3), sy)
        rows = oracle.dem_qubit_table(d, q, c, np.full(3 * n, p / 3))
    elif mode == "table":
        noise = synth.depolarizing(n, p).astype(np.float32)
        lp, _ = code.decode(torch.tensor(noise, device="cuda"), sy, 2 ** (d // 2))
        rows = noise.astype(np.float64)
    else:
        f = np.float32(p)
        lp, _ = code.decode(torch.full((4,), p, dtype=torch.float32, device="cuda"), sy, 2 ** (d // 2))
        rows = np.tile(np.array([np.float32(1) - f] + [f * np.float32(1 / 3)] * 3, np.float64), (n, 1))
    torch.cuda.synchronize()
    assert code.status() == 0
    ref, _ = oracle.decode(d, rows, syn)
    assert np.isfinite(ref).all()
    return lp.cpu().numpy(), ref


@pytest.mark.parametrize("mode", ["table", "shots", "detector picture"])
@pytest.mark.parametrize("d,p", [(3, 1e-15), (5, 1e-12), (7, 1e-9), (9, 2e-7), (11, 3e-6), (13, 3e-5)])
def test_light_syndromes(mld, d, p, mode):
    if mode == "detector picture" and d > 11:
        pytest.skip("d <= 11")
    for rate in (p, 10 * p, 1e-4):
        lp, ref = _decode(mld, d, rate, mode)
        np.testing.assert_allclose(lp, ref, rtol=0, atol=1e-5)


@pytest.mark.parametrize("mode", ["table", "shots"])
@pytest.mark.parametrize("d,p", [(7, 1e-12), (9, 1e-9), (11, 1e-9), (13, 1e-7)])
def test_no_possible_class_is_lost(mld, d, p, mode):
    lp, _ = _decode(mld, d, p, mode)
    assert np.isfinite(lp).all()
