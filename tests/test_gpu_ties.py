"""Ties of the column transfer at d <= 9 (two classes equal up to rounding, as
uniform noise makes them): ln Z and the decision are the boundary-MPS sweep's,
the same bits whether or not decisions are asked for, from a single shot to
batches that fill a block's list of ties, with no tie, some and only ties."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("d", [3, 5, 7, 9])
@pytest.mark.parametrize("B", [1, 2, 3, 65, 1029, 20011])
@pytest.mark.parametrize("p", [0.1, 0.18, 0.75])
def test_same_with_and_without_decisions(mld, d, B, p):
    n, chi = d * d, 2 ** (d // 2)
    E = synth.sample_errors(d, synth.depolarizing(n, p), min(B, 1024), seed=d)
    syn = synth.syndromes_of(d, E)[np.random.default_rng(d).permutation(B) % min(B, 1024)]
    sy = torch.tensor(syn.view(np.int64), device="cuda")
    code, swept = mld.Code(d), mld.Code(d)
    swept.set_exact_kernel(1)
    precisions = [mld.MLD_FP32, mld.MLD_MIXED_TF32] if d == 9 else [mld.MLD_FP32]
    for noise in (torch.tensor(synth.depolarizing(n, p).astype(np.float32), device="cuda"),
                  torch.full((B,), p, dtype=torch.float32, device="cuda")):
        for precision in precisions:
            lp, am = code.decode(noise, sy, chi, precision)
            alone, none = code.decode(noise, sy, chi, precision, with_argmax=False)
            ref, ram = swept.decode(noise, sy, chi, precision)
            torch.cuda.synchronize()
            assert none is None and code.status() == 0
            assert torch.equal(lp, alone) and torch.isfinite(lp).all()
            assert torch.equal(am.long(), lp.argmax(1))
            best = ref.sort(1).values
            tied = best[:, 3] - best[:, 2] < 2e-6           # well inside the 1e-5 that is decided again
            assert torch.equal(lp[tied], ref[tied]) and torch.equal(am[tied], ram[tied])
            if p == 0.75:
                assert tied.float().mean() > 0.9
