"""The truncated sweep keeps one order of every sum wherever a step's buffers
lie: the same syndromes in batches that give a unit 13,500, 6,500 and 3,072
floats on chip (steps stay on chip, spill in part or spill altogether) have the
same bits."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,chi,p", [(11, 16, 0.15), (13, 32, 0.16), (17, 32, 0.15), (17, 128, 0.13)])
def test_bits_do_not_depend_on_the_arena(d, chi, p):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_17230_gb300 as mld
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, few = d * d, 24
    noise = synth.depolarizing(n, p).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, few, seed=d + chi))
    easy = synth.syndromes_of(d, synth.sample_errors(d, synth.depolarizing(n, 0.01), 5 * sms, seed=1))
    nz = torch.tensor(noise, device="cuda")
    out, spilled = [], []
    for extra in (0, 3 * sms, 5 * sms):           # 2 units each: up to 4, 8 and more per SM
        code = mld.Code(d)
        code.set_truncation_kernel(1)
        batch = np.concatenate([syn, easy[:extra]])
        lp, am = code.decode(nz, torch.tensor(batch.view(np.int64), device="cuda"), chi)
        torch.cuda.synchronize()
        assert code.status() == 0
        out.append((lp[:few].cpu().numpy(), am[:few].cpu().numpy()))
        spilled.append(int(code.bond_histogram()[0]))
    assert spilled[2] >= spilled[1] >= spilled[0] and spilled[2] > 0
    for lp, am in out[1:]:
        np.testing.assert_array_equal(lp, out[0][0])
        np.testing.assert_array_equal(am, out[0][1])


@pytest.mark.parametrize("d,chi", [(7, 4), (11, 8)])
def test_a_queued_batch_has_the_bits_of_its_parts(d, chi):
    """A batch long enough to be taken heaviest syndrome first (one and two
    words a syndrome, empty and repeated ones among them) against the same
    syndromes in batches that are not."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_17230_gb300 as mld
    n, part = d * d, 500
    B = 12 * torch.cuda.get_device_properties(0).multi_processor_count + 17     # 24 units an SM and more
    noise = synth.depolarizing(n, 0.1).astype(np.float32)
    syn = synth.syndromes_of(d, synth.sample_errors(d, noise, B, seed=d))
    syn[:3] = 0
    syn[B - 5:] = syn[7]
    nz = torch.tensor(noise, device="cuda")
    dev = torch.tensor(syn.view(np.int64), device="cuda")
    code = mld.Code(d)
    code.set_truncation_kernel(1)
    lp, am = code.decode(nz, dev, chi)
    for b in range(0, B, part):
        lq, aq = code.decode(nz, dev[b:b + part], chi)
        assert torch.equal(lp[b:b + part], lq) and torch.equal(am[b:b + part], aq)
    torch.cuda.synchronize()
    assert code.status() == 0
