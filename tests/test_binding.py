"""The native part of the Python binding: what the calls refuse, and that every form of fan-outs gives the same answer."""
import numpy as np
import pytest
import torch

from paper_2605_02218_b200 import api, workloads


def test_correct_refuses_what_it_does_not_take():
    z = torch.zeros(2, 64, dtype=torch.float16)
    u = torch.zeros(2)
    with pytest.raises(AssertionError):
        api.correct(z, z, u, 0.02)                                   # not on a device
    with pytest.raises(AssertionError):
        api.query_score_static(z, z, [0, 2], [0, 2])


@pytest.mark.gpu
def test_correct_argument_errors_keep_their_kind():
    d = workloads.make_logits(seed=1, rows=2, vocab=512, dtype=torch.float16, device="cuda:0")
    z, u = d["z_draft"], d["uniforms"]
    with pytest.raises(AssertionError):
        api.correct(z, z[:1], u, 0.02)
    with pytest.raises(AssertionError):
        api.correct(z, z.float(), u, 0.02)
    with pytest.raises(AssertionError):
        api.correct(z[:, ::2], z[:, ::2], u, 0.02)
    with pytest.raises(KeyError):
        api.correct(z.double(), z.double(), u, 0.02)
    with pytest.raises(ValueError):
        api.correct(z[0], z[0], u, 0.02)
    with pytest.raises(api.CovspecError) as e:
        api.correct(z, z, None, 0.02)
    assert e.value.status == -1
    for gamma in (np.float32(0.02), torch.tensor(0.02), 0):
        assert len(api.correct(z, z, u, gamma)) == 5
    own = api.correct(z, z, u, 0.02, d["drafted"])
    assert len({t.data_ptr() for t in own}) == 5 and [t.dtype for t in own] == [torch.float32, torch.int32, torch.float32,
                                                                               torch.float32, torch.int32]


@pytest.mark.gpu
@pytest.mark.parametrize("vocab,fan", [(40000, 8), (40000, 70), (600, 5), (40000, 0)])
def test_fanouts_of_every_form_give_the_same_candidates(vocab, fan):
    # 70: the general selection; 600: a row too short for the cluster kernel; 0: no candidates at all
    d = workloads.make_logits(seed=2, rows=3, vocab=vocab, dtype=torch.float32, device="cuda:0")
    f = [fan, max(fan - 3, 0), min(fan, 1)]
    want, off = api.branch_candidates(d["z_draft"], f, d["drafted"], vocab=d["vocab"])
    assert off.dtype == np.int32 and off.tolist() == [0] + np.cumsum(f).tolist() and want.numel() == sum(f)
    for form in (tuple(f), np.array(f), np.array(f, dtype=np.int32), [np.int64(v) for v in f], [float(v) for v in f]):
        got, off2 = api.branch_candidates(d["z_draft"], form, d["drafted"], vocab=d["vocab"])
        assert torch.equal(want, got) and np.array_equal(off, off2)
    with pytest.raises(AssertionError):
        api.branch_candidates(d["z_draft"], f[:2], d["drafted"], vocab=d["vocab"])
    with pytest.raises(api.CovspecError) as e:
        api.branch_candidates(d["z_draft"], [-1, 2, 2], d["drafted"], vocab=d["vocab"])
    assert e.value.status == -2
