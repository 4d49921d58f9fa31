"""The native part of the Python binding: what the calls refuse, and that every form of fan-outs gives the same answer."""
import sys

import numpy as np
import pytest
import torch

from paper_2605_02218_b200 import api, build, workloads


def test_the_native_part_holds_to_one_python_and_one_torch():
    lib = api.load_library()
    assert api._native is not None
    path = build.binding_path()
    assert torch.__version__ in path and sys.implementation.cache_tag in path
    assert api._load_native(lib, path.replace("torch-", "torch-0")) is None       # another version's: not there


def test_a_native_part_that_does_not_load_is_named_and_done_without(tmp_path):
    broken = tmp_path / "_binding.so"
    broken.write_bytes(b"no library")
    with pytest.warns(RuntimeWarning, match="_binding.so"):
        assert api._load_native(api.load_library(), str(broken)) is None


def test_a_failed_build_of_the_native_part_leaves_the_library(monkeypatch, capsys):
    monkeypatch.setattr(build, "build_binding", lambda force=False: (_ for _ in ()).throw(RuntimeError("no Python.h")))
    assert build.build() == build.LIB and "no Python.h" in capsys.readouterr().err


@pytest.mark.gpu
def test_without_the_native_part_the_calls_give_the_same(monkeypatch):
    d = workloads.make_logits(seed=4, rows=8, vocab=40000, dtype=torch.float16, device="cuda:0")
    wl = workloads.make_workload("static", seed=5, dtype=torch.bfloat16, batch=3, n_vis=(90, 300), n_txt=(1, 20), d=264, n_heads=0,
                                 rank=8, keep_ratio=0.2, act_layers=0, device="cuda:0")

    def calls():
        cand, off = api.branch_candidates(d["z_draft"], [8, 5, 3, 2, 1, 0, 1, 2], d["drafted"], vocab=40000)
        return [*api.correct(d["z_draft"], d["z_target"], d["uniforms"], 0.02, d["drafted"], vocab=40000), cand,
                torch.from_numpy(off), api.query_score_static(wl.X, wl.Q, wl.vis_offsets, wl.txt_offsets)]
    want = calls()
    monkeypatch.setattr(api, "_native", None)
    for a, b in zip(want, calls()):
        assert torch.equal(a, b)
    with pytest.raises(TypeError):
        api.correct(d["z_draft"], d["z_target"], d["uniforms"].double(), 0.02)


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


def _z(rows=4, ld=64, dtype=torch.float16):
    return torch.zeros(rows, ld, dtype=dtype, device="cuda:0")


@pytest.mark.gpu
@pytest.mark.parametrize("error,kw", [
    (TypeError, dict(uniforms=lambda: torch.zeros(4, dtype=torch.float64, device="cuda:0"))),
    (TypeError, dict(uniforms=lambda: [0.0] * 4)),
    (ValueError, dict(uniforms=lambda: torch.zeros(4))),                              # not on the device
    (ValueError, dict(uniforms=lambda: torch.zeros(3, device="cuda:0"))),             # too short
    (ValueError, dict(uniforms=lambda: torch.zeros(1, device="cuda:0").expand(4))),   # no dense memory
    (TypeError, dict(drafted=lambda: torch.zeros(4, dtype=torch.int64, device="cuda:0"))),
    (ValueError, dict(drafted=lambda: torch.zeros(4, dtype=torch.int32))),
    (ValueError, dict(drafted=lambda: torch.zeros(3, dtype=torch.int32, device="cuda:0"))),
    (ValueError, dict(drafted=lambda: torch.zeros(8, dtype=torch.int32, device="cuda:0")[::2])),
    (ValueError, dict(z_target=lambda: _z().cpu())),
    (ValueError, dict(vocab=lambda: 2 ** 32 + 32)),
])
def test_correct_refuses_memory_that_the_kernel_must_not_read(error, kw):
    # all of these return before anything is launched
    args = dict(z_draft=_z(), z_target=_z(), uniforms=torch.zeros(4, device="cuda:0"), gamma=0.02,
                drafted=torch.zeros(4, dtype=torch.int32, device="cuda:0"))
    with pytest.raises(error):
        api.correct(**{**args, **{k: make() for k, make in kw.items()}})


@pytest.mark.gpu
@pytest.mark.parametrize("fans", [[2] * 4, (2,) * 4])                   # the native call and the general one
@pytest.mark.parametrize("error,kw", [
    (ValueError, dict(z_draft=lambda: _z().cpu())),
    (ValueError, dict(z_draft=lambda: _z(4, 128)[:, :64])),              # rows are not back to back
    (KeyError, dict(z_draft=lambda: _z(dtype=torch.float64))),
    (TypeError, dict(drafted=lambda: torch.zeros(4, dtype=torch.int64, device="cuda:0"))),
    (ValueError, dict(drafted=lambda: torch.zeros(3, dtype=torch.int32, device="cuda:0"))),
    (ValueError, dict(drafted=lambda: torch.zeros(4, dtype=torch.int32))),
    (ValueError, dict(vocab=lambda: 2 ** 32 + 32)),
])
def test_candidates_refuse_memory_that_the_kernel_must_not_read(error, kw, fans):
    args = dict(z_draft=_z(), fanouts=fans, drafted=torch.zeros(4, dtype=torch.int32, device="cuda:0"))
    with pytest.raises(error):
        api.branch_candidates(**{**args, **{k: make() for k, make in kw.items()}})


@pytest.mark.gpu
@pytest.mark.parametrize("error,kw", [
    (TypeError, dict(X=lambda: _z(), Q=lambda: _z())),                   # float16
    (ValueError, dict(Q=lambda: torch.zeros(4, 32, device="cuda:0"))),   # another width
    (ValueError, dict(vis_offsets=lambda: [0, 5])),                      # past the end of X
    (ValueError, dict(txt_offsets=lambda: [0, 5])),
    (ValueError, dict(vis_offsets=lambda: [0, 2, 4])),                   # more requests than in the other list
    (ValueError, dict(vis_offsets=lambda: [4], txt_offsets=lambda: [4])),
    (TypeError, dict(out=lambda: torch.zeros(4, dtype=torch.bfloat16, device="cuda:0"))),
    (ValueError, dict(out=lambda: torch.zeros(3, device="cuda:0"))),
    (ValueError, dict(out=lambda: torch.zeros(4))),
    (ValueError, dict(out=lambda: torch.zeros(8, device="cuda:0")[::2])),
])
def test_static_score_refuses_memory_that_the_kernel_must_not_touch(error, kw):
    args = dict(X=_z(dtype=torch.float32), Q=_z(dtype=torch.float32), vis_offsets=[0, 4], txt_offsets=[0, 4])
    with pytest.raises(error):
        api.query_score_static(**{**args, **{k: make() for k, make in kw.items()}})


@pytest.mark.gpu
def test_pinned_host_memory_is_taken_and_gives_the_same():
    d = workloads.make_logits(seed=3, rows=4, vocab=1000, dtype=torch.float16, device="cuda:0")
    z, y = d["z_draft"], d["drafted"]
    want = api.correct(z, d["z_target"], d["uniforms"], 0.02, y, vocab=1000)
    got = api.correct(z, d["z_target"], d["uniforms"].cpu().pin_memory(), 0.02, y.cpu().pin_memory(), vocab=1000)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    want, off = api.branch_candidates(z, [3, 2, 1, 0], y, vocab=1000)
    got, off2 = api.branch_candidates(z, [3, 2, 1, 0], y.cpu().pin_memory(), vocab=1000)
    torch.cuda.synchronize()
    assert torch.equal(want, got) and np.array_equal(off, off2)
