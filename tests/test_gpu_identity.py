"""Eq. 10 with the identity embedding on the tensor cores (bf16): sizes at the edges of its tiles, passes
and accumulation groups, against the oracle's definition in float64, through both entry points."""
import numpy as np
import pytest
import torch

from paper_2605_02218_b200 import workloads

pytestmark = pytest.mark.gpu

# bf16 products are exact in float32; sums of at most 512 terms per truncating tensor-core chain (32 steps
# of 16 terms, 2^-23 each, all of one sign at worst) plus a few float32 roundings: below 32 * 2^-23 + 8 * 2^-24
TOL = 4.5e-6


@pytest.mark.parametrize("d", [64, 72, 1032, 4104])
@pytest.mark.parametrize("n_txt", [1, 17, 64, 128, 129, 300])
def test_identity_scores_at_the_edges(d, n_txt):
    from paper_2605_02218_b200 import api, build
    from oracle import covspec_oracle as O
    build.build()
    ns = [1, 127, 128, 129, 300]
    ts = [max(1, n_txt - i) for i in range(len(ns))]
    wl = workloads.make_workload("identity", seed=d + n_txt, dtype=torch.bfloat16, batch=len(ns), sizes=(ns, ts), d=d,
                                 n_heads=0, rank=8, keep=1, act_layers=2)
    wl.X[1] = 0                                          # a zero token has cosine 0
    dev = wl.to("cuda:0")
    pr = api.Pruner.for_workload(dev)
    sq, _, _ = pr.score(pr.marshal(dev))
    pr.check_device_status()
    pr.close()
    got = [sq.cpu().numpy()]
    if int(wl.txt_offsets[-1]) * d <= api.STATIC_MAX_QUERY_ELEMS:
        got.append(api.query_score_static(dev.X, dev.Q, wl.vis_offsets, wl.txt_offsets).cpu().numpy())
    # more accumulation chunks than groups: the chains get longer in proportion
    chunks, cols = -(-d // 64), min(128, -(-max(ts) // 16) * 16)
    steps = 4 * -(-chunks // min(256 // (-(-cols // 32) * 32), -(-chunks // 8)))
    tol = max(TOL, steps * 2.0 ** -23 + 8 * 2.0 ** -24)
    for b in range(wl.batch):
        v0, v1, t0, t1 = (int(x) for x in (*wl.vis_offsets[b:b + 2], *wl.txt_offsets[b:b + 2]))
        want = O.query_relevance(wl.X[v0:v1].double().numpy(), wl.Q[t0:t1].double().numpy())
        for g in got:
            assert np.abs(g[v0:v1] - want).max() <= tol, (b, np.abs(g[v0:v1] - want).max())


def test_more_requests_than_one_launch_carries():
    from paper_2605_02218_b200 import api, build
    build.build()
    wl = workloads.make_workload("many", seed=3, dtype=torch.bfloat16, batch=150, n_vis=(3, 200), n_txt=(1, 9), d=64,
                                 n_heads=0, rank=4, keep=1, act_layers=0).to("cuda:0")
    pr = api.Pruner.for_workload(wl)
    sq, _, _ = pr.score(pr.marshal(wl))
    st = api.query_score_static(wl.X, wl.Q, wl.vis_offsets, wl.txt_offsets)
    # rows that start 8 bytes off a 16-byte boundary take the CUDA-core kernel: every score again
    off = lambda t: torch.cat([t.new_zeros(4), t.reshape(-1)])[4:].view(t.shape)
    simt = api.query_score_static(off(wl.X), off(wl.Q), wl.vis_offsets, wl.txt_offsets)
    torch.cuda.synchronize()
    assert torch.equal(sq, st)
    assert (sq - simt).abs().max().item() <= 2 * TOL
    pr.close()


def test_static_scores_are_nan_where_a_wait_gave_up():
    # the allocation-free entry point has no status word: a kernel that gave up must not leave the old contents behind
    import ctypes as C
    from paper_2605_02218_b200 import api, build
    build.build()
    wl = workloads.make_workload("timeout", seed=8, dtype=torch.bfloat16, batch=3, n_vis=(60, 300), n_txt=(1, 140), d=256,
                                 n_heads=0, rank=4, keep=1, act_layers=0).to("cuda:0")
    out = torch.full((wl.total_vis,), 7.0, device="cuda:0")
    ip = lambda a: a.ctypes.data_as(C.POINTER(C.c_int))
    vis, txt = (np.ascontiguousarray(a, dtype=np.int32) for a in (wl.vis_offsets, wl.txt_offsets))
    st = api.load_library().covspec_selftest_static_timeout(wl.d, wl.batch, wl.X.data_ptr(), ip(vis), wl.Q.data_ptr(), ip(txt),
                                                            out.data_ptr(), api._raw_stream())
    assert st == 0
    torch.cuda.synchronize()
    assert torch.isnan(out).all()
    again = api.query_score_static(wl.X, wl.Q, wl.vis_offsets, wl.txt_offsets)
    assert torch.isfinite(again).all()
