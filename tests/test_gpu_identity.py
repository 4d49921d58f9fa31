"""Eq. 10 with the identity embedding on the tensor cores (bf16): sizes at the edges of its tiles, passes
and accumulation groups, against the oracle's definition in float64, through both entry points."""
import numpy as np
import pytest
import torch

from paper_2605_02218_b200 import workloads

pytestmark = pytest.mark.gpu

# bf16 products are exact in float32; a lane adds up at most 129 of them (d = 4104), five additions join the lanes, a few
# roundings make up the lengths: each below 2^-24 of at most |x| |q|
TOL = 140 * 2.0 ** -24


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
    for b in range(wl.batch):
        v0, v1, t0, t1 = (int(x) for x in (*wl.vis_offsets[b:b + 2], *wl.txt_offsets[b:b + 2]))
        want = O.query_relevance(wl.X[v0:v1].double().numpy(), wl.Q[t0:t1].double().numpy())
        for g in got:
            assert np.abs(g[v0:v1] - want).max() <= TOL, (b, np.abs(g[v0:v1] - want).max())


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


def _both_routes(wl):
    """Query scores on the tensor cores and on the CUDA cores (relevance_path = 1)."""
    from paper_2605_02218_b200 import api
    out = []
    for path in (0, 1):
        pr = api.Pruner.for_workload(wl, relevance_path=path)
        out.append(pr.score(pr.marshal(wl))[0])
        pr.device_status()                               # scores that are not finite are reported there as well
        pr.close()
    return out


@pytest.mark.parametrize("d", [64, 72, 520, 1032, 2048, 4096])
@pytest.mark.parametrize("n_txt", [1, 17, 100, 128, 129, 300])
def test_identity_scores_have_the_bits_of_the_cuda_core_kernel(d, n_txt):
    # candidates come from truncating sums, the scores from float32 sums in one fixed order: no less precise than the
    # CUDA-core kernel, at any width and query length
    from paper_2605_02218_b200 import api, build
    build.build()
    ns = [1, 127, 128, 129, 1100]
    ts = [max(1, n_txt - i) for i in range(len(ns))]
    wl = workloads.make_workload("identity", seed=d + n_txt, dtype=torch.bfloat16, batch=len(ns), sizes=(ns, ts), d=d,
                                 n_heads=0, rank=8, keep=1, act_layers=0).to("cuda:0")
    tc, simt = _both_routes(wl)
    assert torch.equal(tc, simt)
    if int(wl.txt_offsets[-1]) * d <= api.STATIC_MAX_QUERY_ELEMS:
        assert torch.equal(api.query_score_static(wl.X, wl.Q, wl.vis_offsets, wl.txt_offsets), simt)


def test_identity_scores_of_unusual_rows():
    # many candidates (repeated query elements, all of them alike, tokens along a query element), zero and tiny rows on either
    # side (products below the float32 range), rows that are not finite or whose length is not
    from paper_2605_02218_b200 import build
    build.build()
    d, ns, ts = 1024, [300, 200, 260, 200, 130, 140], [40, 200, 9, 64, 30, 150]
    wl = workloads.make_workload("unusual", seed=3, dtype=torch.bfloat16, batch=len(ns), sizes=(ns, ts), d=d, n_heads=0,
                                 rank=8, keep=1, act_layers=0).to("cuda:0")
    v, t = [int(a) for a in wl.vis_offsets], [int(a) for a in wl.txt_offsets]
    X, Q = wl.X, wl.Q
    Q[t[0] + 5:t[0] + 12] = Q[t[0] + 4]                  # repeated
    X[v[0]:v[0] + 50] = Q[t[0] + 4] * 3
    Q[t[1]:t[2]] = Q[t[1]]                               # all alike, over two passes
    X[v[2] + 3] = 0
    X[v[2] + 4] *= 1e-21
    X[v[2] + 5:v[2] + 9] *= 2e-20
    X[v[2] + 9:v[2] + 40] *= 1e-18
    Q[t[2]] = 0
    Q[t[2] + 1] *= 1e-21
    Q[t[2] + 2:t[2] + 9] *= 1e-18
    X[v[3] + 7, 11] = float("nan")
    X[v[3] + 8, 0] = float("inf")
    X[v[3] + 9] = 3e38
    X[v[3] + 10:v[3] + 20] *= 1e16
    Q[t[3]:t[3] + 4] *= 1e16
    Q[t[4] + 3, 5] = float("nan")                        # the whole request
    Q[t[5] + 140, 9] = float("-inf")
    tc, simt = _both_routes(wl)
    assert torch.equal(torch.isnan(tc), torch.isnan(simt))
    assert int(torch.isnan(tc).sum()) == 3 + ns[4] + ns[5]
    assert torch.equal(torch.nan_to_num(tc), torch.nan_to_num(simt))


def test_identity_scores_do_not_depend_on_the_batch():
    # a request alone, and beside one with a much longer query and with enough tokens for whole 128-token tiles
    from paper_2605_02218_b200 import api, build
    build.build()
    d, ns, ts = 4096, [333, 20000], [30, 250]
    wl = workloads.make_workload("batch", seed=4, dtype=torch.bfloat16, batch=2, sizes=(ns, ts), d=d, n_heads=0, rank=8,
                                 keep=1, act_layers=0).to("cuda:0")
    both = _both_routes(wl)[0][:ns[0]]
    alone = api.query_score_static(wl.X[:ns[0]], wl.Q[:ts[0]], wl.vis_offsets[:2], wl.txt_offsets[:2])
    assert torch.equal(both, alone)


def test_identity_scores_with_more_query_rows_than_a_pair_code_holds():
    # up to 16384 query rows a token hands on two candidates, beyond only one; three and more stay where they were found
    from paper_2605_02218_b200 import build
    build.build()
    batch, t, d = 129, 128, 64
    wl = workloads.make_workload("many-queries", seed=5, dtype=torch.bfloat16, batch=batch, sizes=([40] * batch, [t] * batch),
                                 d=d, n_heads=0, rank=4, keep=1, act_layers=0).to("cuda:0")
    for b in range(0, batch, 3):
        q0, x0 = int(wl.txt_offsets[b]), int(wl.vis_offsets[b])
        wl.Q[q0 + 100:q0 + 100 + b % 4] = wl.Q[q0 + 3]       # none, one, two or three repetitions
        wl.X[x0:x0 + 20] = wl.Q[q0 + 3] * 2
    assert int(wl.txt_offsets[-1]) > 1 << 14
    for n in (batch, 128):                                    # 16512 and 16384 rows
        part = workloads.Workload(**{**wl.__dict__, "vis_offsets": wl.vis_offsets[:n + 1], "txt_offsets": wl.txt_offsets[:n + 1],
                                     "keep": wl.keep[:n], "X": wl.X[:40 * n], "Q": wl.Q[:t * n]})
        tc, simt = _both_routes(part)
        assert torch.equal(tc, simt)
