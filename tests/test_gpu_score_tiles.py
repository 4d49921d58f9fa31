"""Relevance kernel and Gram kernel at the edges of their work split: pairs of token tiles (odd numbers of tiles, pairs
that belong to two requests), logits tiles of up to 128 query elements, items of one and two heads, the shared columns of the Gram items, CTAs with many row tiles."""
import numpy as np
import pytest
import torch

from paper_2605_02218_b200 import api, workloads
from tests import parity

pytestmark = pytest.mark.gpu


def _workload(name, n, t, **kw):
    kw = dict(dict(seed=5, dtype=torch.bfloat16, rank=8, keep_ratio=0.2, act_layers=1, device="cuda:0"), **kw)
    return workloads.make_workload(name, batch=len(n), sizes=(n, t), **kw)


def _query_scores(wl, path):
    pr = api.Pruner.for_workload(wl, relevance_path=path)
    s = pr.score(pr.marshal(wl))[0].cpu().numpy()
    status = pr.device_status()
    pr.close()
    return s, status


@pytest.mark.parametrize("n,t,heads,d", [
    ([129], [1], 1, 64),                                            # a pair whose second tile has one row; one logit
    ([100], [32], 2, 64),                                           # one tile: the pair's second CTA has none
    ([128, 1, 300], [32, 33, 65], 3, 72),                           # pairs of two requests, a lone last head, a partial chunk
    ([130, 257, 64, 500, 127], [1, 128, 129, 300, 64], 2, 200),     # logits tiles of every width, up to three of them
    ([128 * 151 + 5], [40], 1, 64),                                 # more single-head items than clusters
    ([576], [31], 16, 2048),                                        # one item per cluster; a query tile of 31 rows
    ([700] * 9, [96, 97, 2, 64, 31, 160, 7, 128, 255], 7, 328),     # several items per cluster
    ([100, 90, 128, 77, 5, 60], [16, 16, 1, 15, 17, 31], 2, 128),   # pairs of two requests: columns from 16, 1 and 17 on
    ([100, 90, 128, 77, 5, 60, 9], [100, 100, 127, 2, 128, 129, 64], 3, 72),   # a request's columns in two logits tiles
    ([60] * 160, [33] * 160, 1, 64),                                # every pair of two requests, several items per cluster
])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_query_scores_against_the_cuda_core_kernels(n, t, heads, d, dtype):
    wl = _workload("tiles", n, t, d=d, n_heads=heads, dtype=dtype)
    got, st = _query_scores(wl, 0)
    want, _ = _query_scores(wl, 1)
    assert st == 0
    # hi + lo operands of both products (2^-16 each) and the sums of d / 16 truncating steps, which a projected feature's
    # cancellation magnifies
    tol = 2.0 ** -15 + d / 16 * 2.0 ** -23 * 8
    assert np.abs(got - want).max() <= tol


def test_restaged_heads_are_complete_when_the_other_sm_multiplies_them():
    # the leader of a pair multiplies shared memory that its peer's threads have written: with several items and heads per
    # cluster the same tiles are overwritten again and again, and a product of a half-written one would change a score
    wl = _workload("restaged", [700] * 9, [96, 97, 2, 64, 31, 160, 7, 128, 255], d=72, n_heads=12)
    pr = api.Pruner.for_workload(wl)
    m = pr.marshal(wl)
    first = pr.score(m)[0]
    for _ in range(100):
        assert torch.equal(first, pr.score(m)[0])
    pr.close()


@pytest.mark.parametrize("where", [0, 40, 70, 99])
def test_a_query_element_that_is_not_finite_is_reported(where):
    wl = _workload("nan", [200, 40], [100, 3], d=128, n_heads=1)
    wl.Q[where, 5] = float("nan")
    assert _query_scores(wl, 0)[1] == -6
    assert _query_scores(wl, 1)[1] == -6


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("batch", [1, 37, 38, 74, 75])
def test_gram_items_with_shared_columns(batch, dtype):
    # one 128 x 128 item per request: four CTAs an item up to 37, two up to 74, then one
    wl = workloads.make_workload(f"gram{batch}", seed=31, dtype=dtype, batch=batch, n_vis=200, n_txt=3, d=136, n_heads=1,
                                 rank=8, keep=[64] * batch, act_layers=1)
    parity.run_gpu(wl, requests=sorted({0, batch // 2, batch - 1}))


@pytest.mark.parametrize("m", [130, 256, 300, 420])
def test_gram_items_of_several_tiles_with_shared_columns(m):
    wl = workloads.make_workload(f"gram-m{m}", seed=32, dtype=torch.bfloat16, batch=2, n_vis=m + 40, n_txt=3, d=200, n_heads=1,
                                 rank=8, keep=[m // 2] * 2, act_layers=1)
    parity.run_gpu(wl)


def test_more_row_tiles_per_cta_than_are_looked_up_in_advance():
    # 2500 requests of one row tile each on 148 CTAs: 17 tiles per CTA, the last one looked up when its turn comes
    wl = workloads.make_workload("many-tiles-per-cta", seed=33, dtype=torch.bfloat16, batch=2500, n_vis=(40, 90), n_txt=1, d=64,
                                 n_heads=1, rank=4, keep_ratio=0.2, act_layers=1)
    parity.run_gpu(wl, requests=[0, 1, 777, 1480, 2110, 2400, 2499])


@pytest.mark.parametrize("layers,n,d", [(4, 16384, 2048),      # long enough for the stream to follow the relevance kernel
                                        (10, 700, 256), (6, 3000, 1024), (4, 300, 264), (1, 5, 64), (8, 4800, 1336),
                                        (16, 129, 520)])
def test_activity_is_the_same_wherever_it_runs(layers, n, d):
    wl = _workload("activity", [n], [9], d=d, n_heads=1, act_layers=layers)
    got = []
    for overlap in (0, 1, 2):
        pr = api.Pruner.for_workload(wl, activity_overlap=overlap)
        got.append([t.clone() for t in pr.score(pr.marshal(wl))])
        assert pr.device_status() == 0
        pr.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert torch.equal(a, b)

