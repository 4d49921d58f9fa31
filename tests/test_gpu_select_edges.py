"""Top-k selections at the sizes where their form changes (1, 4 and 16 keys per thread, longer segments) and on
keys with ties, signed zeros and shared prefixes, through covspec_select, against the oracle's top_k."""
import numpy as np
import pytest
import torch

from paper_2605_02218_b200 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 4096, 4097, 16384, 16385, 20011])
def test_preselection_matches_top_k(n):
    from paper_2605_02218_b200 import api, build
    from oracle import covspec_oracle as O
    build.build()
    batch, rng = 5, np.random.default_rng(n)
    keep = [1, max(1, n // 7), max(1, n // 3), max(1, n - 1), n]
    wl = workloads.make_workload("select", seed=1, dtype=torch.bfloat16, batch=batch, n_vis=n, n_txt=1, d=64, n_heads=0,
                                 rank=4, keep=keep, act_layers=0).to("cuda:0")
    pr = api.Pruner.for_workload(wl, presel_factor=1.0)          # M = B_vis: the keep-set is the preselection
    m = pr.marshal(wl)
    scores = rng.standard_normal((batch, n)).astype(np.float32)
    scores[1] = np.round(scores[1] * 2) / 2                      # ties, both zeros
    scores[1][::3] = -0.0
    scores[2] = 1.0 + 1e-6 * scores[2]                           # a long shared prefix
    scores[3] = 0.25                                             # all equal
    keep_idx, ko, presel, po, _ = pr.select(m, torch.from_numpy(scores.reshape(-1)).cuda())
    pr.check_device_status()
    for b in range(batch):
        want = O.top_k(scores[b].astype(np.float64), keep[b])
        assert np.array_equal(presel.cpu().numpy()[po[b]:po[b + 1]], want)
        assert np.array_equal(keep_idx.cpu().numpy()[ko[b]:ko[b + 1]], want)
    pr.close()


@pytest.mark.parametrize("act_layers", [0, 2])
@pytest.mark.parametrize("n", [1, 33, 1023, 1024, 1025, 4096, 4097, 16384, 16385, 20011])
def test_fused_preselection_matches_the_separate_stages(n, act_layers):
    # the fused call normalises, fuses and selects in one kernel (keys in registers, beyond 16384 tokens through memory)
    from paper_2605_02218_b200 import api, build
    build.build()
    keep = [max(1, n // 7), max(1, n - 1), 1]
    wl = workloads.make_workload("fused", seed=n, dtype=torch.bfloat16, batch=3, n_vis=n, n_txt=3, d=64, n_heads=0, rank=4,
                                 keep=keep, act_layers=act_layers).to("cuda:0")
    for norm in ("minmax", "zscore", "none"):
        pr = api.Pruner.for_workload(wl, presel_factor=1.0, norm_mode=norm)       # M = B_vis: the keep-set is the preselection
        m = pr.marshal(wl)
        _, _, sf = pr.score(m)
        keep_idx, ko, _, _, _ = pr.select(m, sf)
        out, kept, ko2 = pr.prune(m)
        pr.check_device_status()
        assert np.array_equal(ko, ko2) and torch.equal(kept, keep_idx)
        assert torch.equal(out, pr.compact(m, keep_idx, ko)[0])
        pr.close()
