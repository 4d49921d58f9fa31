"""Parity of covspec_correct (through the C ABI) with the float64 oracle: margin, gate, acceptance
probability, residual mass and the drawn token, for the three logit types, vocabulary sizes that
are not multiples of the vector width, and the degenerate rows (identical distributions, ties)."""
import numpy as np
import pytest
import torch

from oracle import correction_oracle as C
from paper_2605_02218_b200 import workloads

pytestmark = pytest.mark.gpu

TOL = 2e-4        # float32 softmax sums over up to 152k terms against float64; relative to 1


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_02218_b200 import build
    build.build()


def _check(data, gamma, got, rows=None):
    margin, gate, accept, mass, token = [t.cpu().numpy() for t in got]
    zd = data["z_draft"].cpu().double().numpy()[:, :data["vocab"]]
    zt = data["z_target"].cpu().double().numpy()[:, :data["vocab"]]
    xs, ys = data["uniforms"].cpu().numpy(), data["drafted"].cpu().numpy()
    exact = 0
    for i in (range(data["rows"]) if rows is None else rows):
        ref = C.correct_position(zd[i], zt[i], float(xs[i]), gamma, y=int(ys[i]))
        assert abs(margin[i] - ref["margin"]) <= TOL, (i, margin[i], ref["margin"])
        if abs(ref["margin"] - gamma) > TOL:
            assert gate[i] == ref["gate"]
        assert abs(accept[i] - ref["accept"]) <= TOL * max(1.0, ref["accept"]) + 2e-3 * ref["accept"]
        assert abs(mass[i] - ref["resid_mass"]) <= TOL
        tk, cdf, x = int(token[i]), ref["cdf"], float(xs[i])
        assert 0 <= tk < data["vocab"]
        # the token is the oracle's, or the uniform number sits within the tolerance of a step of the
        # oracle's cumulative distribution between the two
        assert cdf[tk] > x - TOL and (tk == 0 or cdf[tk - 1] <= x + TOL), (i, tk, ref["token"])
        assert cdf[tk] - (cdf[tk - 1] if tk else 0.0) > 0.0          # never a zero-probability token
        exact += tk == ref["token"]
    return exact


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vocab", [2, 37, 1000, 5003, 40000])
def test_small_vocabularies(dtype, vocab):
    from paper_2605_02218_b200 import api
    data = workloads.make_logits(seed=vocab, rows=24, vocab=vocab, dtype=dtype, device="cuda:0")
    got = api.correct(data["z_draft"], data["z_target"], data["uniforms"], 0.05, data["drafted"], vocab=vocab)
    torch.cuda.synchronize()
    exact = _check(data, 0.05, got)
    assert exact >= 22


def test_full_vocabulary_sampled_rows():
    from paper_2605_02218_b200 import api
    data = workloads.make_logits(seed=7, rows=512, vocab=151674, dtype=torch.float16, device="cuda:0")
    got = api.correct(data["z_draft"], data["z_target"], data["uniforms"], 0.02, data["drafted"], vocab=151674)
    torch.cuda.synchronize()
    exact = _check(data, 0.02, got, rows=[0, 1, 100, 255, 511])
    assert exact >= 4


def test_degenerate_rows():
    from paper_2605_02218_b200 import api
    vocab = 96
    data = workloads.make_logits(seed=3, rows=6, vocab=vocab, dtype=torch.float32, device="cuda:0")
    zd, zt = data["z_draft"], data["z_target"]
    zt[0] = zd[0]                                    # identical distributions: draw from p_t
    zd[1, :vocab] = 0.0                              # uniform draft: tie for the top, margin 0
    zd[2, :vocab] = -30.0; zd[2, 5] = 30.0           # one-hot draft: margin 1
    zt[3, :vocab] = -30.0; zt[3, 95] = 30.0          # one-hot target on the last token
    data["uniforms"][4] = 0.0
    data["uniforms"][5] = 0.99999994
    got = api.correct(zd, zt, data["uniforms"], 0.5, data["drafted"], vocab=vocab)
    torch.cuda.synchronize()
    _check(data, 0.5, got)
    margin, gate, accept, mass, token = [t.cpu().numpy() for t in got]
    assert mass[0] == 0.0 and margin[1] == 0.0 and gate[1] == 1
    assert margin[2] > 0.999 and gate[2] == 0 and token[3] == 95


def test_argument_errors():
    from paper_2605_02218_b200 import api
    z = torch.zeros(2, 12, dtype=torch.float16, device="cuda:0")          # 24-byte rows
    u = torch.zeros(2, device="cuda:0")
    with pytest.raises(api.CovspecError) as e:
        api.correct(z, z, u, 0.1)
    assert e.value.status == -2


def test_missing_random_numbers_are_an_argument_error():
    from paper_2605_02218_b200 import api
    z = torch.zeros(2, 16, dtype=torch.float16, device="cuda:0")
    with pytest.raises(api.CovspecError) as e:
        api.correct(z, z, None, 0.1)
    assert e.value.status == -1


def test_every_result_of_a_correction_has_memory_of_its_own():
    # kept or passed on by itself: no result holds another one's memory, each base is aligned for vector loads
    from paper_2605_02218_b200 import api
    data = workloads.make_logits(seed=6, rows=3, vocab=1000, dtype=torch.float16, device="cuda:0")
    got = api.correct(data["z_draft"], data["z_target"], data["uniforms"], 0.05, data["drafted"], vocab=1000)
    assert len({t.untyped_storage().data_ptr() for t in got}) == len(got)
    for t in got:
        assert t.untyped_storage().nbytes() == 4 * 3 and t._base is None and t.data_ptr() % 16 == 0


@pytest.mark.parametrize("dtype", [torch.float16, torch.float32])
def test_branch_candidates(dtype):
    from paper_2605_02218_b200 import api
    for vocab, rows in [(37, 6), (5003, 8), (151674, 4)]:
        data = workloads.make_logits(seed=vocab + 1, rows=rows, vocab=vocab, dtype=dtype, device="cuda:0")
        fan = [api.fanout(8, 0.6, j) for j in range(rows)]
        assert fan == [C.fanout(8, 0.6, j) for j in range(rows)]
        if vocab == 5003:
            fan[0] = 1500                                         # beyond the direct-ranking size
        cand, off = api.branch_candidates(data["z_draft"], fan, data["drafted"], vocab=vocab)
        torch.cuda.synchronize()
        cand = cand.cpu().numpy()
        zd = data["z_draft"].cpu().double().numpy()[:, :vocab]
        ys = data["drafted"].cpu().numpy()
        for i in range(rows):
            want = C.bonus_candidates(zd[i], int(ys[i]), min(fan[i], vocab - 1))
            assert np.array_equal(cand[off[i]:off[i + 1]], want), (vocab, i)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vocab,rows,fan", [(16384, 3, 64), (16391, 2, 64), (32767, 520, 3), (40961, 5, 1), (151674, 4, 65)])
def test_branch_candidates_at_the_limits_of_the_cluster_kernel(dtype, vocab, rows, fan):
    # shortest rows and largest fan-out the cluster kernel takes, ragged ends, more rows than one launch
    # carries, one past the largest fan-out; mass ties (more entries at the threshold than are ranked
    # directly), the largest entry drafted, the last entry drafted
    from paper_2605_02218_b200 import api
    data = workloads.make_logits(seed=vocab, rows=rows, vocab=vocab, dtype=dtype, device="cuda:0")
    z, y = data["z_draft"], data["drafted"]
    y[0] = int(z[0, :vocab].float().argmax())
    if rows > 1:
        z[1, :vocab] = z[1, :vocab].clamp(-1, 1)
        y[1] = vocab - 1
    fans = [max(0, fan - i % 3) for i in range(rows)]
    cand, off = api.branch_candidates(z, fans, y, vocab=vocab)
    torch.cuda.synchronize()
    cand = cand.cpu().numpy()
    for i in sorted({0, 1, rows // 2, rows - 1} & set(range(rows))):
        want = C.bonus_candidates(z[i, :vocab].cpu().double().numpy(), int(y[i]), fans[i])
        assert np.array_equal(cand[off[i]:off[i + 1]], want), i


@pytest.mark.parametrize("rows", [1, 37, 38, 74, 75])
def test_result_of_a_position_does_not_depend_on_the_call_size(rows):
    # 8, 4 or 2 CTAs share a position, by the number of positions of the call; every split adds its sums
    # up in the same order, so a position gives the same bits in a call of 160 positions as in a small one;
    # a spread-out row makes the running reference of the sums move in the middle of a segment
    from paper_2605_02218_b200 import api
    vocab = 40013
    data = workloads.make_logits(seed=5, rows=160, vocab=vocab, dtype=torch.float32, device="cuda:0")
    data["z_draft"][0, 20000:vocab] += 200.0
    data["z_target"][min(36, rows - 1), 30000:vocab] += 150.0
    args = lambda n: (data["z_draft"][:n], data["z_target"][:n], data["uniforms"][:n], 0.05, data["drafted"][:n])
    whole = api.correct(*args(160), vocab=vocab)
    part = api.correct(*args(rows), vocab=vocab)
    torch.cuda.synchronize()
    for a, b in zip(whole, part):
        assert torch.equal(a[:rows], b)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rows", [1, 16, 17, 32, 33])
def test_call_size_at_the_limits_of_the_cluster_sizes(rows, dtype):
    # the same for all logit types at the limits of the 8, 4 and 2 CTAs per position, a vocabulary that ends inside a vector
    from paper_2605_02218_b200 import api
    vocab = 40013
    data = workloads.make_logits(seed=9, rows=160, vocab=vocab, dtype=dtype, device="cuda:0")
    data["z_draft"][rows - 1, 20000:vocab] += 200.0
    args = lambda n: (data["z_draft"][:n], data["z_target"][:n], data["uniforms"][:n], 0.05, data["drafted"][:n])
    whole = api.correct(*args(160), vocab=vocab)
    part = api.correct(*args(rows), vocab=vocab)
    torch.cuda.synchronize()
    for a, b in zip(whole, part):
        assert torch.equal(a[:rows], b)


@pytest.mark.parametrize("dtype,value", [(torch.float16, None), (torch.bfloat16, None), (torch.float32, None),
                                         (torch.float32, -1e30), (torch.float32, -1e9), (torch.float16, -np.inf)])
@pytest.mark.parametrize("rows", [2, 24, 40])
def test_masked_logits(dtype, value, rows):
    # most of the vocabulary masked in both rows (None: the type's lowest value), the beginning of the row included;
    # one row unmasked in the draft with the drafted token masked in the target
    from paper_2605_02218_b200 import api
    vocab = 20011
    value = torch.finfo(dtype).min if value is None else value
    data = workloads.make_logits(seed=11, rows=rows, vocab=vocab, dtype=dtype, device="cuda:0")
    zd, zt = data["z_draft"], data["z_target"]
    allowed = torch.zeros(vocab, dtype=torch.bool, device="cuda:0")
    allowed[torch.arange(50, vocab, 701)] = True
    plain = zd[1].clone()
    zd[:, :vocab][:, ~allowed] = value
    zt[:, :vocab][:, ~allowed] = value
    zd[1] = plain
    data["drafted"][:] = 50 + 701 * 3
    data["drafted"][1] = 7
    got = api.correct(zd, zt, data["uniforms"], 0.05, data["drafted"], vocab=vocab)
    torch.cuda.synchronize()
    _check(data, 0.05, got)
    assert all(bool(allowed[t]) for t in got[4].tolist())


def test_branch_candidates_beyond_the_stated_fan_out():
    # device offsets that ask one position for more than max_fanout says: every position gets what its offsets ask for
    from paper_2605_02218_b200 import api
    lib, vocab, fans = api.load_library(), 40000, [4, 65, 200, 0, 1500, 8]
    data = workloads.make_logits(seed=13, rows=len(fans), vocab=vocab, dtype=torch.float16, device="cuda:0")
    off = np.concatenate([[0], np.cumsum(fans)]).astype(np.int32)
    d_off = torch.from_numpy(off).cuda()
    cand = torch.full((int(off[-1]),), -1, dtype=torch.int32, device="cuda:0")
    st = lib.covspec_branch_candidates(api.COVSPEC_F16, len(fans), vocab, data["ld"], data["z_draft"].data_ptr(),
                                       data["drafted"].data_ptr(), d_off.data_ptr(), 8, cand.data_ptr(), api._raw_stream())
    assert st == 0
    torch.cuda.synchronize()
    cand = cand.cpu().numpy()
    for i, f in enumerate(fans):
        want = C.bonus_candidates(data["z_draft"][i, :vocab].cpu().double().numpy(), int(data["drafted"][i]), f)
        assert np.array_equal(cand[off[i]:off[i + 1]], want), i
    with pytest.raises(api.CovspecError) as e:
        api.branch_candidates(data["z_draft"], [2, -1, 3, 0, 1, 1], data["drafted"], vocab=vocab)
    assert e.value.status == -2


@pytest.mark.parametrize("vocab", [5003, 40013])
def test_drafted_token_is_no_candidate_among_masked_ones(vocab):
    # fewer unmasked tokens than candidates: the rest are masked ones by their ids, never the drafted token
    from paper_2605_02218_b200 import api
    data = workloads.make_logits(seed=15, rows=2, vocab=vocab, dtype=torch.float16, device="cuda:0")
    z, y = data["z_draft"], data["drafted"]
    z[:, 4:vocab] = -np.inf
    y[0], y[1] = 6, 2
    cand, off = api.branch_candidates(z, [9, 9], y, vocab=vocab)
    torch.cuda.synchronize()
    for i in range(2):
        want = C.bonus_candidates(z[i, :vocab].cpu().double().numpy(), int(y[i]), 9)
        assert np.array_equal(cand.cpu().numpy()[off[i]:off[i + 1]], want), i


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vocab", [16390, 40013])
def test_branch_candidates_among_mass_ties(dtype, vocab):
    # rows whose F_j-th largest logit is shared by most of the row: masked down to a few tokens (-inf and the type's lowest
    # value; the drafted token among them or among the masked ones), one value throughout, ties only at the end,
    # and more entries above the ties than are ranked directly (bunched, and rising to the end of the row)
    from paper_2605_02218_b200 import api
    rows = 8
    data = workloads.make_logits(seed=14, rows=rows, vocab=vocab, dtype=dtype, device="cuda:0")
    z, y = data["z_draft"], data["drafted"]
    allowed = torch.zeros(vocab, dtype=torch.bool, device="cuda:0")
    allowed[[3, 9000, 9001, vocab - 1]] = True
    for i, value in enumerate((-np.inf, torch.finfo(dtype).min, -np.inf)):
        z[i, :vocab][~allowed] = value
    y[0], y[1], y[2] = 9000, 5, 0
    z[3, :vocab] = 1.5
    y[3] = 0
    z[4, :vocab] = -2.0
    z[4, vocab - 3000:vocab] = 4.0
    z[4, 17] = 5.0
    z[5, :vocab] = 0.0
    z[5, 100:2500] = torch.linspace(1, 9, 2400, device="cuda:0").to(dtype)
    stride = torch.arange(vocab, device="cuda:0") % 32768 < (256 if dtype != torch.float32 else 128)
    z[6, :vocab] = torch.where(stride, 2.0 + torch.rand(vocab, device="cuda:0"), torch.zeros(vocab, device="cuda:0")).to(dtype)
    z[7, :vocab] = 0.0
    z[7, vocab - 9000:vocab] = torch.linspace(1, 9, 9000, device="cuda:0").to(dtype)
    for fan in (1, 3, 4, 32, 64):
        cand, off = api.branch_candidates(z, [fan] * rows, y, vocab=vocab)
        torch.cuda.synchronize()
        cand = cand.cpu().numpy()
        for i in range(rows):
            want = C.bonus_candidates(z[i, :vocab].cpu().double().numpy(), int(y[i]), fan)
            assert np.array_equal(cand[off[i]:off[i + 1]], want), (i, fan)


@pytest.mark.parametrize("dtype,vocab", [(torch.float32, 200003), (torch.float32, 420001), (torch.float16, 420001)])
def test_rows_too_long_for_sums_in_shared_memory(dtype, vocab):
    # the largest rows of the cluster sizes: fewer CTAs per position than the call's size asks for, and no kept sums
    from paper_2605_02218_b200 import api
    data = workloads.make_logits(seed=17, rows=160, vocab=vocab, dtype=dtype, device="cuda:0")
    args = lambda n: (data["z_draft"][:n], data["z_target"][:n], data["uniforms"][:n], 0.05, data["drafted"][:n])
    whole = api.correct(*args(160), vocab=vocab)
    for rows in (1, 24):
        for a, b in zip(whole, api.correct(*args(rows), vocab=vocab)):
            assert torch.equal(a[:rows], b)
    torch.cuda.synchronize()
    _check(data, 0.05, whole, rows=[0, 1, 159])
