"""GPU-vs-oracle parity of the token-chunked linear cross-entropy, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import linear_ce_oracle as lce
from paper_2609_19242_b200 import binding, synth
from paper_2609_19242_b200.synth import LceWorkload

pytestmark = pytest.mark.gpu

# bf16 inputs, fp32 accumulation and fp32 softmax statistics; dz rounded to bf16 before the gradient products
TOL_LSE = 1e-3        # max |lse - oracle|, as for the attention layer's LSE
TOL_NLL = 2e-3        # max |nll - oracle| (lse and the target logit each carry fp32 accumulation error)
TOL_LOSS_REL = 1e-4   # |loss - oracle| / |oracle|
TOL_GRAD = 2e-2       # relative L2 of dH and dW


def _rel(got, ref):
    return float(np.linalg.norm((got - ref).ravel()) / max(np.linalg.norm(ref.ravel()), 1e-300))


def _check(w, token_chunk=0, weighted=True, grad_loss=1.0):
    inp = synth.make_lce_inputs(w, "cpu")
    g = {k: v.cuda() for k, v in inp.items()}
    tw = g["weight"] if weighted else None
    loss, nll, lse = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], tw)
    dh, dw = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, tw, grad_loss=grad_loss, token_chunk=token_chunk)
    torch.cuda.synchronize()
    assert binding.bdlm_get_device_status() == 0
    h64, w64 = synth.to_f64(inp["h"]), synth.to_f64(inp["w"])
    y = inp["labels"].numpy()
    wt = inp["weight"].double().numpy() if weighted else None
    ref_loss, ref_nll, ref_lse = lce.linear_ce_forward(h64, w64, y, wt, token_chunk=97)
    ref_dh, ref_dw = lce.linear_ce_backward(h64, w64, y, wt, grad_loss=grad_loss, token_chunk=97)
    assert np.abs(synth.to_f64(lse) - ref_lse).max() <= TOL_LSE
    assert np.abs(synth.to_f64(nll) - ref_nll).max() <= TOL_NLL
    assert abs(float(loss) - ref_loss) <= TOL_LOSS_REL * abs(ref_loss)
    got_dh, got_dw = synth.to_f64(dh), synth.to_f64(dw)
    assert np.isfinite(got_dh).all() and np.isfinite(got_dw).all()
    assert _rel(got_dh, ref_dh) <= TOL_GRAD, _rel(got_dh, ref_dh)
    assert _rel(got_dw, ref_dw) <= TOL_GRAD, _rel(got_dw, ref_dw)
    ign = y < 0
    if ign.any():
        assert np.abs(got_dh[ign]).max() == 0.0 and np.abs(synth.to_f64(nll)[ign]).max() == 0.0
    return loss, nll, lse, dh, dw


@pytest.mark.parametrize("w", [
    LceWorkload("one_tile", 128, 64, 256),
    LceWorkload("tiny", 200, 64, 1000),                       # ragged token tile and ragged vocabulary tile
    LceWorkload("several_tiles", 400, 192, 2568),             # several vocabulary runs (> 8 tiles of 256), K not a multiple of 64
    LceWorkload("wide", 300, 520, 776, logit_std=4.0),        # D beyond one 256-column N tile in the gradient products
    LceWorkload("one_token", 1, 64, 512),
], ids=lambda w: w.name)
def test_matches_oracle(w):
    _check(w)


def test_token_chunks_accumulate_dw_in_fp32_and_agree_with_one_chunk():
    w = LceWorkload("chunks", 600, 128, 1544)
    one = _check(w, token_chunk=0)
    three = _check(w, token_chunk=256, grad_loss=1.0)          # 256 + 256 + 88 tokens
    many = _check(w, token_chunk=128)                          # five chunks, the last one ragged
    assert torch.equal(one[3], three[3]) and torch.equal(one[3], many[3])   # dH rows do not depend on the chunking
    for other in (three, many):
        assert _rel(synth.to_f64(other[4]), synth.to_f64(one[4])) <= 4e-3   # dW: other fp32 summation order, one bf16 rounding


def test_unweighted_and_scaled_gradient():
    _check(LceWorkload("plain", 256, 64, 512), weighted=False, grad_loss=-0.37)


def test_results_are_bitwise_reproducible():
    w = LceWorkload("repro", 384, 128, 2048)
    inp = {k: v.cuda() for k, v in synth.make_lce_inputs(w, "cpu").items()}
    runs = []
    for _ in range(2):
        loss, nll, lse = binding.bdlm_linear_ce_fwd(inp["h"], inp["w"], inp["labels"], inp["weight"])
        dh, dw = binding.bdlm_linear_ce_bwd(inp["h"], inp["w"], inp["labels"], lse, inp["weight"], token_chunk=128)
        runs.append([t.clone() for t in (loss, nll, lse, dh, dw)])
    torch.cuda.synchronize()
    for a, b in zip(*runs):
        assert torch.equal(a, b)


def test_full_size_sampled_tokens():
    """The benchmark's size (8192 tokens, D = 4096, V = 128256): lse and nll of 64 sampled tokens against the oracle;
    dH rows of those tokens against the oracle (a token's dH depends on that token only); dW through linearity: a
    second backward whose weights are zero outside the sample is compared with the oracle's sum over the sample."""
    w = synth.LCE_WORKLOADS["lce_8k"]
    g = synth.make_lce_inputs(w, "cuda")
    loss, nll, lse = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"])
    rng = np.random.default_rng(3)
    rows = np.unique(np.concatenate([[0, 127, 128, 4095, 4096, w.T - 1], rng.choice(w.T, size=58, replace=False)]))
    rt = torch.from_numpy(rows).cuda()
    w_sp = torch.zeros_like(g["weight"])
    w_sp[rt] = g["weight"][rt]
    dh, _ = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, g["weight"], token_chunk=2048)
    _, dw_sp = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, w_sp, token_chunk=4096)
    torch.cuda.synchronize()
    assert binding.bdlm_get_device_status() == 0
    W64 = synth.to_f64(g["w"])
    h_rows = synth.to_f64(g["h"][rt])
    y_rows = g["labels"][rt].cpu().numpy()
    wt_rows = g["weight"][rt].double().cpu().numpy()
    ref_nll, ref_lse = lce.linear_ce_rows(h_rows, W64, y_rows)
    assert np.abs(synth.to_f64(lse[rt]) - ref_lse).max() <= TOL_LSE
    assert np.abs(synth.to_f64(nll[rt]) - ref_nll).max() <= TOL_NLL
    ref_dh, ref_dw = lce.linear_ce_backward(h_rows, W64, y_rows, wt_rows, token_chunk=16)
    assert _rel(synth.to_f64(dh[rt]), ref_dh) <= TOL_GRAD
    assert _rel(synth.to_f64(dw_sp), ref_dw) <= TOL_GRAD
    # the scalar loss against the per-token values the kernel itself wrote (the sum is the only new arithmetic here)
    want = float((g["weight"].double() * nll.double()).sum())
    assert abs(float(loss) - want) <= 1e-5 * abs(want)


def test_all_positions_ignored_gives_zero_loss_and_zero_gradients():
    w = LceWorkload("all_ignored", 130, 64, 520)
    inp = {k: v.cuda() for k, v in synth.make_lce_inputs(w, "cpu").items()}
    labels = torch.full_like(inp["labels"], -1)
    loss, nll, lse = binding.bdlm_linear_ce_fwd(inp["h"], inp["w"], labels, None)
    dh, dw = binding.bdlm_linear_ce_bwd(inp["h"], inp["w"], labels, lse, None)
    torch.cuda.synchronize()
    assert float(loss) == 0.0 and float(nll.abs().max()) == 0.0
    assert float(dh.float().abs().max()) == 0.0 and float(dw.float().abs().max()) == 0.0
    ref = lce.linear_ce_forward(synth.to_f64(inp["h"]), synth.to_f64(inp["w"]), labels.cpu().numpy())
    assert np.abs(synth.to_f64(lse) - ref[2]).max() <= TOL_LSE


@pytest.mark.parametrize("w", [
    LceWorkload("split_contraction", 150, 72, 8200),           # few dH tiles, each a long contraction
    LceWorkload("narrow_tiles", 520, 264, 9000),               # D one tile and 8 columns: tiles narrower than 256
    LceWorkload("odd_half_chunks", 390, 512, 5000),            # 144-column tiles: the last 32-column chunk reaches past them
    LceWorkload("many_short_runs", 260, 64, 20008),            # 79 vocabulary runs with a full workspace, 10 with the smallest
], ids=lambda w: w.name)
def test_tilings_and_split_contraction(w):
    one = _check(w)
    # dH does not depend on the token chunks; the smallest accepted workspace has longer runs and no copies
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(w, "cpu").items()}
    dh, _ = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], one[2], g["weight"], token_chunk=128)
    assert torch.equal(dh, one[3])
    per = (w.T * 4 + 255) // 256 * 256
    runs = (((w.V + 255) // 256) + 7) // 8
    least = torch.empty((2 * runs + 1) * per + 256, dtype=torch.uint8, device="cuda")
    loss, nll, lse = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"], workspace=least)
    least = torch.empty((w.T + 127) // 128 * 128 * w.V * 2, dtype=torch.uint8, device="cuda")
    dh, dw = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, g["weight"], workspace=least)
    torch.cuda.synchronize()
    assert float((lse - one[2]).abs().max()) <= TOL_LSE and abs(float(loss) - float(one[0])) <= TOL_LOSS_REL * abs(float(one[0]))
    # another order of the fp32 sums, then one bf16 rounding (2^-9 of an element where it falls the other way)
    assert _rel(synth.to_f64(dh), synth.to_f64(one[3])) <= 4e-3 and _rel(synth.to_f64(dw), synth.to_f64(one[4])) <= 4e-3


@pytest.mark.parametrize("w", [
    LceWorkload("pairs_rank_1_without_rows", 640, 520, 20008),   # the last tile of 256 rows has 128, the last of V and D 8 columns
    LceWorkload("pairs_rank_1_with_four_rows", 900, 384, 9000),
    LceWorkload("pairs_whole_tiles", 1024, 512, 10240),
    LceWorkload("pairs_several_rounds", 2000, 392, 16392),
], ids=lambda w: w.name)
def test_tiles_on_pairs_of_ctas(w):
    one = _check(w)
    # a token's results do not depend on the tile it is in: the same bits from calls of 128 tokens and from chunks of 128
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(w, "cpu").items()}
    for t in (0, w.T // 256 * 128, (w.T - 1) // 128 * 128):
        s = slice(t, t + 128)
        _, nll, lse = binding.bdlm_linear_ce_fwd(g["h"][s].contiguous(), g["w"], g["labels"][s].contiguous(), g["weight"][s].contiguous())
        assert torch.equal(lse, one[2][s]) and torch.equal(nll, one[1][s])
    dh, _ = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], one[2], g["weight"], token_chunk=128)
    assert torch.equal(dh, one[3])


@pytest.mark.parametrize("w", [
    LceWorkload("copied_for_the_backward", 400, 72, 1032),
    LceWorkload("copied_for_both", 1030, 200, 1544),
    LceWorkload("copied_wide", 1100, 264, 1000),
], ids=lambda w: w.name)
def test_rows_that_are_no_whole_number_of_lines(w):
    """From a number of tokens on, W and h are copied to padded rows (D no multiple of 64): one chunk and several."""
    one = _check(w)
    several = _check(w, token_chunk=256)
    assert torch.equal(one[3], several[3])


@pytest.mark.parametrize("D", [264, 256], ids=["copied_rows", "whole_rows"])
def test_dh_of_a_token_does_not_depend_on_the_other_tokens(D):
    """The same tokens by themselves and among many: every bit of their dH (one accumulation over the vocabulary)."""
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(LceWorkload("among_others", 1531, D, 9000), "cpu").items()}
    _, _, lse = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"])
    dh, _ = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, g["weight"])
    for n in (1, 130, 700):
        few = [g[k][:n].contiguous() for k in ("h", "labels", "weight")]
        dh_n, _ = binding.bdlm_linear_ce_bwd(few[0], g["w"], few[1], lse[:n].contiguous(), few[2])
        torch.cuda.synchronize()
        assert torch.equal(dh_n, dh[:n]), n


@pytest.mark.parametrize("V,least", [(512, False), (2048, False), (16384, True), (20008, True), (20008, False)])
def test_nan_in_the_vocabulary_and_in_a_token_reaches_the_results(V, least):
    T = 140
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(LceWorkload("nan", T, 64, V), "cpu").items()}
    per, runs = (T * 4 + 255) // 256 * 256, (((V + 255) // 256) + 7) // 8
    ws = torch.empty((2 * runs + 1) * per + 256, dtype=torch.uint8, device="cuda") if least else None
    clean = [t.clone() for t in binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"], workspace=ws)]
    # a token whose hidden state is NaN: its lse and the loss, and nobody else's lse
    bad = 77
    h = g["h"].clone()
    h[bad] = float("nan")
    labels = g["labels"].clone()
    labels[bad] = 1
    loss, nll, lse = binding.bdlm_linear_ce_fwd(h, g["w"], labels, g["weight"], workspace=ws)
    assert bool(lse[bad].isnan()) and bool(nll[bad].isnan()) and bool(loss.isnan().all())
    rest = torch.arange(T, device="cuda") != bad
    assert torch.equal(lse[rest], clean[2][rest])
    # a stretch of the vocabulary as long as the longest run: every token's lse, wherever its label lies
    n = min(2048, V // 2)
    for first in (0, V // n * n // 2 // n * n, V - n):
        w = g["w"].clone()
        w[first:first + n] = float("nan")
        away = torch.full_like(labels, (first + n) % V if first + n < V else 0)
        loss, nll, lse = binding.bdlm_linear_ce_fwd(g["h"], w, away, g["weight"], workspace=ws)
        assert bool(lse.isnan().all()) and bool(nll.isnan().all()) and bool(loss.isnan().all()), first
    torch.cuda.synchronize()
    assert binding.bdlm_get_device_status() == 0


@pytest.mark.parametrize("D", [264, 256], ids=["copied_rows", "whole_rows"])
def test_lse_of_a_token_does_not_depend_on_the_other_tokens(D):
    """The same tokens by themselves and among many: every bit of their lse and nll (the vocabulary runs end at the same
    places, whatever the tiling)."""
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(LceWorkload("among_others", 1531, D, 20008), "cpu").items()}
    _, nll, lse = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"])
    for n in (1, 130, 700, 1100):
        few = [g[k][:n].contiguous() for k in ("h", "labels", "weight")]
        _, nll_n, lse_n = binding.bdlm_linear_ce_fwd(few[0], g["w"], few[1], few[2])
        torch.cuda.synchronize()
        assert torch.equal(lse_n, lse[:n]) and torch.equal(nll_n, nll[:n]), n


@pytest.mark.parametrize("least", [False, True])
def test_vocabulary_entries_of_minus_infinity_are_left_out(least):
    """Logits of -inf (h positive, rows of W -inf): whole tiles, a whole run of the smallest workspace, single entries."""
    T, D, V = 140, 64, 5000
    gen = torch.Generator().manual_seed(1)
    h = (torch.rand(T, D, generator=gen) + 0.1).to(torch.bfloat16)
    w = (torch.randn(V, D, generator=gen) * 0.3).to(torch.bfloat16)
    out = torch.zeros(V, dtype=torch.bool)
    out[0:300] = True
    out[2048:4096] = True
    out[4990:] = True
    out[700::97] = True
    w[out] = float("-inf")
    keep = torch.nonzero(~out)[:, 0]
    labels = keep[torch.randint(len(keep), (T,), generator=gen)].int()
    per, runs = (T * 4 + 255) // 256 * 256, (((V + 255) // 256) + 7) // 8
    ws = torch.empty((2 * runs + 1) * per + 256, dtype=torch.uint8, device="cuda") if least else None
    loss, nll, lse = binding.bdlm_linear_ce_fwd(h.cuda(), w.cuda(), labels.cuda(), workspace=ws)
    where = {int(v): i for i, v in enumerate(keep)}
    y = np.array([where[int(v)] for v in labels])
    ref_loss, ref_nll, ref_lse = lce.linear_ce_forward(synth.to_f64(h), synth.to_f64(w[keep]), y)
    assert np.abs(synth.to_f64(lse) - ref_lse).max() <= TOL_LSE
    assert np.abs(synth.to_f64(nll) - ref_nll).max() <= TOL_NLL
    assert abs(float(loss) - ref_loss) <= TOL_LOSS_REL * abs(ref_loss)


@pytest.mark.parametrize("w", [
    LceWorkload("dh_64_columns", 130, 200, 3000, seed=1),      # whole panels, one past the matrix; and 64-column boxes
    LceWorkload("dh_64_whole", 260, 320, 3000, seed=2),
    LceWorkload("dh_192_columns", 1531, 1544, 1032, seed=3),
], ids=lambda w: w.name)
def test_dh_tiles_narrower_than_256_columns(w):
    _check(w)


def test_the_smallest_workspaces_serve_where_memory_is_short(monkeypatch):
    """With no room for the copies of W and h a call does what it did without them: the backward to the bit."""
    w = LceWorkload("short_of_memory", 1100, 264, 3000)
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(w, "cpu").items()}
    p = binding.make_lce_params(w.T, w.D, w.V)
    sizes = [binding.bdlm_linear_ce_workspace_bytes(p, i) for i in range(4)]
    assert 0 < sizes[2] < sizes[0] and 0 < sizes[3] < sizes[1]
    loss, nll, lse = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"])
    dh, dw = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, g["weight"])
    empty, refused = torch.empty, []

    def short(*size, **kw):
        if kw.get("dtype") == torch.uint8 and size[0] in sizes[:2]:
            refused.append(size[0])
            raise torch.OutOfMemoryError("no room")
        return empty(*size, **kw)
    monkeypatch.setattr(torch, "empty", short)
    dh2, dw2 = binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], lse, g["weight"])
    loss2, nll2, lse2 = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"])
    monkeypatch.undo()
    torch.cuda.synchronize()
    assert refused == [sizes[1], sizes[0]]
    assert torch.equal(dh, dh2) and torch.equal(dw, dw2)
    assert float((lse - lse2).abs().max()) <= TOL_LSE and float((nll - nll2).abs().max()) <= TOL_NLL
