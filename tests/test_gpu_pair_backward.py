"""The backward on pairs of CTAs (large calls of head dimension 128).  Its dQ is compared with the two-pass backward's, whose dQ
comes from another kernel; dK and dV with the mma.sync kernels', since the two-pass backward forms its own on pairs as well, and
with the oracle's on sampled rows.  The kernel without dQ has to give the bits of the kernel with one CTA per key tile.  An odd
number of key tiles, ragged lengths with rows that are not 16-byte aligned, windows, blocks of several tiles, both mask modes, the
packed form with repeated and empty prefixes, a clean run by itself, gathered K/V in chunks of an odd number of tiles; workspaces
full of NaN; how far a NaN among the inputs reaches; a CTA that gives up."""
import pytest
import torch

from paper_2609_19242_b200 import binding, synth
from paper_2609_19242_b200.synth import Workload

import parity_util as pu

pytestmark = pytest.mark.gpu

# Both paths round the same P and dS to bf16 before the products and the sums to bf16 after them; the fp32 sums between are
# formed in another order, which changes the last bf16 bit of a small share of the elements (2^-9 each): 1e-3 in the 2-norm.
# The mma.sync kernels round alike but scale and exponentiate in another order, which turns the last bit of a share of P and dS
# too: 2^-9 of the elements that turn, 4e-4 measured in the 2-norm of dK and dV.
TOL = 1e-3


def _close(a, b, i):
    a, b = a.double(), b.double()
    assert bool(torch.isfinite(a).all()), i
    assert float((a - b).norm()) <= TOL * float(b.norm()), i


def _fused(call, pairs):
    """The fused call's results and, from a second one with the kernels' step counter on, that pairs of CTAs ran it: they count
    a step per 256 keys x 128 queries, the other kernel one per 128 x 64."""
    out = call()
    tr = torch.zeros(binding.TRACE_SLOTS, dtype=torch.int64, device="cuda")
    binding.bdlm_set_trace_buffer(tr)
    try:
        again = call()
        torch.cuda.synchronize()
    finally:
        binding.bdlm_set_trace_buffer(None)
    assert binding.bdlm_get_device_status() == 0
    assert pairs / (256 * 128) <= int(tr[16]) <= 0.5 * pairs / (128 * 64)
    return out, again


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("w", [
    Workload("odd_tiles", 1, 24, 6, 128, 6016, 32, seed=1),
    Workload("ragged", 2, 12, 3, 128, 6040, 40, seed=2),
    Workload("unaligned_rows", 1, 24, 6, 128, 6005, 5, seed=3),
    Workload("three_heads", 2, 15, 5, 128, 8192, 128, seed=4),
    Workload("blocks_of_four_tiles", 1, 24, 6, 128, 6144, 512, seed=5),
    Workload("window", 2, 16, 4, 128, 12000, 96, seed=6, window=3500),
], ids=lambda w: w.name)
def test_plain_layer(w, mode):
    g = synth.make_inputs(w, "cuda")
    kw = dict(window=w.window, clean_mask_mode=mode)
    out = pu.gpu_fwd(g, w.block_size, **kw)
    pairs = sum(w.pairs_per_head()) * w.batch * w.H
    got, again = _fused(lambda: pu.gpu_bwd(g, out, w.block_size, single_pass=True, **kw), pairs)
    want = pu.gpu_bwd(g, out, w.block_size, single_pass=False, **kw)
    for i in range(6):
        _close(got[i], want[i], i)
    for i in (1, 2, 4, 5):   # dK, dV: a fixed order of summation
        assert torch.equal(got[i], again[i]), i
    want = pu.gpu_bwd(g, out, w.block_size, impl=binding.IMPL_PORTABLE, **kw)
    for i in range(6):
        _close(got[i], want[i], i)


@pytest.mark.parametrize("w", [
    Workload("two_pass", 1, 24, 6, 128, 6016, 32, seed=1),
    Workload("two_pass_ragged", 2, 12, 3, 128, 6040, 40, seed=2),
    Workload("two_pass_window", 1, 16, 4, 128, 12000, 96, seed=6, window=3500),
], ids=lambda w: w.name)
def test_two_pass_gradients(w):
    """The two-pass backward's dK/dV pass runs on pairs as well: the gradients of sampled rows against the oracle."""
    pu.check_sampled(w, binding.IMPL_TCGEN05, n_rows=96, single_pass=False)


@pytest.mark.parametrize("case", ["blocks", "blocks_and_clean", "clean_run", "gathered", "gathered_on_pairs"])
def test_packed_form(case):
    L, M, H, Hkv, batch = 12160, 24, 24, 6, 1     # 95 key tiles
    gen = torch.Generator("cuda").manual_seed(7)
    mk = lambda rows, heads, s: (torch.randn(batch, rows, heads, 128, device="cuda", generator=gen) * s).bfloat16()
    nb = 0 if case == "clean_run" else 700
    pos0, Lq = {"blocks": (0, 0), "blocks_and_clean": (3001, 4000), "clean_run": (100, 12000), "gathered": (2048, 5000),
                "gathered_on_pairs": (2048, 5000)}[case]
    k, v = mk(L, Hkv, 0.5), mk(L, Hkv, 0.5)
    qc, doc = (mk(Lq, H, 0.5), mk(Lq, H, 1.0)) if Lq else (None, None)
    qn, kn, vn, don = (mk(nb * M, H, 0.5), mk(nb * M, Hkv, 0.5), mk(nb * M, Hkv, 0.5), mk(nb * M, H, 1.0)) if nb else (None,) * 4
    kw = dict(clean_q_pos0=pos0)
    pairs = Lq * pos0 + Lq * (Lq + 1) // 2
    if nb:
        prefix = torch.sort(torch.randint(0, L + 1, (nb,), device="cuda", generator=gen, dtype=torch.int32)).values
        prefix[:3], prefix[10:14], prefix[-2:] = 0, prefix[10].item(), L
        kw["block_prefix"] = prefix
        pairs += int((M * (M + prefix.long())).sum())
    if "gathered" in case:
        chunk = (5 if case == "gathered" else 19) * 128
        order = torch.randperm(L // chunk, generator=torch.Generator().manual_seed(3)).tolist()
        kw["kv_chunks"] = (chunk, [c * chunk for c in order])
    out = binding.bdlm_attn_fwd_packed(qc, k, v, qn, kn, vn, M, **kw)
    run = lambda sp, **more: binding.bdlm_attn_bwd_packed(qc, k, v, qn, kn, vn, *out, doc, don, M, single_pass=sp, **kw, **more)
    if case == "gathered":   # chunks of five tiles: too many pairs would join two of them, one CTA takes each tile
        got, again = run(True), run(True)
    else:
        got, again = _fused(lambda: run(True), pairs * H * batch)
    for i, (a, b) in enumerate(zip(got, run(False))):
        assert (a is None) == (b is None)
        if a is not None:
            _close(a, b, i)
    want = run(False, impl=binding.IMPL_PORTABLE)
    for i in (1, 2, 4, 5):
        if got[i] is not None:
            assert torch.equal(got[i], again[i])
            _close(got[i], want[i], i)
    if case == "gathered_on_pairs":   # the steps that a pair takes for one of its tiles alone add nothing to the other's sums
        by_position = torch.cat([torch.arange(p, p + chunk) for p in kw["kv_chunks"][1]]).cuda()
        at = torch.empty_like(by_position)
        at[by_position] = torch.arange(L, device="cuda")
        del kw["kv_chunks"]
        k, v = k[:, at].contiguous(), v[:, at].contiguous()
        out = binding.bdlm_attn_fwd_packed(qc, k, v, qn, kn, vn, M, **kw)
        straight = run(True)
        for i in (1, 2):
            assert torch.equal(got[i][:, at], straight[i])
        for i in (4, 5):
            assert torch.equal(got[i], straight[i])


def _steps(call):
    """The call's results and the steps its kernels took, from a second call: 256 keys x 128 queries where pairs of CTAs run the
    two-pass backward's dK/dV pass, otherwise 128 x 128."""
    out = call()
    tr = torch.zeros(binding.TRACE_SLOTS, dtype=torch.int64, device="cuda")
    binding.bdlm_set_trace_buffer(tr)
    try:
        call()
        torch.cuda.synchronize()
    finally:
        binding.bdlm_set_trace_buffer(None)
    assert binding.bdlm_get_device_status() == 0
    return out, int(tr[16])


@pytest.mark.parametrize("w,mode", [
    (Workload("odd_tiles", 1, 24, 6, 128, 6016, 32, seed=1), 0),
    (Workload("odd_tiles", 1, 24, 6, 128, 6016, 32, seed=1), 1),
    (Workload("three_heads", 2, 15, 5, 128, 8192, 128, seed=4), 0),
    (Workload("blocks_of_four_tiles", 1, 24, 6, 128, 6144, 512, seed=5), 1),
], ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_two_pass_gradients_are_the_same_bits_on_pairs_and_with_one_cta_per_tile(w, mode):
    """Keys stored by position go to pairs; the same keys in chunks of one tile, in reverse, do not."""
    g = synth.make_inputs(w, "cuda")
    q, k, v, qn, kn, vn = (g[n] for n in pu.NAMES6)
    M, n = w.block_size, w.L // 128
    back = torch.cat([torch.arange(128 * c, 128 * c + 128) for c in reversed(range(n))]).cuda()
    out = binding.bdlm_attn_fwd_packed(q, k, v, qn, kn, vn, M, clean_mask_mode=mode)

    def run(k, v, **kw):
        return _steps(lambda: binding.bdlm_attn_bwd_packed(q, k, v, qn, kn, vn, *out, g["do_clean"], g["do_noisy"], M, single_pass=False,
                                                           clean_mask_mode=mode, **kw))
    on_pairs, s_pairs = run(k, v)
    alone, s_alone = run(k[:, back].contiguous(), v[:, back].contiguous(), kv_chunks=(128, [128 * c for c in reversed(range(n))]))
    assert s_pairs < 0.62 * s_alone   # (half, and the hulls)
    for i, (a, b) in enumerate(zip(on_pairs, alone)):
        assert torch.equal(a[:, back] if i in (1, 2) else a, b), i


def test_two_pass_gradients_on_pairs_do_not_depend_on_the_batch():
    w = Workload("batch", 2, 12, 3, 128, 6040, 40, seed=2)
    g = synth.make_inputs(w, "cuda")
    out = pu.gpu_fwd(g, w.block_size)
    whole = pu.gpu_bwd(g, out, w.block_size, single_pass=False)
    for b in range(w.batch):
        gb = {n: t[b:b + 1].contiguous() for n, t in g.items()}
        ob = tuple(t[b:b + 1].contiguous() for t in out)
        for x, y in zip(pu.gpu_bwd(gb, ob, w.block_size, single_pass=False), whole):
            assert torch.equal(x[0], y[b])


@pytest.mark.parametrize("w", [
    Workload("ragged", 2, 12, 3, 128, 6040, 40, seed=2),           # 24 rows in the accumulators' last block of 64
    Workload("unaligned_rows", 1, 24, 6, 128, 6005, 5, seed=3),
], ids=lambda w: w.name)
def test_nothing_in_the_workspace_matters(w):
    """The accumulators lie in halves of 64-row blocks, so that the last rows share a block with padding: a whole call and passes
    called one by one, which clear them in different launches."""
    g = synth.make_inputs(w, "cuda")
    out = pu.gpu_fwd(g, w.block_size)
    want = pu.gpu_bwd(g, out, w.block_size, single_pass=False)
    p = binding.make_params(w.batch, w.L, w.block_size, w.H, w.H_kv, w.d, bwd_single_pass=True)
    ws = torch.empty(binding.bdlm_workspace_bytes(p, binding.BDLM_WS_BWD) // 4, dtype=torch.float32, device="cuda")
    first = None
    for order in ((0,), (binding.PASS_DSUM, binding.PASS_DKDV, binding.PASS_DQ), (binding.PASS_DSUM | binding.PASS_DKDV,)):
        ws.fill_(float("nan"))
        grads = tuple(torch.full_like(t, float("nan")) for t in want)
        for bits in order:
            pu.gpu_bwd(g, out, w.block_size, single_pass=True, passes=bits, workspace=ws.view(torch.uint8), out=grads)
        first = grads if first is None else first
        for i, (a, b) in enumerate(zip(grads, want)):
            _close(a, b, i)
            assert i in (0, 3) or torch.equal(a, first[i]), (order, i)


@pytest.mark.parametrize("single_pass", [True, False], ids=["fused", "two_pass"])
def test_how_far_a_nan_among_the_inputs_reaches(single_pass):
    """A product with a NaN is NaN for whatever it meets, hidden elements included, so it reaches the rest of its tile: on pairs of
    CTAs up to 256 positions.  Beyond that every gradient is what it is without the NaN."""
    w = Workload("nan", 1, 24, 6, 128, 6016, 32, seed=1)
    M, at = w.block_size, 3005
    g = synth.make_inputs(w, "cuda")
    out = pu.gpu_fwd(g, M)
    clean = pu.gpu_bwd(g, out, M, single_pass=single_pass)
    same = (lambda a, b, i: _close(a, b, i)) if single_pass else (lambda a, b, i: torch.equal(a, b) or pytest.fail(str(i)))

    # a clean query's dO: its own dQ and the keys it sees; later keys and every other query's dQ are untouched
    bad = dict(g, do_clean=g["do_clean"].clone())
    bad["do_clean"][:, at] = float("nan")
    got = pu.gpu_bwd(bad, out, M, single_pass=single_pass)
    assert bool(torch.isnan(got[0][:, at]).all()) and bool(torch.isnan(got[1][:, :at + 1]).any(dim=-1).all())
    for i in (1, 2):
        assert torch.equal(got[i][:, at + 256:], clean[i][:, at + 256:])
    for i in (4, 5):
        assert torch.equal(got[i], clean[i])
    same(got[0][:, :at], clean[0][:, :at], 0)
    same(got[0][:, at + 1:], clean[0][:, at + 1:], 0)
    same(got[3], clean[3], 3)

    # a clean key: every query that sees it; earlier ones keep their outputs and their dQ
    bad = dict(g, k_clean=g["k_clean"].clone())
    bad["k_clean"][:, at] = float("nan")
    o = pu.gpu_fwd(bad, M)
    got = pu.gpu_bwd(bad, o, M, single_pass=single_pass)
    for i in (0, 2):
        assert torch.equal(o[i][:, :at - 255], out[i][:, :at - 255]) and bool(torch.isnan(o[i][:, at + M:]).all())
    for i in (0, 3):
        same(got[i][:, :at - 255], clean[i][:, :at - 255], i)
    assert binding.bdlm_get_device_status() == 0


def test_a_cta_that_gives_up_makes_the_other_one_of_its_pair_give_up():
    """The self-test kernel is a pair of CTAs: one wait of the first runs out after about a millisecond of clock ticks, the other
    CTA's waits have a limit of a second or more and nothing that would complete them.  They have to end because of the flag the
    first CTA raises in the other one's shared memory."""
    binding.bdlm_selftest_wait_timeout(1_000)   # (loads the kernel)
    assert binding.bdlm_get_device_status() == -5
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    begin.record()
    binding.bdlm_selftest_wait_timeout(2_000_000)
    end.record()
    assert binding.bdlm_get_device_status() == -5
    assert binding.bdlm_get_device_status() == 0
    assert 0.5 < begin.elapsed_time(end) < 200.0   # ms; 2e6 + 2^18 ticks (twice) at 1 to 2 GHz, the other CTA's own limit is 2^31
