"""The backward on pairs of CTAs (large calls of head dimension 128): the fused one against the two-pass one, that one against
the oracle on sampled rows.  An odd number of key tiles, ragged lengths with rows that are not 16-byte aligned, windows, blocks of
several tiles, both mask modes, the packed form with repeated and empty prefixes, a clean run by itself, gathered K/V in chunks
of an odd number of tiles."""
import pytest
import torch

from paper_2609_19242_b200 import binding, synth
from paper_2609_19242_b200.synth import Workload

import parity_util as pu

pytestmark = pytest.mark.gpu

# Both paths round the same P and dS to bf16 before the products and the sums to bf16 after them; the fp32 sums between are
# formed in another order, which changes the last bf16 bit of a small share of the elements (2^-9 each): 1e-3 in the 2-norm.
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


@pytest.mark.parametrize("w", [
    Workload("two_pass", 1, 24, 6, 128, 6016, 32, seed=1),
    Workload("two_pass_ragged", 2, 12, 3, 128, 6040, 40, seed=2),
    Workload("two_pass_window", 1, 16, 4, 128, 12000, 96, seed=6, window=3500),
], ids=lambda w: w.name)
def test_two_pass_gradients(w):
    """The two-pass backward's dK/dV pass runs on pairs as well: the gradients of sampled rows against the oracle."""
    pu.check_sampled(w, binding.IMPL_TCGEN05, n_rows=96, single_pass=False)


@pytest.mark.parametrize("case", ["blocks", "blocks_and_clean", "clean_run", "gathered"])
def test_packed_form(case):
    L, M, H, Hkv, batch = 12160, 24, 24, 6, 1     # 95 key tiles
    gen = torch.Generator("cuda").manual_seed(7)
    mk = lambda rows, heads, s: (torch.randn(batch, rows, heads, 128, device="cuda", generator=gen) * s).bfloat16()
    nb = 0 if case == "clean_run" else 700
    pos0, Lq = {"blocks": (0, 0), "blocks_and_clean": (3001, 4000), "clean_run": (100, 12000), "gathered": (2048, 5000)}[case]
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
    if case == "gathered":
        chunk = 5 * 128
        order = torch.randperm(L // chunk, generator=torch.Generator().manual_seed(3)).tolist()
        kw["kv_chunks"] = (chunk, [c * chunk for c in order])
    out = binding.bdlm_attn_fwd_packed(qc, k, v, qn, kn, vn, M, **kw)
    run = lambda sp: binding.bdlm_attn_bwd_packed(qc, k, v, qn, kn, vn, *out, doc, don, M, single_pass=sp, **kw)
    if case == "gathered":   # neighbours in memory are far apart in position: a pair's hull holds many tiles one of them does not see
        got = again = run(True)
    else:
        got, again = _fused(lambda: run(True), pairs * H * batch)
    for i, (a, b) in enumerate(zip(got, run(False))):
        assert (a is None) == (b is None)
        if a is not None:
            _close(a, b, i)
    for i in (1, 2):
        assert torch.equal(got[i], again[i])


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
