"""Backward calls short enough that a cluster of CTAs shares each clean key tile: the partial dK / dV tiles are added up
through distributed shared memory (fused kernel).  Two and four CTAs per tile, step counts that the CTAs do not divide,
ragged last tiles, one head per group, key tiles only some of the CTAs have steps for (sliding window).  The two-pass kernels,
one CTA per key tile, at the same sizes: there a batch element's gradients do not depend on the batch."""
import pytest
import torch

from paper_2609_19242_b200 import binding, synth
from paper_2609_19242_b200.synth import Workload

import parity_util as pu

pytestmark = pytest.mark.gpu

CASES = [
    Workload("two", 4, 16, 8, 128, 512, 32, seed=1),               # heaviest tile 1.6 times the mean load per SM
    Workload("two_ragged_d64", 4, 24, 8, 64, 440, 40, seed=2),
    Workload("four", 1, 4, 1, 128, 640, 64, seed=3),
    Workload("four_one_head", 1, 1, 1, 128, 1000, 40, seed=4),     # the CTAs of a cluster take different query tiles
    Workload("four_three_heads_d64", 1, 3, 1, 64, 776, 8, seed=5),
    Workload("four_window", 1, 4, 1, 128, 1024, 16, window=130, seed=6),
]


@pytest.mark.parametrize("single_pass", [True, False], ids=["fused", "two_pass"])
@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_split_key_tiles_match_the_oracle_and_are_reproducible(w, single_pass):
    pu.check_full(w, binding.IMPL_TCGEN05, single_pass=single_pass)
    g = synth.make_inputs(w, "cuda")
    out = pu.gpu_fwd(g, w.block_size, window=w.window)
    a, b = (pu.gpu_bwd(g, out, w.block_size, window=w.window, single_pass=single_pass) for _ in range(2))
    for i in (1, 2, 4, 5):   # dK, dV of both streams: a fixed order of summation
        assert torch.equal(a[i], b[i])


@pytest.mark.parametrize("w", [
    Workload("ten", 10, 8, 2, 128, 512, 32, seed=7),
    Workload("odd_group_d64", 20, 3, 1, 64, 776, 8, seed=8),
    Workload("window", 24, 8, 2, 128, 512, 16, window=130, seed=9),
], ids=lambda w: w.name)
def test_two_pass_gradients_of_a_batch_element_do_not_depend_on_the_batch(w):
    g = synth.make_inputs(w, "cuda")
    out = pu.gpu_fwd(g, w.block_size, window=w.window)
    whole = pu.gpu_bwd(g, out, w.block_size, window=w.window, single_pass=False)
    for i in (0, w.batch - 1):
        gi = {k: (v[i:i + 1].contiguous() if v.dim() == 4 else v) for k, v in g.items()}
        oi = pu.gpu_fwd(gi, w.block_size, window=w.window)
        for a, b in zip(oi, out):
            assert torch.equal(a[0], b[i])
        for a, b in zip(pu.gpu_bwd(gi, oi, w.block_size, window=w.window, single_pass=False), whole):
            assert torch.equal(a[0], b[i])


@pytest.mark.parametrize("w", [
    Workload("shared_tiles", 1, 4, 1, 128, 1000, 40, seed=10),
    Workload("shared_tiles_d64", 2, 6, 2, 64, 776, 8, seed=11),
    Workload("one_cta_per_tile", 1, 2, 2, 128, 296, 8, seed=12),
    Workload("one_cta_per_tile_d64", 1, 2, 2, 64, 296, 8, seed=13),
], ids=lambda w: w.name)
def test_fused_passes_called_one_by_one_agree_with_the_whole_call(w):
    """By themselves the passes clear the fp32 dQ accumulators in another launch than the whole call does, and are not
    chained.  Nothing in the workspace may matter; lengths are no multiple of the 64-row step."""
    g = synth.make_inputs(w, "cuda")
    out = pu.gpu_fwd(g, w.block_size)
    whole = pu.gpu_bwd(g, out, w.block_size, single_pass=True)
    p = binding.make_params(w.batch, w.L, w.block_size, w.H, w.H_kv, w.d, bwd_single_pass=True)
    ws = torch.empty(binding.bdlm_workspace_bytes(p, binding.BDLM_WS_BWD) // 4, dtype=torch.float32, device="cuda")
    for order in ((binding.PASS_DSUM, binding.PASS_DKDV, binding.PASS_DQ), (binding.PASS_DSUM | binding.PASS_DKDV,),
                  (binding.PASS_DSUM, binding.PASS_DKDV | binding.PASS_DQ)):
        ws.fill_(float("nan"))
        grads = tuple(torch.full_like(t, float("nan")) for t in whole)
        for bits in order:
            pu.gpu_bwd(g, out, w.block_size, single_pass=True, passes=bits, workspace=ws.view(torch.uint8), out=grads)
        for i, (a, b) in enumerate(zip(grads, whole)):
            if i in (0, 3):   # dQ: the order in which the key tiles' sums arrive, then one bf16 rounding
                assert pu.rel_l2(synth.to_f64(a), synth.to_f64(b)) <= 1e-3
            else:
                assert torch.equal(a, b), (order, i)
