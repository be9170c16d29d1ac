"""The forward hands its work units from CTA to CTA: grids of several times the number of SMs, with runs of units that see
no key (queries before a clean K/V shard, the diagonal-only partial), one query stream only, ragged last tiles, both ways
of pairing tiles (even and odd group sizes) and packed calls whose streams differ in length."""
import pytest
import torch

from paper_2609_19242_b200 import binding, synth
from paper_2609_19242_b200.synth import Workload

import parity_util as pu

pytestmark = pytest.mark.gpu

CASES = [
    Workload("even", 1, 16, 4, 128, 6144, 32, seed=1),
    Workload("odd_d64", 2, 6, 2, 64, 8192, 64, seed=2),
    Workload("ragged", 3, 8, 4, 128, 5000, 40, seed=3),
    Workload("two_waves", 1, 8, 1, 128, 4096, 32, seed=5),
]


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_shards_with_unseen_tiles_merge_to_the_whole(w):
    g = synth.make_inputs(w, "cuda", with_grad=False)
    args, L, M = [g[n] for n in pu.NAMES6], w.L, w.block_size
    whole = binding.bdlm_attn_fwd(*args, M)
    cuts = [0, L // 8, L // 2, L - 64, L]
    parts = [binding.bdlm_attn_fwd(*args, M, kv_range=(a, b), include_noisy_diag=False) for a, b in zip(cuts, cuts[1:])]
    diag = binding.bdlm_attn_fwd(None, *args[1:], M, kv_range=(0, 0))
    torch.cuda.synchronize()
    assert binding.bdlm_get_device_status() == 0
    for (a, _), p in zip(zip(cuts, cuts[1:]), parts):   # rows before the shard see nothing of it
        assert float(p[0][:, :a].abs().max() if a else 0) == 0.0 and bool(torch.isneginf(p[1][:, :, :a]).all())
    clean = binding.bdlm_lse_merge([p[0] for p in parts], [p[1] for p in parts])
    noisy = binding.bdlm_lse_merge([p[2] for p in parts] + [diag[2]], [p[3] for p in parts] + [diag[3]])
    for got, want, tol in zip(clean + noisy, whole, (1e-2, 1e-3, 1e-2, 1e-3)):   # partials are rounded to bf16 once more
        assert float((got.float() - want.float()).abs().max()) <= tol


def test_one_stream_and_streams_of_different_lengths():
    w = Workload("x", 1, 16, 4, 128, 6144, 32, seed=4)
    g = synth.make_inputs(w, "cuda", with_grad=False)
    args, M = [g[n] for n in pu.NAMES6], w.block_size
    whole = binding.bdlm_attn_fwd(*args, M)
    clean = binding.bdlm_attn_fwd(*args[:3], None, None, None, M)
    noisy = binding.bdlm_attn_fwd(None, *args[1:], M)
    # the clean queries of the last third with the first 20 blocks
    q, n = args[0][:, 4096:].contiguous(), 20 * M
    few = [t[:, :n].contiguous() for t in args[3:]]
    packed = binding.bdlm_attn_fwd_packed(q, args[1], args[2], *few, M, clean_q_pos0=4096)
    torch.cuda.synchronize()
    assert binding.bdlm_get_device_status() == 0
    for i in (0, 1):
        assert torch.equal(clean[i], whole[i]) and torch.equal(noisy[i + 2], whole[i + 2])
    assert torch.equal(packed[0], whole[0][:, 4096:]) and torch.equal(packed[1], whole[1][:, :, 4096:])
    assert torch.equal(packed[2], whole[2][:, :n]) and torch.equal(packed[3], whole[3][:, :, :n])
