"""The entry points enqueue kernels only (no allocation, no synchronisation), so a forward + backward step
can be captured once into a CUDA graph and replayed."""
import pytest
import torch

from paper_2609_19242_b200 import binding, synth
from paper_2609_19242_b200.synth import Workload

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [False, True], ids=["two_pass", "fused"])
def test_forward_backward_replay_from_a_cuda_graph(fused):
    w = Workload("graph", 1, 4, 2, 128, 512, 32)
    g = pu.to_cuda(synth.make_inputs(w, "cpu"))
    M = w.block_size
    args = [g[n] for n in pu.NAMES6]
    # eager reference (also performs the library's one-time per-device setup outside the capture)
    ref_o = binding.bdlm_attn_fwd(*args, M)
    ref_g = binding.bdlm_attn_bwd(*args, ref_o[0], ref_o[1], ref_o[2], ref_o[3], g["do_clean"], g["do_noisy"], M,
                                  single_pass=fused)
    torch.cuda.synchronize()
    out = tuple(torch.zeros_like(t) for t in ref_o)
    grads = tuple(torch.zeros_like(t) for t in ref_g)
    p = binding.make_params(w.batch, w.L, M, w.H, w.H_kv, w.d, bwd_single_pass=fused)
    ws = torch.empty(binding.bdlm_workspace_bytes(p, binding.BDLM_WS_BWD), dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        binding.bdlm_attn_fwd(*args, M, out=out)
        binding.bdlm_attn_bwd(*args, out[0], out[1], out[2], out[3], g["do_clean"], g["do_noisy"], M,
                              out=grads, workspace=ws, single_pass=fused)
    for t in out + grads:
        t.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert binding.bdlm_get_device_status() == 0
    for i, (a, b) in enumerate(zip(out + grads, ref_o + ref_g)):
        if fused and i in (4, 7):   # dQ of the fused backward: fp32 summation order of the key tiles' reductions
            assert pu.rel_l2(synth.to_f64(a), synth.to_f64(b)) <= 1e-3
        else:
            assert torch.equal(a, b)
    # new inputs in the same buffers, same graph
    g["q_clean"].copy_(g["q_clean"].flip(1))
    ref_o2 = binding.bdlm_attn_fwd(*args, M)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out[0], ref_o2[0]) and torch.equal(out[1], ref_o2[1])


@pytest.mark.parametrize("T,D", [(300, 256), (1100, 264)], ids=["plain", "copied_rows"])
def test_loss_head_replays_from_a_cuda_graph_and_runs_on_any_stream(T, D):
    w = synth.LceWorkload("graph", T, D, 3000)
    g = {k: v.cuda() for k, v in synth.make_lce_inputs(w, "cpu").items()}

    def step(out=None, grads=None, ws=(None, None)):
        out = binding.bdlm_linear_ce_fwd(g["h"], g["w"], g["labels"], g["weight"], out=out, workspace=ws[0])
        return out, binding.bdlm_linear_ce_bwd(g["h"], g["w"], g["labels"], out[2], g["weight"], token_chunk=256, out=grads, workspace=ws[1])

    def same(a, b):
        return all(torch.equal(x, y) for x, y in zip(a[0] + a[1], b[0] + b[1]))
    ref = step()
    torch.cuda.synchronize()
    # several streams at once, each with its own buffers
    streams = [torch.cuda.Stream() for _ in range(3)]
    got = []
    for _ in range(3):
        for s in streams:
            with torch.cuda.stream(s):
                got.append(step())
    torch.cuda.synchronize()
    assert all(same(x, ref) for x in got)
    # one graph, replayed with other contents of the same buffers
    out, grads = tuple(torch.zeros_like(t) for t in ref[0]), tuple(torch.zeros_like(t) for t in ref[1])
    p = binding.make_lce_params(T, D, w.V, token_chunk=256)
    ws = [torch.empty(binding.bdlm_linear_ce_workspace_bytes(p, i), dtype=torch.uint8, device="cuda") for i in (binding.LCE_WS_FWD, binding.LCE_WS_BWD)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(out, grads, ws)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert same((out, grads), ref)
    g["h"].copy_(g["h"].flip(0))
    g["labels"].copy_(g["labels"].flip(0))
    ref = step()
    graph.replay()
    torch.cuda.synchronize()
    assert same((out, grads), ref)
    assert binding.bdlm_get_device_status() == 0
