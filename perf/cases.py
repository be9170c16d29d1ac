"""What a user of this library has it do, as measurable cases.

Four kinds of call sequences, all through the public binding, with the outputs and the workspace allocated by the
binding as it does by default:

  layer   one training step of the attention layer: forward, then backward (`bdlm_attn_fwd`, `bdlm_attn_bwd`)
  packed  the same for sampled blocks over a clean sequence, without clean queries (`bdlm_attn_*_packed`)
  rank    the launches of one rank of the context-sharded schedule: its corrupted blocks and its two runs of clean
          queries against the gathered clean K/V, forward and backward
  shards  the forward as one partial per shard of the clean K/V plus the noisy-diagonal partial, merged by LSE
  lce     the loss head: linear cross-entropy forward and backward

Sizes are those of the repository's own workloads (synth.WORKLOADS, synth.LCE_WORKLOADS) and of its tests, with
generic ones between them.
"""
import math

import torch

from paper_2609_19242_b200 import binding, schedule, synth

NAMES6 = ("q_clean", "k_clean", "v_clean", "q_noisy", "k_noisy", "v_noisy")


def _layer(name, batch, H, H_kv, d, L, M, window=0, rope=0.0, two_pass=False):
    return {"name": name, "kind": "layer", "batch": batch, "H": H, "H_kv": H_kv, "d": d, "L": L, "M": M,
            "window": window, "rope": rope, "two_pass": two_pass}


def listed():
    return [
        # the smallest call anyone makes: a unit-test sized layer, where launches and host time are everything
        _layer("layer_tiny", 1, 2, 2, 64, 256, 16),
        # a small model on short sequences with nothing aligned: odd group size, head dimension 64, a ragged length
        _layer("layer_ragged", 3, 12, 4, 64, 1000, 40),
        # a fine-tuning step at a short context: few tiles per head, so the chip is hard to fill
        _layer("layer_2k", 1, 32, 8, 128, 2048, 32),
        # a medium context with a batch of two
        _layer("layer_8k", 2, 16, 4, 128, 8192, 32),
        # the layer the library is benchmarked on
        _layer("layer_32k", 1, 32, 8, 128, 32768, 64, rope=5e5),
        # a sliding-window layer of a hybrid model
        _layer("layer_32k_window", 1, 32, 8, 128, 32768, 64, window=1024, rope=5e5),
        # attention without KV sharing, and the bitwise reproducible backward a debugging run asks for
        _layer("layer_mha_reproducible", 1, 8, 8, 128, 16384, 32, two_pass=True),
        # a drafter's layer: 2048 sampled blocks of 16 tokens over 32K clean keys
        {"name": "packed_32k", "kind": "packed", "batch": 1, "H": 32, "H_kv": 8, "d": 128, "L": 32768, "M": 16, "n_blocks": 2048},
        # one of eight ranks of a 64K sequence: gathered clean K/V, two runs of clean queries, its share of the blocks
        {"name": "rank_64k_of_8", "kind": "rank", "batch": 1, "H": 32, "H_kv": 8, "d": 128, "L": 65536, "M": 32, "P": 8, "rank": 3},
        # a 128K forward with the clean K/V in eight context shards; the largest
        {"name": "shards_128k", "kind": "shards", "batch": 1, "H": 32, "H_kv": 8, "d": 128, "L": 131072, "M": 32, "shards": 8},
        # the loss head of a small model on a micro-batch with ragged sizes
        {"name": "lce_ragged", "kind": "lce", "T": 1531, "D": 1544, "V": 32008},
        # the loss head the library is benchmarked on
        {"name": "lce_8k", "kind": "lce", "T": 8192, "D": 4096, "V": 128256},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    while True:
        kind = rng.choice(["layer", "layer", "layer", "layer", "packed", "rank", "shards", "lce", "lce"])
        if kind == "lce":
            D = 8 * _log_uniform(rng, 8, 512)
            case = {"kind": "lce", "T": _log_uniform(rng, 100, 8192), "D": D, "V": 8 * _log_uniform(rng, 125, 16032)}
        else:
            M = rng.choice([4, 16, 16, 24, 32, 32, 40, 64, 64, 128, 256, 512])
            H_kv = rng.choice([1, 2, 4, 8])
            H = H_kv * rng.choice([1, 2, 3, 4, 4, 5, 8])
            case = {"kind": kind, "batch": rng.choice([1, 1, 1, 2, 3]), "H": H, "H_kv": H_kv, "d": rng.choice([64, 128, 128]),
                    "M": M, "L": M * max(2, _log_uniform(rng, 256, 65536) // M)}
            if kind == "layer":
                case.update(window=rng.choice([0, 0, 0, _log_uniform(rng, 64, 4096)]), rope=rng.choice([0.0, 5e5]),
                            two_pass=rng.random() < 0.2)
            elif kind == "packed":
                case["n_blocks"] = _log_uniform(rng, 4, 4096)
            elif kind == "rank":
                P = rng.choice([2, 4, 8])
                unit = math.lcm(2 * P * 128, 2 * P * M)   # whole 128-row tiles per chunk, two blocks at least per rank
                case.update(L=unit * max(1, case["L"] // unit), P=P, rank=rng.randrange(P))
            else:
                case["shards"] = rng.choice([2, 3, 4, 8])
        w = work(case)
        # no larger than the largest listed case, in operations or in what has to lie in memory
        if w["flops"] <= 1.0e14 and w["bytes"] <= 8.0e9:
            return case


def _workload(case, seed):
    # the shard and rank kinds start from the plain layer's tensors
    return synth.Workload("case", case["batch"], case["H"], case["H_kv"], case["d"], case["L"], case["M"],
                          rope_theta=case.get("rope", 0.0), window=case.get("window", 0), n_blocks=case.get("n_blocks", 0),
                          seed=seed)


def prepare(case, seed):
    if case["kind"] == "lce":
        g = synth.make_lce_inputs(synth.LceWorkload("case", case["T"], case["D"], case["V"], seed=seed), "cuda")
        return {"case": case, **g}
    w = _workload(case, seed)
    g = synth.make_inputs(w, "cuda", with_grad=case["kind"] != "shards")
    state = {"case": case}
    if case["kind"] != "rank":
        state.update(g)
        return state
    # what a rank holds: the clean K/V as the all-gather left them (rank by rank, each rank's two zigzag chunks), its
    # own two runs of clean queries and its packed corrupted blocks with their prefix table
    P, M, L = case["P"], case["M"], case["L"]
    plan = schedule.csbp_plan(L, M, P)[case["rank"]]
    chunk = L // (2 * P)
    order = [c for r in range(P) for c in (r, 2 * P - 1 - r)]
    by_chunk = lambda t: torch.cat([t[:, c * chunk:(c + 1) * chunk] for c in order], dim=1).contiguous()
    state["k_clean"], state["v_clean"] = by_chunk(g["k_clean"]), by_chunk(g["v_clean"])
    state["kv_chunks"] = (chunk, [c * chunk for c in order])
    blocks = torch.tensor(plan.blocks, device="cuda")
    for n in ("q_noisy", "k_noisy", "v_noisy", "do_noisy"):
        t = g[n]
        state[n] = t.view(t.shape[0], L // M, M, *t.shape[2:])[:, blocks].flatten(1, 2).contiguous()
    state["block_prefix"] = torch.tensor(plan.block_prefix, dtype=torch.int32, device="cuda")
    state["runs"] = [(p0, g["q_clean"][:, p0:p1].contiguous(), g["do_clean"][:, p0:p1].contiguous())
                     for p0, p1 in plan.clean_ranges]
    return state


def _run_layer(s):
    c = s["case"]
    args, M = [s[n] for n in NAMES6], c["M"]
    out = binding.bdlm_attn_fwd(*args, M, window=c["window"])
    grads = binding.bdlm_attn_bwd(*args, *out, s["do_clean"], s["do_noisy"], M, window=c["window"],
                                  single_pass=False if c["two_pass"] else None)
    return out, grads


def _run_packed(s):
    args, M, pfx = [s[n] for n in NAMES6], s["case"]["M"], s["block_prefix"]
    out = binding.bdlm_attn_fwd_packed(*args, M, block_prefix=pfx)
    grads = binding.bdlm_attn_bwd_packed(*args, *out, None, s["do_noisy"], M, block_prefix=pfx)
    return out, grads


def _run_rank(s):
    M, kv = s["case"]["M"], (s["k_clean"], s["v_clean"])
    noisy = (s["q_noisy"], s["k_noisy"], s["v_noisy"])
    (p0, q0, do0), (p1, q1, do1) = s["runs"]
    first = dict(block_prefix=s["block_prefix"], clean_q_pos0=p0, kv_chunks=s["kv_chunks"])
    second = dict(clean_q_pos0=p1, kv_chunks=s["kv_chunks"])
    # the first run of clean queries goes with the corrupted blocks, the second one by itself
    out0 = binding.bdlm_attn_fwd_packed(q0, *kv, *noisy, M, **first)
    out1 = binding.bdlm_attn_fwd_packed(q1, *kv, None, None, None, M, **second)
    g0 = binding.bdlm_attn_bwd_packed(q0, *kv, *noisy, *out0, do0, s["do_noisy"], M, **first)
    g1 = binding.bdlm_attn_bwd_packed(q1, *kv, None, None, None, *out1, do1, None, M, **second)
    return out0, out1, g0, g1


def _run_shards(s):
    c = s["case"]
    args, M, L, n = [s[n] for n in NAMES6], c["M"], c["L"], c["shards"]
    cuts = [L * i // n for i in range(n + 1)]
    parts = [binding.bdlm_attn_fwd(*args, M, kv_range=(a, b), include_noisy_diag=False) for a, b in zip(cuts, cuts[1:])]
    diag = binding.bdlm_attn_fwd(None, *args[1:], M, kv_range=(0, 0))
    clean = binding.bdlm_lse_merge([p[0] for p in parts], [p[1] for p in parts])
    noisy = binding.bdlm_lse_merge([p[2] for p in parts] + [diag[2]], [p[3] for p in parts] + [diag[3]])
    return clean, noisy


def _run_lce(s):
    loss, nll, lse = binding.bdlm_linear_ce_fwd(s["h"], s["w"], s["labels"], s["weight"])
    dh, dw = binding.bdlm_linear_ce_bwd(s["h"], s["w"], s["labels"], lse, s["weight"])
    return loss, nll, lse, dh, dw


_RUN = {"layer": _run_layer, "packed": _run_packed, "rank": _run_rank, "shards": _run_shards, "lce": _run_lce}


def run(state):
    return _RUN[state["case"]["kind"]](state)


def _rank_pairs(case):
    """Visible (query, key) pairs per query head of one rank's launches."""
    plan = schedule.csbp_plan(case["L"], case["M"], case["P"])[case["rank"]]
    noisy = sum(case["M"] * (case["M"] + p) for p in plan.block_prefix)
    clean = sum(p1 * (p1 + 1) // 2 - p0 * (p0 + 1) // 2 for p0, p1 in plan.clean_ranges)
    rows_noisy = case["M"] * len(plan.blocks)
    rows_clean = sum(p1 - p0 for p0, p1 in plan.clean_ranges)
    return clean + noisy, rows_clean, rows_noisy


def work(case):
    if case["kind"] == "lce":
        T, D, V = case["T"], case["D"], case["V"]
        # the projection, and the two gradient products; h and W in, dH and dW out, per token a label, a weight, nll, lse
        return {"bytes": 2 * (2 * T * D + 2 * V * D) + 16 * T, "flops": 6 * T * D * V}
    b, H, H_kv, d = case["batch"], case["H"], case["H_kv"], case["d"]
    if case["kind"] == "rank":
        pairs, rows_c, rows_n = _rank_pairs(case)
    else:
        pairs = sum(_workload(case, 0).pairs_per_head())
        rows_n = case["n_blocks"] * case["M"] if case["kind"] == "packed" else case["L"]
        rows_c = 0 if case["kind"] == "packed" else case["L"]
    q = b * H * (rows_c + rows_n) * d * 2               # one bf16 query-side tensor
    kv = 2 * b * H_kv * (case["L"] + rows_n) * d * 2    # K and V of both streams
    lse = b * H * (rows_c + rows_n) * 4
    if case["kind"] == "shards":
        return {"bytes": 2 * q + kv + lse, "flops": 4 * d * pairs * b * H}
    # q, dO in, O and dQ out; K, V in and dK, dV out; LSE out (4 and 10 d operations per pair, forward and backward)
    return {"bytes": 4 * q + 2 * kv + lse, "flops": 14 * d * pairs * b * H}


def tolerance(case):
    # bf16 tensors throughout: outputs and gradients carry the roundings of O, P, dS and dz (2^-9 each).  Measured:
    # against an explicit-mask evaluation in 64 bits O 2.3e-3, gradients 2.5e-3, the loss head's gradients 2.3e-3;
    # between the tensor-core kernels and the mma.sync ones (64-key tiles, another order) up to 3.1e-3.  The largest
    # single difference is a dQ element of the first rows, where dP - D cancels: 0.098 of the tensor's root mean square
    # (0.06 for an element of the loss head's dW).
    return {"rel": 1e-2, "max": 0.25 if case["kind"] == "lce" else 0.4}


# ---- the same outputs from the definitions, in 64 bits ----

def _attend64(q, pos, k, v, window, own=None, do=None):
    """Rows q [R, G, d] at positions `pos` [R] over the visible keys of one KV head: clean keys k, v [n, d] with
    j < lim[r] and pos[r] - j < window, and the rows' own blocks.  `own` = (lim [R], k [R, d], v [R, d], block of each
    row [R]) for corrupted rows; clean rows see the keys up to their own position.  Returns o, lse and, with `do`, dq,
    (dk, dv) of the clean keys and (dk, dv) of the own keys."""
    d = q.shape[-1]
    j = torch.arange(k.shape[0], device=q.device)
    lim = pos + 1 if own is None else own[0]
    seen = j[None, :] < lim[:, None]
    if window > 0:
        seen &= pos[:, None] - j[None, :] < window
    keys, vals = k, v
    if own is not None:
        keys, vals = torch.cat([k, own[1]]), torch.cat([v, own[2]])
        seen = torch.cat([seen, own[3][:, None] == own[3][None, :]], dim=1)
    s = torch.einsum("rgd,nd->grn", q, keys) / math.sqrt(d)
    s.masked_fill_(~seen, -math.inf)
    lse = torch.logsumexp(s, dim=-1)                       # [G, R]
    p = s.sub_(lse[..., None]).exp_()
    o = torch.einsum("grn,nd->rgd", p, vals)
    if do is None:
        return o, lse, None, None, None
    dv = torch.einsum("grn,rgd->nd", p, do)
    ds = torch.einsum("rgd,nd->grn", do, vals).sub_((do * o).sum(-1).T[..., None]).mul_(p).div_(math.sqrt(d))
    dq = torch.einsum("grn,nd->rgd", ds, keys)
    dk = torch.einsum("grn,rgd->nd", ds, q)
    n = k.shape[0]
    return o, lse, dq, (dk[:n], dv[:n]), (dk[n:], dv[n:])


def _stream64(q, k, v, do, pos, window, lim=None, M=1, kn=None, vn=None):
    """One query stream over the clean keys in position order (and its own blocks, with `lim`): o, lse, dq, dk and dv of
    the clean keys, dk and dv of the own keys."""
    batch, rows, H, d = q.shape
    H_kv, G = k.shape[2], H // k.shape[2]
    f = lambda *s: torch.zeros(*s, dtype=torch.float64, device=q.device)
    o, lse, dq = f(*q.shape), f(batch, H, rows), f(*q.shape)
    dk, dv = f(*k.shape), f(*k.shape)
    dkn, dvn = (f(*kn.shape), f(*kn.shape)) if lim is not None else (None, None)
    step = M * max(1, 1024 // M)
    for b in range(batch):
        for hk in range(H_kv):
            h = slice(hk * G, hk * G + G)
            kd, vd = k[b, :, hk].double(), v[b, :, hk].double()
            for r0 in range(0, rows, step):
                r = slice(r0, min(rows, r0 + step))
                n = int(lim[r].max()) if lim is not None else int(pos[r].max()) + 1
                own = None
                if lim is not None:
                    own = (lim[r], kn[b, r, hk].double(), vn[b, r, hk].double(), torch.arange(r.start, r.stop, device=q.device) // M)
                got = _attend64(q[b, r, h].double(), pos[r], kd[:n], vd[:n], window, own, None if do is None else do[b, r, h].double())
                o[b, r, h], lse[b, h, r] = got[0], got[1]
                if do is not None:
                    dq[b, r, h] = got[2]
                    dk[b, :n, hk] += got[3][0]
                    dv[b, :n, hk] += got[3][1]
                    if lim is not None:
                        dkn[b, r, hk], dvn[b, r, hk] = got[4]
    return o, lse, dq, dk, dv, dkn, dvn


def _exact_lce(s):
    h, w, y, wt = s["h"].double(), s["w"].double(), s["labels"].long(), s["weight"].double()
    nll, lse = torch.zeros_like(wt), torch.zeros_like(wt)
    dh, dw = torch.zeros_like(h), torch.zeros_like(w)
    for t0 in range(0, h.shape[0], 2048):
        t = slice(t0, t0 + 2048)
        z = h[t] @ w.T
        lse[t] = torch.logsumexp(z, dim=-1)
        at, on = y[t].clamp(min=0)[:, None], y[t] >= 0
        nll[t] = torch.where(on, lse[t] - z.gather(1, at)[:, 0], 0.0)
        z = z.sub_(lse[t][:, None]).exp_()
        z.scatter_add_(1, at, torch.full_like(at, -1, dtype=torch.float64))
        z.mul_((wt[t] * on)[:, None])
        dh[t] = z @ w
        dw += z.T @ h[t]
    return (wt * nll).sum().reshape(1), nll, lse, dh, dw


def exact(case, seed):
    if work(case)["flops"] > 8.0e13:   # over about 20 seconds
        return None
    s = prepare(case, seed)
    if case["kind"] == "lce":
        return _exact_lce(s)
    M, L, window, dev = case["M"], case["L"], case.get("window", 0), s["k_clean"].device
    k, v = s["k_clean"], s["v_clean"]
    at = lambda p0, p1: torch.arange(p0, p1, device=dev)
    rows = s["q_noisy"].shape[1]
    block = at(0, rows) // M
    prefix = (s["block_prefix"].long() if "block_prefix" in s else at(0, L // M) * M)[block]
    noisy = lambda kc, vc: _stream64(s["q_noisy"], kc, vc, s.get("do_noisy"), prefix + at(0, rows) % M, window, prefix, M,
                                     s["k_noisy"], s["v_noisy"])
    if case["kind"] == "rank":
        chunk, positions = s["kv_chunks"]
        where = torch.cat([at(p, p + chunk) for p in positions])     # position of each stored row
        by_pos = torch.argsort(where)
        k, v = k[:, by_pos], v[:, by_pos]
        n = noisy(k, v)
        (p0, q0, do0), (p1, q1, do1) = s["runs"]
        c0, c1 = (_stream64(q, k, v, do, at(p, p + q.shape[1]), 0) for p, q, do in ((p0, q0, do0), (p1, q1, do1)))
        return ((c0[0], c0[1], n[0], n[1]), (c1[0], c1[1], None, None),
                (c0[2], (c0[3] + n[3])[:, where], (c0[4] + n[4])[:, where], n[2], n[5], n[6]),
                (c1[2], c1[3][:, where], c1[4][:, where], None, None, None))
    n = noisy(k, v)
    if case["kind"] == "packed":
        return (None, None, n[0], n[1]), (None, n[3], n[4], n[2], n[5], n[6])
    c = _stream64(s["q_clean"], k, v, s.get("do_clean"), at(0, L), window)
    if case["kind"] == "shards":
        return (c[0], c[1]), (n[0], n[1])
    return (c[0], c[1], n[0], n[1]), (c[2], c[3] + n[3], c[4] + n[4], n[2], n[5], n[6])
