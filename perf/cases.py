"""The workloads whose speed this framework is held to, as a user's program calls them.

Three kinds, all through the public entry points of `paper_2605_18753_b200.binding`:

* ``decode``    one new token per sequence against a KV cache (contiguous or paged), `dash_attn_fwd_decode*`;
* ``prefill``   a whole prompt, `dash_attn_fwd_prefill`, or the three stages by themselves (``staged``: what a training
                program calls, because it keeps the thresholds and lists for its backward pass);
* ``backward``  the gradients of the whole layer from a given dO: `dash_attn_bwd_attend_prefill*`, then
                `dash_attn_bwd_select_prefill`, then `dash_attn_bwd_block_summaries`.

Inputs are the seeded tensors of `synth` (queries around a direction, a few chunks whose keys are shifted towards it).
"""
import math

import numpy as np
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth

# A routed chunk closer to the threshold than this is left out of the lists a backward case is given: log w has a pole
# at the threshold, and a gradient right beside it says nothing about the rest (see _routing).
MARGIN = 1e-3


def _case(kind, name=None, *, batch=1, seq=8192, h_q=32, h_kv=8, head_dim=128, block=64, alpha=1.5, gamma=1.0, sigma=10.0,
          shift=2.0, dtype="bf16", recipe="planted", local_blocks=0, **more):
    c = dict(kind=kind, batch=batch, seq=seq, h_q=h_q, h_kv=h_kv, head_dim=head_dim, block=block, alpha=alpha, gamma=gamma,
             sigma=sigma, shift=shift, dtype=dtype, recipe=recipe, local_blocks=local_blocks, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one user's chat on an 8K cache: three short kernels, where launches and latency count
        _case("decode", "decode_1x8k", seq=8192, ragged=0.97),
        # a server's full batch on long contexts: 16 caches of 131072 tokens, about 90 % of the chunks not read
        _case("decode", "decode_16x128k", batch=16, seq=131072, shift=1.42, ragged=1.0),
        # a server's paged cache: many sequences of very different lengths, the trained models' window of one chunk, and
        # the prior strength the models are deployed with
        _case("decode", "decode_paged_48x32k", batch=48, seq=32768, shift=1.6, sigma=1e8, local_blocks=1, page_size=64, ragged=0.03),
        # a short prompt of odd length
        _case("prefill", "prefill_500", seq=500),
        # the ordinary prompt
        _case("prefill", "prefill_8k", seq=8192),
        # the long prompt
        _case("prefill", "prefill_64k", seq=65536, shift=2.10),
        # coarse chunks and sparsemax routing on two prompts at once
        _case("prefill", "prefill_2x32k_b128_a2", batch=2, seq=32768, block=128, alpha=2.0),
        # the fine chunks that the chunk-size study prefers for accuracy
        _case("prefill", "prefill_8k_b16", seq=8192, block=16, shift=1.77),
        # single precision: the exact check of one head that every installation is tried with
        _case("prefill", "prefill_1k_f32", seq=1024, h_q=1, h_kv=1, head_dim=64, gamma=512.0, dtype="f32", recipe="tiny"),
        # a small multi-head model's training forward: an odd length, learned summary queries, the training
        # window, thresholds and lists kept
        _case("prefill", "train_fwd_3x1999_mha", batch=3, seq=1999, h_q=12, h_kv=12, head_dim=64, block=32, local_blocks=1, staged=True),
        # the backward of a small grouped-query model, through the entry point that takes every shape
        _case("backward", "train_bwd_2x1500_d64", batch=2, seq=1500, h_q=8, h_kv=2, head_dim=64, block=32, local_blocks=1),
        # the backward of the ordinary prompt, through the entry point for these shapes
        _case("backward", "train_bwd_8k", seq=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds, every option in the range the listed cases stand for."""
    most = work(next(c for c in listed() if c["name"] == "prefill_64k"))["flops"]
    while True:
        h_q, h_kv = rng.choice([(32, 8), (32, 8), (32, 2), (16, 2), (8, 2), (16, 8), (12, 12)])
        shape = dict(h_q=h_q, h_kv=h_kv, head_dim=rng.choice([128, 128, 64]), block=rng.choice([16, 32, 64, 64, 64, 128]),
                     alpha=rng.choice([1.25, 1.5, 1.5, 1.5, 2.0]), sigma=rng.choice([1.0, 10.0, 1e8]), local_blocks=rng.choice([0, 0, 1]),
                     shift=round(rng.uniform(1.5, 2.2), 2))
        kind = rng.choice(["decode", "decode", "prefill", "prefill", "prefill", "backward"])
        if kind == "decode":
            batch, seq = _log_int(rng, 1, 64), _log_int(rng, 1024, 131072)
            more = dict(ragged=round(rng.uniform(0.03, 1.0), 2))
            if rng.random() < 0.5:
                more["page_size"] = rng.choice([64, 128, 256]) if shape["block"] < 128 else rng.choice([128, 256])
                seq = max(1, round(seq / more["page_size"])) * more["page_size"]
            if batch * seq > 2 ** 21 or seq // shape["block"] > 8192:
                continue
            return _case(kind, batch=batch, seq=seq, **shape, **more)
        if kind == "backward":
            # α = 1.5 is what models are trained with; the tensor-core kernels' shapes go further than the others
            large = h_q > h_kv and shape["head_dim"] == 128 and shape["block"] >= 64
            shape.update(alpha=1.5)
            case = _case(kind, batch=rng.choice([1, 2]), seq=_log_int(rng, 300, 8192 if large else 1600), **shape)
            if not large and case["batch"] * case["seq"] * h_q > 2 * 1600 * 16:
                continue
            return case
        if h_q == h_kv or rng.random() < 0.15:     # multi-head or single-precision models: small ones
            shape.update(h_q=min(h_q, 12), h_kv=min(h_kv, 12))
            if shape["h_q"] % shape["h_kv"] or shape["h_q"] // shape["h_kv"] not in (1, 2, 4, 8, 16):
                continue
            dtype = "bf16" if rng.random() < 0.5 and h_q == h_kv else "f32"
            return _case(kind, batch=rng.choice([1, 2, 3]), seq=_log_int(rng, 200, 2000), dtype=dtype, **shape, staged=rng.random() < 0.5)
        case = _case(kind, batch=rng.choice([1, 1, 2, 3]), seq=_log_int(rng, 200, 65536 if shape["block"] >= 64 else 12000), **shape,
                     staged=rng.random() < 0.3)
        if work(case)["flops"] <= most:
            return case


def _workload(case, seed, batch=None, seq=None):
    return synth.Workload("case", "decode" if case["kind"] == "decode" else "prefill", batch or case["batch"], seq or case["seq"], case["h_q"],
                          case["h_kv"], case["head_dim"], case["block"], case["alpha"], case["dtype"], case["recipe"],
                          gamma=case["gamma"], sigma=case["sigma"], shift=case["shift"], seed=seed)


def _lengths(case):
    """Tokens in each sequence's cache: spread from `ragged` of the capacity to all of it (one sequence: that share)."""
    b, seq, low = case["batch"], case["seq"], case["ragged"]
    part = [0.0] if b == 1 else [(i * 7 % b) / (b - 1) if math.gcd(7, b) == 1 else i / (b - 1) for i in range(b)]
    return [max(1, min(seq, round(seq * (low + (1.0 - low) * f)))) for f in part]


def _summary_query(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000 + 500)
    return torch.randn(case["h_kv"], case["head_dim"], generator=g, device="cuda")


def _options(case):
    return dict(block=case["block"], alpha=case["alpha"], gamma=case["gamma"], sigma=case["sigma"], local_blocks=case["local_blocks"])


def _prepare_decode(case, seed):
    lens = _lengths(case)
    if not case.get("page_size"):
        s = synth.make_decode_inputs(_workload(case, seed), "cuda", kv_len=lens)
        s["O"] = torch.empty_like(s["Q"])
        s["p"] = B.params_for_decode(s["Q"], s["K"], s["V"], s["O"], **_options(case))
        s["Kbar"] = B.alloc_kbar(s["p"])
        B.dash_attn_block_summaries(s["p"], s["K"], s["Kbar"], kv_len=s["kv_len"])
    else:
        # pools filled sequence by sequence, pages handed out in a random order
        page = case["page_size"]
        per = [-(-n // page) for n in lens]
        order = torch.randperm(sum(per), generator=torch.Generator().manual_seed(seed)).tolist()
        pool = lambda: torch.empty(sum(per), page, case["h_kv"], case["head_dim"], dtype=torch.bfloat16, device="cuda")
        s = {"K": pool(), "V": pool(), "kv_len": torch.tensor(lens, dtype=torch.int32, device="cuda")}
        table = torch.zeros(case["batch"], case["seq"] // page, dtype=torch.int32)
        queries = []
        for i, n in enumerate(per):
            one = synth.make_decode_inputs(_workload(case, seed * 64 + i, batch=1, seq=n * page), "cuda")
            ids = torch.tensor([order.pop() for _ in range(n)])
            table[i, :n] = ids
            for key in ("K", "V"):
                s[key][ids.to("cuda")] = one[key].view(n, page, case["h_kv"], case["head_dim"])
            queries.append(one["Q"])
        s["Q"], s["table"] = torch.cat(queries), table.to("cuda")
        s["O"] = torch.empty_like(s["Q"])
        s["p"] = B.params_for_paged_decode(s["Q"], s["K"], s["V"], s["O"], max_pages=case["seq"] // page, **_options(case))
        s["Kbar"] = B.alloc_kbar(s["p"])
        B.dash_attn_block_summaries_paged(s["p"], s["K"], s["table"], s["Kbar"], kv_len=s["kv_len"])
    s["ws"] = B.alloc_workspace(s["p"])
    return s


def _prepare_prefill(case, seed):
    s = synth.make_prefill_inputs(_workload(case, seed), "cuda")
    s["O"] = torch.empty_like(s["Q"])
    s["p"] = B.params_for_prefill(s["Q"], s["K"], s["V"], s["O"], **_options(case))
    s["ws"] = B.alloc_workspace(s["p"])
    if case.get("staged"):
        s["qbar"], s["Kbar"] = _summary_query(case, seed), B.alloc_kbar(s["p"])
        s["routing"] = B.alloc_routing(s["p"], with_tau=True)
    return s


def _routing(case, p, Q, Kbar):
    """Routing of every row in double precision, in the layout of dash_attn_select.

    dlog w/dx grows as 1/margin towards the threshold, so that without a gap the norm of the gradient would be that of its
    one entry nearest to the threshold, which single precision does not determine."""
    n, T, L, blk = case["seq"], case["seq"] // case["block"], case["local_blocks"], case["block"]
    g, e = case["h_q"] // case["h_kv"], 1.0 / (case["alpha"] - 1.0)
    out = B.alloc_routing(p, with_tau=True)
    out["tau"].zero_(), out["blk_idx"].zero_(), out["blk_bias"].zero_()
    row = torch.arange(n, device="cuda")
    own, chunk = row // blk, torch.arange(T, device="cuda")
    cand = chunk[None] < (own[:, None] - L)
    window = (chunk[None] >= own[:, None] - L) & (chunk[None] < own[:, None])
    start = blk * own * (own - 1) // 2 + (row % blk) * own
    per_head = B.dash_attn_list_capacity(p) // (case["batch"] * case["h_kv"])
    words = out["mask"].shape[-1]
    bit = (2 ** torch.arange(32, device="cuda", dtype=torch.int64))[None, None]
    for b in range(case["batch"]):
        for r in range(case["h_kv"]):
            q = Q[b, :, r * g:(r + 1) * g].double()
            x = torch.einsum("nhd,td->nht", q, Kbar[b, r].double()) * (case["gamma"] * (case["alpha"] - 1.0) / math.sqrt(case["head_dim"]))
            x = x.masked_fill(~cand[:, None], -math.inf)
            some = cand.any(1)
            high = torch.where(some[:, None], x.amax(2), 0.0)
            low = high - 1.0
            for _ in range(48):
                mid = 0.5 * (low + high)
                above = (x - mid[..., None]).clamp(min=0.0).pow(e).sum(2) >= 1.0
                low, high = torch.where(above, mid, low), torch.where(above, high, mid)
            tau = torch.where(some[:, None], 0.5 * (low + high), 0.0)
            margin = x - tau[..., None]
            routed = margin.amax(1) > MARGIN
            logw = torch.log(margin.clamp(min=0.0).pow(e).mean(1).clamp(min=1e-300))
            count = routed.sum(1)
            mu = torch.where(routed, logw, 0.0).sum(1) / count.clamp(min=1)
            bias = torch.where(routed, (logw - mu[:, None]) / case["sigma"], 0.0)
            member = routed | window
            at = (b * case["h_kv"] + r) * per_head + start[:, None] + member.cumsum(1) - 1
            out["blk_idx"][at[member]] = chunk[None].expand(n, T)[member].int()
            out["blk_bias"][at[member]] = bias[member].float()
            out["count"][b, r] = member.sum(1).int()
            out["tau"][b, r * g:(r + 1) * g] = tau.T.float()
            bits = torch.zeros(n, words * 32, dtype=torch.bool, device="cuda")
            bits[:, :T] = member
            bits[row, own] = True
            out["mask"][b, r] = (bits.view(n, words, 32) * bit).sum(2).to(torch.int32)
    return out


def _prepare_backward(case, seed):
    s = synth.make_prefill_inputs(_workload(case, seed), "cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000 + 501)
    Q, K, V = s["Q"], s["K"], s["V"]
    s["dO"] = torch.randn(Q.shape, generator=g, device="cuda").to(Q.dtype)
    s["p"] = B.params_for_prefill(Q, K, V, s["dO"], **_options(case))
    s["qbar"], s["Kbar"] = _summary_query(case, seed), B.alloc_kbar(s["p"])
    B.dash_attn_block_summaries(s["p"], K, s["Kbar"], qbar=s["qbar"])
    s["routing"] = _routing(case, s["p"], Q, s["Kbar"])
    s["dQ"] = torch.empty_like(Q)
    s["dK"] = torch.empty(K.shape, device="cuda")
    s["dV"], s["dbias"] = torch.empty_like(s["dK"]), torch.zeros_like(s["routing"]["blk_bias"])
    s["dQ_route"], s["dKbar"], s["dqbar"] = torch.empty(Q.shape, device="cuda"), torch.empty_like(s["Kbar"]), torch.empty_like(s["qbar"])
    # what the header says of the two entry points: the tensor-core one for these shapes, the other for the rest
    if case["dtype"] == "bf16" and case["head_dim"] == 128 and case["block"] >= 64 and case["h_q"] > case["h_kv"]:
        s["ws"] = B.alloc_bwd_workspace(s["p"])
    return s


def prepare(case, seed):
    s = {"decode": _prepare_decode, "prefill": _prepare_prefill, "backward": _prepare_backward}[case["kind"]](case, seed)
    s.pop("planted", None)
    s["case"] = case
    return s


def run(s):
    p, case = s["p"], s["case"]
    if case["kind"] == "decode":
        if "table" in s:
            B.dash_attn_fwd_decode_paged(p, s["Q"], s["K"], s["V"], s["table"], s["Kbar"], s["kv_len"], s["O"], s["ws"])
        else:
            B.dash_attn_fwd_decode(p, s["Q"], s["K"], s["V"], s["Kbar"], s["kv_len"], s["O"], s["ws"])
        return s["O"]
    if case["kind"] == "prefill":
        if not case.get("staged"):
            B.dash_attn_fwd_prefill(p, s["Q"], s["K"], s["V"], s["O"], s["ws"])
            return s["O"]
        rt = s["routing"]
        B.dash_attn_block_summaries(p, s["K"], s["Kbar"], qbar=s["qbar"])
        B.dash_attn_select(p, s["Q"], s["Kbar"], rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], s["ws"], tau=rt["tau"])
        B.dash_attn_attend_prefill(p, s["Q"], s["K"], s["V"], rt["mask"], rt["blk_bias"], s["O"], s["ws"])
        return {"O": s["O"], "Kbar": s["Kbar"], "tau": rt["tau"], "count": rt["count"]}
    rt = s["routing"]
    grads = (s["dQ"], s["dK"], s["dV"], s["dbias"])
    if "ws" in s:
        B.dash_attn_bwd_attend_prefill_tc(p, s["Q"], s["K"], s["V"], s["dO"], rt["mask"], rt["blk_bias"], *grads, s["ws"])
    else:
        B.dash_attn_bwd_attend_prefill(p, s["Q"], s["K"], s["V"], s["dO"], rt["mask"], rt["blk_bias"], *grads)
    B.dash_attn_bwd_select_prefill(p, s["Q"], s["Kbar"], rt["count"], rt["blk_idx"], rt["tau"], s["dbias"], s["dQ_route"], s["dKbar"])
    B.dash_attn_bwd_block_summaries(p, s["K"], s["dKbar"], s["dK"], qbar=s["qbar"], dqbar=s["dqbar"])
    return {k: s[k] for k in ("dQ", "dK", "dV", "dbias", "dQ_route", "dKbar", "dqbar")}


def _routed(case, counts):
    """Expected number of routed chunks of a row with so many candidates, for each of `counts`: the logits of `synth`'s
    recipe are normal with known moments (planted chunks with another mean), thresholded here."""
    rng, g, e = np.random.default_rng(0), case["h_q"] // case["h_kv"], 1.0 / (case["alpha"] - 1.0)
    scale, sd = case["gamma"] * (case["alpha"] - 1.0), 1.0 / math.sqrt(case["block"])
    at = sorted({int(round(c)) for c in np.geomspace(1, max(1, max(counts)), 24)})
    mean = []
    for n in at:
        k = max(4, min(32, 4096 // n))
        whole = n if case["kind"] == "decode" else case["seq"] // case["block"]     # chunks the eight planted ones are among
        planted = rng.random((k, n)) < min(1.0, 8.0 / max(1, whole))
        if case["recipe"] == "tiny":
            x = scale * rng.normal(0.0, sd / case["head_dim"], (k, g, n))
        else:
            a = rng.normal(0.0, sd, (k, n)) + case["shift"] * planted
            x = scale * (0.72 * a[:, None] + rng.normal(0.0, sd, (k, g, n)))
        high = x.max(2)
        low = high - 1.0
        for _ in range(30):
            mid = 0.5 * (low + high)
            above = (np.maximum(x - mid[..., None], 0.0) ** e).sum(2) >= 1.0
            low, high = np.where(above, mid, low), np.where(above, high, mid)
        mean.append(float((x > low[..., None]).any(1).sum(1).mean()))
    return np.where(np.asarray(counts) > 0, np.interp(counts, at, mean), 0.0)


def work(case):
    b, h_q, h_kv, d, blk, L = (case[k] for k in ("batch", "h_q", "h_kv", "head_dim", "block", "local_blocks"))
    size = 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "decode":
        lens = np.asarray(_lengths(case))
        own = (lens - 1) // blk
        cand = np.maximum(own - L, 0)
        tokens = (_routed(case, cand) + np.minimum(own, L)) * blk + (lens - 1) % blk + 1
        return {"bytes": float(h_kv * (tokens.sum() * d * 2 * size + cand.sum() * d * 4) + 2 * b * h_q * d * size),
                "flops": float(h_q * (4 * d * tokens.sum() + 2 * d * cand.sum()))}
    n = case["seq"]
    row = np.arange(n)
    own = row // blk
    cand = np.maximum(own - L, 0)
    tokens = float(((_routed(case, cand) + np.minimum(own, L)) * blk + row % blk + 1).sum())
    picked = float((_routed(case, cand) + np.minimum(own, L)).sum())
    score = b * h_q * 2.0 * d * float(cand.sum())
    q, kv, kbar = b * n * h_q * d, b * n * h_kv * d, b * h_kv * (n // blk) * d
    if case["kind"] == "prefill":
        moved = size * (2 * q + 2 * kv)
        if case.get("staged"):
            moved += 4 * kbar + b * (h_q + h_kv) * n * 4
        return {"bytes": float(moved), "flops": b * h_q * 4.0 * d * tokens + score + 2.0 * kv}
    # backward: five products per attended token, three per routed chunk; lists and their gradients beside the tensors
    moved = size * (3 * q + 2 * kv) + 4 * (q + 2 * kv + 2 * kbar) + b * h_kv * picked * 12 + b * h_q * n * 4
    return {"bytes": float(moved), "flops": b * h_q * (10.0 * d * tokens + 6.0 * d * picked) + 6.0 * kv}


def tolerance(case):
    if case["kind"] == "prefill":
        # a chunk on the threshold may fall to either side: counts of a few rows differ by one
        if case["dtype"] == "f32":
            # 1e-5 of 32-bit sums; log w of chunks near the threshold multiplies it
            return {"rel": 5e-5, "max": 5e-3, "differ": 1e-3}
        return {"rel": 1e-2, "differ": 1e-3}
    return {"rel": 1e-2}
