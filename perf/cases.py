"""Performance cases of the KeepKV library: what a serving loop has it do, at the sizes it does it.

Every case goes through the binding's entry points, eagerly, on the current stream.  Operations (``op``):

  step      decode: ``steps`` tokens through ``layers`` layer caches, ``keepkv_decode_step`` per token and layer
            (append, attention and score update in one launch).  The lengths are set back at the start of a pass,
            so that every pass does the same work.
  host      the same from pinned host memory: ``keepkv_decode_step_host_layers`` per token, and the wait for its
            result, as a loop does that samples the next token on the host.
  attend    ``keepkv_decode_attention`` with score update over a complete cache (first token after a prompt; the
            periodic mode's scoring of the complete cache).
  scores    ``keepkv_prefill_scores``: score estimate of a whole prompt from its last ``window`` queries.
  compress  ``keepkv_compress`` of ``layers`` caches to the budget: a prompt's first compression, or (``steady``) the
            recurring one of a cache that is one period over its budget.
  merge     a prompt's keys and values are put into the cache and ``keepkv_compress_merge_first`` cuts it.

The data follow ``workloads.py``: normal keys with four outlier channels per unit, planted heavy hitters that share a
direction with the queries, normal values; caches that have been compressed before also carry votes above 1.
``n`` is the number of entries per sequence; with ``n_min`` > 0 the lengths of a batch are spread evenly over
[n_min, n] in an order drawn from the seed, and budgets follow the lengths.
"""
import math

import torch

from paper_2504_09936_b200 import binding as kk

N_SINK, RECENT, THRESHOLD, ALPHA = 4, 0.8, 0.8, 0.9


def listed():
    return [
        # A toy-sized model (64 channels, a few dozen entries): nothing but the cost of a call.
        _step("step-tiny", B=1, H_q=8, H_kv=2, d=64, n=67, layers=4, steps=4),
        # One user chatting with a Llama-3-8B-shaped model, cache cut to 20 % of 8k: one token through 32 layers.
        _step("step-single", B=1, H_q=32, H_kv=8, d=128, n=1655, layers=32, steps=1),
        # The same model serving a small batch in the middle of a compression period.
        _step("step-gqa", B=8, H_q=32, H_kv=8, d=128, n=1702, layers=8, steps=2),
        # Llama-2-7B-shaped multi-head attention with a short cache (10 % of 4k): many units, few entries each.
        _step("step-mha", B=16, H_q=32, H_kv=32, d=128, n=442, layers=6, steps=2),
        # Serving-scale batch of a 64-head model, sequences of unequal length.
        _step("step-ragged", B=64, H_q=64, H_kv=8, d=128, n=1702, n_min=418, layers=2, steps=2),
        # A decode loop whose queries and new tokens come from, and results go to, the host every token.
        _step("host-gqa", op="host", B=8, H_q=32, H_kv=8, d=128, n=1702, layers=8, steps=2),
        # First token after two 32k prompts of a Mistral-7B-shaped model, before anything is evicted.
        _case("attend-long", "attend", B=2, H_q=32, H_kv=8, d=128, n=32768, layers=1),
        # End of a batch's prefill: scores of every prompt entry from the last 32 queries.
        _case("scores-gqa", "scores", B=8, H_q=32, H_kv=8, d=128, n=8192, layers=1, window=32),
        # The first compression of these prompts, 8k to 20 %.
        _case("compress-prompt", "compress", B=8, H_q=32, H_kv=8, d=128, n=8192, layers=1, ratio=0.2),
        # The first compression of long prompts of unequal length, 10 % of each.
        _case("compress-ragged", "compress", B=16, H_q=64, H_kv=8, d=128, n=16384, n_min=4096, layers=1, ratio=0.1),
        # The recurring compression: every layer is 128 tokens over its budget of 1638.
        _case("compress-steady", "compress", B=8, H_q=32, H_kv=8, d=128, n=1766, layers=4, excess=128),
        # Prefill compression under the merge-first policy, prompts of about 6k.
        _case("merge-prompt", "merge", B=4, H_q=32, H_kv=8, d=128, n=6007, layers=1, ratio=0.2),
    ]


def draw(rng):
    while True:
        case = _drawn(rng)
        w = work(case)
        if w["bytes"] <= 1e9 and w["flops"] <= 3e11:   # no more than the largest listed case
            return case


def _drawn(rng):
    op = rng.choice(["step", "step", "step", "host", "attend", "scores", "compress", "compress", "steady", "merge"])
    d = rng.choice([128, 128, 128, 64])
    H_q, H_kv = rng.choice([(32, 8), (32, 8), (32, 32), (16, 8), (64, 8), (8, 2)])
    if op in ("step", "host"):
        B, n = _log(rng, 1, 64), _log(rng, 48, 4096)
        n_min = rng.choice([0, 0, max(1, n // 4)]) if B > 2 else 0
        layers = max(2, min(32 if op == "step" else 8, int(300e6 / (B * H_kv * n * (4 * d + 12)))))
        return _step(None, op=op, B=B, H_q=H_q, H_kv=H_kv, d=d, n=n, n_min=n_min, layers=layers, steps=rng.choice([1, 2, 3]))
    if op == "steady":
        excess = rng.randint(16, 128)
        return _case(None, "compress", B=_log(rng, 1, 32), H_q=H_q, H_kv=H_kv, d=d, n=_log(rng, 256, 2500) + excess,
                     layers=rng.choice([1, 2, 4]), excess=excess)
    B, n = _log(rng, 1, 16), _log(rng, 700, 8192 if op == "merge" else 32768)
    n_min = rng.choice([0, 0, n // 4]) if B > 2 else 0
    more = {"attend": {}, "scores": {"window": rng.choice([1, 8, 16, 32, 32])}}.get(op, {"ratio": rng.choice([0.1, 0.2, 0.3])})
    return _case(None, op, B=B, H_q=H_q, H_kv=H_kv, d=d, n=n, n_min=n_min, layers=1, **more)


def work(case):
    """Bytes each input or output is read or written with once, and the multiply-adds of the products."""
    B, H_q, H_kv, d, L = case["B"], case["H_q"], case["H_kv"], case["d"], case["layers"]
    G = H_q // H_kv
    lens = _lens(case)
    n = H_kv * sum(lens)
    if case["op"] in ("step", "host"):
        T = case["steps"]
        n = sum(H_kv * sum(v + t + 1 for v in lens) for t in range(T))
        return {"bytes": L * (n * (4 * d + 12) + T * B * (H_q * (4 * d + 4) + H_kv * 8 * d)), "flops": L * n * 4.0 * d * G}
    if case["op"] == "attend":
        return {"bytes": n * (4 * d + 12) + B * H_q * (4 * d + 4), "flops": n * 4.0 * d * G}
    if case["op"] == "scores":
        W = case["window"]
        return {"bytes": n * (2 * d + 4) + B * H_q * W * 2 * d, "flops": n * 2.0 * d * G * W}
    buds = _budgets(case, lens)
    kept = H_kv * sum(buds)
    if case["op"] == "merge":   # the prompt's rows come in once; every pair of a unit's entries is compared
        return {"bytes": n * (4 * d + 4) + kept * (4 * d + 8), "flops": 2.0 * d * H_kv * sum(v * v for v in lens)}
    pairs = H_kv * sum((v - b) * b for v, b in zip(lens, buds))
    return {"bytes": L * (n * (2 * d + 8) + kept * (6 * d + 8)), "flops": L * 2.0 * d * pairs}


def tolerance(case):
    if case["op"] == "scores":   # logarithms of fp32 sums of approximated exponentials, over values of order 1
        return {"rel": 1e-5, "max": 1e-4}
    # bf16 outputs and rows: half a unit in the last place is 2^-9 of the value on either side
    return {"rel": 5e-3, "max": 0.1, "differ": 1e-3}


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    op, B, H_q, H_kv, d, L = case["op"], case["B"], case["H_q"], case["H_kv"], case["d"], case["layers"]
    T = case.get("steps", 0)
    lens = _lens(case)
    lens = [lens[i] for i in torch.randperm(B, device="cuda", generator=g).tolist()]
    N_cap = -(-(case["n"] + max(T, 1)) // 64) * 64
    steady = case.get("excess", 0) > 0
    budget = _budgets(case, lens)
    recent = [int(RECENT * max(b - N_SINK, 0)) for b in budget]
    p = kk.make_params(B, H_q, H_kv, d, N_cap, n_sink=N_SINK, n_recent=recent[0], ema_alpha=ALPHA, merge_threshold=THRESHOLD,
                       flags=kk.FLAG_COMPRESS_STEADY if steady else 0)
    s = {"op": op, "p": p, "ws": kk.new_workspace(p), "status": kk.new_status()}
    s["lens"] = torch.tensor(lens, dtype=torch.int32, device="cuda")
    first = op in ("attend", "scores", "merge") or (op == "compress" and not steady)   # a prompt: nothing merged so far
    anchor = torch.randn(L, B, H_kv, 1, d, device="cuda", generator=g)
    s["K"], s["V"], s["votes"], s["lscore"] = _rows(g, anchor, case, N_cap, lens, first)
    s["seq"] = s["lens"].repeat(L, 1)
    s["caches"] = _caches(s["K"], s["V"], s["votes"], s["lscore"], s["seq"])

    if op in ("step", "host"):
        s["seq0"] = s["seq"].clone()
        # the layers' caches differ, so a call never follows a kernel that writes its own; the pass's first one does
        s["p_idle"] = kk.make_params(B, H_q, H_kv, d, N_cap, n_sink=N_SINK, n_recent=recent[0], ema_alpha=ALPHA,
                                     merge_threshold=THRESHOLD, flags=kk.FLAG_CACHE_IDLE)
        q = _queries(g, anchor, T, H_q)
        k, v = (torch.randn(T, L, B, H_kv, d, device="cuda", generator=g).bfloat16() for _ in range(2))
        if op == "step":
            s["out"] = torch.zeros_like(q)
            s["lse"] = torch.zeros(T, L, B, H_q, device="cuda")
            s["calls"] = [(s["p_idle"] if t + l else p, s["caches"][l], q[t, l], k[t, l], v[t, l], s["out"][t, l], s["lse"][t, l])
                          for t in range(T) for l in range(L)]
        else:
            s["host_in"], s["host_out"], s["dev_in"] = [], [], _packed(q[0].clone(), k[0].clone(), v[0].clone())
            s["dev_out"] = torch.empty_like(q[0])
            for t in range(T):
                s["host_in"].append(_packed(q[t], k[t], v[t], host=True))
                s["host_out"].append(torch.zeros(q[t].shape, dtype=q.dtype, pin_memory=True))
            s["stream"] = torch.cuda.current_stream()
    elif op == "attend":
        s["q"] = _queries(g, anchor, 1, H_q)[0, 0]
        s["out"] = torch.zeros_like(s["q"])
        s["lse"] = torch.zeros(B, H_q, device="cuda")
    elif op == "scores":
        s["q"] = _queries(g, anchor, case["window"], H_q)[:, 0].permute(1, 2, 0, 3).contiguous()
    else:
        ragged = case["n_min"] > 0
        s["budget"] = torch.tensor(budget, dtype=torch.int32, device="cuda") if ragged else budget[0]
        s["recent"] = torch.tensor(recent, dtype=torch.int32, device="cuda") if ragged else None
        s["most"] = max(budget)
        s["other"] = [torch.zeros_like(s[x]) for x in ("K", "V", "votes", "lscore", "seq")]
        s["other_caches"] = _caches(*s["other"])
        s["kept"] = torch.zeros(L, B, H_kv, N_cap, dtype=torch.int32, device="cuda")
        s["target"] = torch.zeros_like(s["kept"])
        s["stats"] = torch.zeros(L, B * H_kv, len(kk.STATS_FIELDS), dtype=torch.int32, device="cuda")
        if op == "merge":   # the prompt's keys and values as the model's prefill leaves them: without spare rows
            n = case["n"]
            s["prompt"] = [s[x][:, :, :, :n].clone() for x in ("K", "V", "lscore")]
    return s


def run(s):
    op, p, ws, status = s["op"], s["p"], s["ws"], s["status"]
    if op == "step":
        s["seq"].copy_(s["seq0"])
        for p_call, cache, q, k, v, out, lse in s["calls"]:
            kk.keepkv_decode_step(p_call, cache, q, k, v, out, lse, True, ws, status)
        return s["out"], s["lse"], s["lscore"], s["K"], s["V"], s["votes"], s["seq"], status
    if op == "host":
        s["seq"].copy_(s["seq0"])
        q_dev, k_dev, v_dev = s["dev_in"]
        for (q, k, v), out in zip(s["host_in"], s["host_out"]):
            kk.keepkv_decode_step_host_layers(s["p_idle"], s["caches"], q, k, v, out, q_dev, k_dev, v_dev, s["dev_out"],
                                              True, ws, status)
            s["stream"].synchronize()
        return s["host_out"], s["lscore"], s["K"], s["V"], s["votes"], s["seq"], status
    if op == "attend":
        kk.keepkv_decode_attention(p, s["caches"][0], s["q"], s["out"], s["lse"], True, ws, status)
        return s["out"], s["lse"], s["lscore"], status
    if op == "scores":
        kk.keepkv_prefill_scores(p, s["caches"][0], s["q"], status)
        return s["lscore"], status
    if op == "compress":
        for l, (src, dst) in enumerate(zip(s["caches"], s["other_caches"])):
            kk.keepkv_compress(p, src, dst, s["budget"], ws, status, n_recent_dev=s["recent"], retained_idx=s["kept"][l],
                               target=s["target"][l], stats=s["stats"][l])
        return _valid(s, *s["other"]), s["target"], s["stats"], status
    K, V, lscore = s["prompt"]
    n = K.shape[3]
    s["K"][:, :, :, :n].copy_(K)
    s["V"][:, :, :, :n].copy_(V)
    s["lscore"][:, :, :, :n].copy_(lscore)
    s["votes"].fill_(1.0)
    s["seq"].copy_(s["lens"])
    kk.keepkv_compress_merge_first(p, s["caches"][0], s["other_caches"][0], s["budget"], ws, status, n_recent_dev=s["recent"],
                                   retained_idx=s["kept"][0], stats=s["stats"][0])
    return _valid(s, s["K"], s["V"], s["votes"], s["lscore"], s["seq"]), s["stats"], status


def _valid(s, K, V, votes, lscore, seq):
    """A compressed cache and the kept entries' places, without the rows that no sequence's budget reaches."""
    m = s["most"]
    return [x[:, :, :, :m] for x in (K, V, votes, lscore, s["kept"])] + [seq]


def _case(name, op, B, H_q, H_kv, d, n, layers, n_min=0, **more):
    case = {"op": op, "B": B, "H_q": H_q, "H_kv": H_kv, "d": d, "n": n, "n_min": n_min, "layers": layers, **more}
    return {"name": name, **case} if name else case


def _step(name, op="step", **more):
    return _case(name, op, **more)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lens(case):
    B, n, lo = case["B"], case["n"], case["n_min"]
    return [n] * B if lo == 0 else [n - (n - lo) * i // (B - 1) for i in range(B)]


def _budgets(case, lens):
    if case.get("excess", 0) > 0:
        return [v - case["excess"] for v in lens]
    return [int(case.get("ratio", 0.2) * v + 0.5) for v in lens]


def _rows(g, anchor, case, N_cap, lens, first):
    """Keys, values, votes and score estimates of ``layers`` caches; rows past a sequence's length hold left-overs."""
    B, H, d, L = case["B"], case["H_kv"], case["d"], case["layers"]
    rand = {"device": "cuda", "generator": g}
    K = torch.randn(L, B, H, N_cap, d, **rand)
    strong = torch.rand(L, B, H, 1, d, **rand).argsort(-1) < 4           # four outlier channels per unit
    K *= torch.where(strong, 8.0, 1.0)
    n_hh = min(64, min(lens) // 8)
    a = anchor / anchor.norm(dim=-1, keepdim=True)
    z = torch.randn(L, B, H, n_hh, d, **rand)
    z -= (z * a).sum(-1, keepdim=True) * a
    size = K[:, :, :, :256].norm(dim=-1).mean(-1)[..., None, None]
    at = torch.rand(L, B, H, min(lens), **rand).topk(n_hh).indices[..., None].expand(-1, -1, -1, -1, d)
    K.scatter_(3, at, size * (0.6 * a + 0.8 * z / z.norm(dim=-1, keepdim=True)))
    seen = 0.9 * anchor + math.sqrt(0.19) * torch.randn(L, B, H, 2, d, **rand)
    lscore = (torch.matmul(K, seen.transpose(-1, -2)) / math.sqrt(d)).logsumexp(-1) - math.log(2.0)
    lscore += 0.1 * torch.randn(lscore.shape, **rand)
    votes = torch.ones(L, B, H, N_cap, device="cuda")
    if not first:   # a tenth of the entries have taken others in
        votes += torch.randint(1, 5, votes.shape, **rand) * (torch.rand(votes.shape, **rand) < 0.1)
    V = torch.randn(L, B, H, N_cap, d, dtype=torch.bfloat16, **rand)
    return K.bfloat16(), V, votes, lscore


def _caches(K, V, votes, lscore, seq):
    return [kk.Cache(*layer) for layer in zip(K, V, votes, lscore, seq)]


def _queries(g, anchor, T, H_q):
    """Queries of T steps that stay near their unit's anchor: bf16 [T, layers, B, H_q, d]."""
    L, B, H, _, d = anchor.shape
    eps = torch.randn(T, L, B, H, H_q // H, d, device="cuda", generator=g)
    return (0.9 * anchor + math.sqrt(0.19) * eps).reshape(T, L, B, H_q, d).bfloat16()


def _packed(q, k, v, host=False):
    """The three, back to back in one buffer of their device, or of pinned host memory."""
    flat = torch.cat([x.reshape(-1) for x in (q, k, v)])
    if host:
        flat = torch.empty(flat.shape, dtype=flat.dtype, pin_memory=True).copy_(flat)
    return [x.view(o.shape) for x, o in zip(flat.split([q.numel(), k.numel(), v.numel()]), (q, k, v))]
