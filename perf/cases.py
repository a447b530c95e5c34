"""The work that is timed when this framework's speed is compared between two states of its code.

A case is one call, or the few calls that belong together, of a serving loop: a prompt batch entering the cache
(`prefill`), one denoise step of a batch (`step`), a whole request (`request`: prefill and block-by-block decoding),
the same with several blocks in flight (`multiblock`), a refresh of the stored prefixes (`refresh`), and the
construction of noisy training sequences from decoding trajectories (`trajectory`).  Model shapes, block sizes,
thresholds and batch sizes are those of `paper_2601_07568_b200/synth_inputs.py`, `bench.py` and the tests.

Weights.  Randomly initialised models put every decision of threshold decoding near a tie, so that two correct
implementations decode different texts.  The weights here are drawn with the usual depth-scaled initialisation
(embeddings N(0, 1), input projections N(0, 1.28^2 / fan_in), output projections divided by sqrt(2 layers) on top),
and one attention head of layer 0 is set to what trained models are full of, a copying head: its query and key
depend on a constant embedding dimension only and are turned against each other by `jump` RoPE positions, so it reads
the token `jump` positions back, and the LM head knows the copied vector of every token.  A masked position whose
source is known is then predicted with certainty (top logit 24 to 40, runner-up about half), one whose source is still
masked is as good as undecided (the best token far below the threshold): every decision has a margin far above
rounding, and a denoise step commits `jump` tokens, about what the benchmark's workloads commit (8 of 32, 17 of 64).
All matrices stay dense, and no kernel does less work on these values than on others.
"""
from __future__ import annotations

import dataclasses
import math

import torch

from paper_2601_07568_b200 import binding as d3
from paper_2601_07568_b200 import synth_inputs as si

# (logits unscaled: the factor 20 of these shapes is there to spread the confidences of a random model)
SHAPES = {name: dataclasses.replace(shape, logit_scale=1.0) for name, shape in (("tiny", si.TINY), ("8b", si.LLADA8B), ("7b", si.QWEN7B))}
ANCHOR = 8.0  # the constant first embedding dimension


# ----------------------------------------------------------------------------- the cases
def _case(name, kind, model, bs, p_min, p_max, block=32, gen=0, jump=8, threshold=0.9, entropy=False, temperature=0.0,
          active=1, refresh=0):
    return {"name": name, "kind": kind, "model": model, "bs": bs, "p_min": p_min, "p_max": p_max, "block": block, "gen": gen,
            "jump": jump, "threshold": threshold, "entropy": entropy, "temperature": temperature, "active": active, "refresh": refresh}


def listed():
    return [
        # The smallest model and the fp32 path: a request on it is launches and round trips.
        _case("tiny_fp32_request", "request", "tiny", 1, 32, 32, block=16, gen=64, jump=4),
        # Data generation for distillation: ranks and noisy sequences of 16384 recorded responses of 256 tokens.
        _case("trajectory_16384x256", "trajectory", "tiny", 16384, 0, 0, gen=256),
        # One user, interactive: a denoise step in the middle of a response, 32 rows, an odd prefix.
        _case("step_8b_b1", "step", "8b", 1, 391, 391),
        # The same user's whole request as the benchmark counts it (256 prompt tokens, 256 generated).
        _case("request_8b_b1", "request", "8b", 1, 256, 256, gen=256),
        # The same with up to four blocks in flight and the entropy criterion: rounds of up to 128 rows.
        _case("multiblock_8b_b1", "multiblock", "8b", 1, 256, 256, gen=256, jump=18, threshold=0.4, entropy=True, active=4),
        # Four users with ragged prompts, temperature 0.1: rounds of 128 rows.
        _case("request_8b_b4_sampled", "request", "8b", 4, 101, 333, gen=64, temperature=0.1),
        # Grouped query heads, batch 8: a step of 256 rows.
        _case("step_7b_b8", "step", "7b", 8, 512, 960),
        # Long prefixes, blocks of 64, batch 4: a step that reads as much cache as weights.
        _case("step_8b_b4_long", "step", "8b", 4, 4096, 4700, block=64, jump=17, threshold=0.8),
        # A full batch of 32 ragged sequences: a step of 1024 rows.
        _case("step_8b_b32", "step", "8b", 32, 128, 735),
        # The same batch's prompts entering the cache, padded to the longest.
        _case("prefill_8b_b32", "prefill", "8b", 32, 128, 512),
        # Refresh of one sequence's stored prefix: 501 rows that all see one another.
        _case("refresh_7b_b1", "refresh", "7b", 1, 501, 501),
        # Four long prompts.
        _case("prefill_8b_b4_long", "prefill", "8b", 4, 4000, 4096, block=64, jump=17),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "prefill", "prefill", "request", "multiblock", "refresh", "tiny", "trajectory"])
    model = rng.choice(["8b", "8b", "7b"])
    entropy = rng.random() < 0.25
    threshold = 0.4 if entropy else rng.choice([0.8, 0.9])
    if kind == "tiny":
        block = rng.choice([8, 16, 32])
        p = _log_int(rng, 16, 90)
        bs = rng.choice([1, 2, 3])
        c = _case("", "request", "tiny", bs, max(8, p - 7 * (bs - 1)), p, block=block, gen=block * rng.randint(2, 5), jump=4,
                  threshold=threshold, entropy=entropy)
    elif kind == "trajectory":
        c = _case("", "trajectory", "tiny", _log_int(rng, 64, 24000), 0, 0, gen=32 * rng.randint(2, 16))
    elif kind == "step":
        block = rng.choice([32, 32, 32, 64])
        bs = _log_int(rng, 1, 32 if block == 32 else 16)
        p = _log_int(rng, 60, min(4500, 24000 // bs))
        c = _case("", "step", model, bs, max(40, int(p * rng.uniform(0.3, 1.0))), p, block=block, jump=block // 4,
                  threshold=threshold, entropy=entropy, temperature=rng.choice([0.0, 0.0, 0.1]))
    elif kind == "prefill":
        bs = _log_int(rng, 1, 32)
        p = _log_int(rng, 40, min(4096, 14000 // bs))
        c = _case("", "prefill", model, bs, max(20, int(p * rng.uniform(0.25, 1.0))), p)
    elif kind == "refresh":
        bs = rng.choice([1, 1, 2, 4])
        p = _log_int(rng, 70, 1500)
        c = _case("", "refresh", model, bs, max(40, int(p * rng.uniform(0.4, 1.0))), p)
    elif kind == "request":
        bs = rng.choice([1, 1, 2, 3, 4, 6])
        p = _log_int(rng, 50, 500)
        c = _case("", "request", model, bs, max(40, int(p * rng.uniform(0.4, 1.0))), p, gen=32 * rng.randint(1, 8 if bs == 1 else 3),
                  threshold=threshold, entropy=entropy, temperature=rng.choice([0.0, 0.1]), refresh=rng.choice([0, 0, 2]))
    else:
        bs = rng.choice([1, 1, 3])
        p = _log_int(rng, 50, 500)
        c = _case("", "multiblock", model, bs, max(40, int(p * rng.uniform(0.4, 1.0))), p, gen=32 * rng.randint(2, 6), jump=18,
                  threshold=threshold, entropy=entropy, active=rng.choice([2, 3, 4]) if bs == 1 else 2)
    if c["bs"] == 2 and c["block"] == 32 and c["model"] == "8b":
        c["bs"] = 3  # (a decode forward of exactly two such blocks was refused when this was written)
    del c["name"]
    return c


def _lengths(case):
    """Prompt lengths of the batch: spread over [p_min, p_max], the longest among them, in mixed order."""
    bs, lo, hi = case["bs"], case["p_min"], case["p_max"]
    if bs == 1:
        return [hi]
    step = next(s for s in (7, 5, 3, 11, 1) if math.gcd(s, bs) == 1)
    return [lo + (hi - lo) * ((i * step) % bs) // (bs - 1) for i in range(bs)]


# ----------------------------------------------------------------------------- what a user's program holds
class _State:
    """A context with its weights, and the buffers of the calls; the context goes when the state does."""

    def __init__(self, case):
        self.case, self.ctx = case, None

    def __del__(self):
        if self.ctx is not None:
            torch.cuda.synchronize()
            d3.d3_destroy(self.ctx)
            self.ctx = None


def _copying_head(shape, jump):
    """Rows (q, k) of one head, per unit of the anchor: RoPE turns them into a score that peaks `jump` positions back."""
    half = shape.d_head // 2
    theta = torch.tensor([float(shape.rope_theta) ** (-2.0 * k / shape.d_head) for k in range(half)], dtype=torch.float64)
    # the neighbour of the source scores 14 nats less
    amp = math.sqrt(14.0 * math.sqrt(shape.d_head) / float((1 - torch.cos(theta)).sum()))
    q = torch.cat([torch.cos(-jump * theta), torch.sin(-jump * theta)]) * amp
    k = torch.cat([torch.ones(half, dtype=torch.float64), torch.zeros(half, dtype=torch.float64)]) * amp
    return q, k


def _weights(shape, seed, jump):
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    dt = torch.bfloat16 if shape.dtype == "bf16" else torch.float32
    d, dh, f, layers, vocab = shape.d_model, shape.d_head, shape.d_ffn, shape.n_layers, shape.vocab
    nq, nkv = shape.n_q_heads * dh, shape.n_kv_heads * dh

    def normal(rows, cols, std):
        return torch.empty(rows, cols, dtype=dt, device="cuda").normal_(0.0, std, generator=gen)

    emb = normal(vocab, d, 1.0)
    emb[:, 1:1 + dh].sign_()
    emb[shape.mask_id, 1:1 + dh] = 0.0  # the mask token has no content to copy
    content = emb[:, 1:1 + dh].clone()
    # rows of one length, so that the anchor is the same after every token's norm
    emb[:, 0] = 0.0
    emb *= math.sqrt(d - 1.0) / emb.norm(dim=1, keepdim=True, dtype=torch.float32).to(dt)
    emb[:, 0] = ANCHOR
    # the copied vector: root mean square 4 where the embedding has 1, so that it outlasts the layers' updates
    basis = torch.linalg.qr(torch.empty(d, dh, dtype=torch.float32, device="cuda").normal_(0.0, 1.0, generator=gen))[0]
    spread = (basis * (4.0 * math.sqrt(d / dh))).to(dt)
    lm_head = normal(vocab, d, 1.3 / math.sqrt(d))
    top = min(40.0, 2.1 * math.sqrt(d))  # logit of a copied token, about
    lm_head.addmm_(content, spread.t(), alpha=top / (4.0 * d))
    out_scale = 1.0 / math.sqrt(2.0 * layers)
    ls = [{"wq": normal(nq, d, 1.28 / math.sqrt(d)), "wk": normal(nkv, d, 1.28 / math.sqrt(d)), "wv": normal(nkv, d, 1.28 / math.sqrt(d)),
           "wo": normal(d, nq, 1.28 / math.sqrt(nq) * out_scale), "w_gate": normal(f, d, 1.28 / math.sqrt(d)),
           "w_up": normal(f, d, 1.28 / math.sqrt(d)), "w_down": normal(d, f, 1.28 / math.sqrt(f) * out_scale)} for _ in range(layers)]
    q, k = _copying_head(shape, jump)
    anchor = ANCHOR / math.sqrt(1.0 + (ANCHOR * ANCHOR - 1.0) / d)  # its value after the norm
    first = ls[0]
    for name, rows in (("wq", q), ("wk", k)):
        first[name][:dh] = 0.0
        first[name][:dh, 0] = (rows / anchor).to(device="cuda", dtype=dt)
    first["wv"][:dh] = 0.0
    first["wv"][torch.arange(dh, device="cuda"), torch.arange(1, dh + 1, device="cuda")] = 1.0
    first["wo"][:, :dh] = spread
    return {"tok_emb": emb, "lm_head": lm_head, "layers": ls}


def _new_context(case, shape, seed):
    bs, block = case["bs"], case["block"]
    new = case["gen"] if case["gen"] else 2 * block
    max_batch = bs * case["active"]  # the workspaces for the windows of multi-block decoding are sized by max_batch
    cfg = d3.make_config(shape, block=block, max_batch=max_batch, max_seq=case["p_max"] + new,
                         max_prefill_rows=bs * (case["p_max"] + (new if case["refresh"] else 0)),
                         decide_mode=d3.D3_DECIDE_ENTROPY if case["entropy"] else d3.D3_DECIDE_CONFIDENCE)
    ctx = d3.d3_create(cfg)
    d3.d3_load_weights(ctx, _weights(shape, seed, case["jump"]), shape.n_layers)
    if case["temperature"] > 0:
        d3.d3_set_sampling(ctx, case["temperature"], seed)
    if case["refresh"]:
        d3.d3_set_cache_policy(ctx, 1, case["refresh"])
    return ctx


def prepare(case, seed):
    s = _State(case)
    gen = torch.Generator("cuda")
    gen.manual_seed(seed + 1)
    bs, block = case["bs"], case["block"]
    if case["kind"] == "trajectory":
        shape = dataclasses.replace(si.TINY, vocab=si.LLADA8B.vocab)
        n = case["gen"]
        s.ctx = d3.d3_create(d3.make_config(shape, block=block, max_batch=1, max_seq=block))
        order = torch.rand(bs, n // block, block, device="cuda", generator=gen)
        s.commit_step = (order.argsort(-1) + 1).to(torch.int32).reshape(bs, n).contiguous()
        s.y = torch.randint(0, shape.vocab - 2, (bs, n), device="cuda", generator=gen, dtype=torch.int32)
        s.start = torch.randint(0, n, (bs,), device="cuda", generator=gen, dtype=torch.int32)
        s.window = torch.randint(1, block + 1, (bs,), device="cuda", generator=gen, dtype=torch.int32)
        ratio = torch.rand(bs, device="cuda", generator=gen)
        s.unmasked = torch.ceil(ratio * s.window).to(torch.int32)
        s.rank, s.out = torch.zeros_like(s.y), torch.zeros_like(s.y)
        return s
    shape = SHAPES[case["model"]]
    s.shape = shape
    s.ctx = _new_context(case, shape, seed)
    s.lens = _lengths(case)
    s.ids = torch.randint(0, shape.vocab - 2, (bs, case["p_max"]), device="cuda", generator=gen, dtype=torch.int32)
    for b, n in enumerate(s.lens):
        s.ids[b, n:] = shape.pad_id
    s.lens_dev = torch.tensor(s.lens, dtype=torch.int32, device="cuda")
    if case["kind"] in ("step", "refresh"):
        d3.d3_prefill(s.ctx, s.ids, s.lens_dev)
    if case["kind"] == "step":
        # a block of which the first tokens have been committed by earlier steps
        known = 1 + seed % case["jump"]
        s.block0 = torch.full((bs, block), shape.mask_id, dtype=torch.int32, device="cuda")
        s.block0[:, :known] = torch.randint(0, shape.vocab - 2, (bs, known), device="cuda", generator=gen, dtype=torch.int32)
        s.mask0 = (s.block0 == shape.mask_id).to(torch.uint8)
        s.block, s.mask = s.block0.clone(), s.mask0.clone()
        s.out_pos, s.out_ids = torch.zeros_like(s.block), torch.zeros_like(s.block)
        s.out_count = torch.zeros(bs, dtype=torch.int32, device="cuda")
        s.conf = torch.zeros(bs * block, dtype=torch.float32, device="cuda")
        s.entropy, s.argmax = torch.zeros_like(s.conf), torch.zeros(bs * block, dtype=torch.int32, device="cuda")
    else:
        # the last layer's keys and values of the stored rows: what the whole forward over them ends in
        heads, dh = shape.n_kv_heads, shape.d_head
        s.kv = [torch.zeros(2, heads, n + case["gen"], dh, dtype=torch.float32, device="cuda") for n in s.lens]
        s.tokens = torch.zeros(bs, max(case["gen"], 1), dtype=torch.int32, device="cuda")
        s.when = torch.zeros_like(s.tokens)
    return s


def _stored(s):
    for b, n in enumerate(s.lens):
        d3.d3_read_kv(s.ctx, s.shape.n_layers - 1, b, 0, n + s.case["gen"], s.kv[b][0], s.kv[b][1])
    return list(s.kv)


def run(s):
    c = s.case
    if c["kind"] == "trajectory":
        d3.d3_trajectory_rank(s.ctx, s.commit_step, s.rank)
        d3.d3_noisy_sequence(s.ctx, s.y, s.rank, s.start, s.window, s.unmasked, s.out)
        return s.rank, s.out
    if c["kind"] == "step":
        s.block.copy_(s.block0)
        s.mask.copy_(s.mask0)
        d3.d3_denoise_step(s.ctx, s.block, s.mask, c["threshold"], s.out_pos, s.out_ids, s.out_count)
        d3.d3_get_step_stats(s.ctx, s.conf, s.entropy, s.argmax, c["bs"])
        # (the arg max of the rows that stay masked is a near-tie of a flat distribution; the committed ones are in out_ids)
        return s.block, s.mask, s.out_pos, s.out_ids, s.out_count, s.conf, s.entropy
    if c["kind"] == "refresh":
        d3.d3_refresh_cache(s.ctx, c["bs"])
        return _stored(s)
    d3.d3_prefill(s.ctx, s.ids, s.lens_dev)
    if c["kind"] == "prefill":
        return _stored(s)
    if c["kind"] == "multiblock":
        d3.d3_generate_multiblock(s.ctx, c["gen"], c["threshold"], s.tokens, c["active"], s.when)
    else:
        d3.d3_generate(s.ctx, c["gen"], c["threshold"], s.tokens, s.when)
    return [s.tokens, s.when] + _stored(s)


# ----------------------------------------------------------------------------- what a pass cannot do without
def _forward_work(shape, rows_of, seen_of, head):
    """(bytes, flops) of one forward: sequence b brings rows_of[b] rows that see seen_of[b] positions each (their own included)."""
    d, f, vocab, dh = shape.d_model, shape.d_ffn, shape.vocab, shape.d_head
    nq, nkv = shape.n_q_heads * dh, shape.n_kv_heads * dh
    e = 2 if shape.dtype == "bf16" else 4
    rows = sum(rows_of)
    layer = (nq + 2 * nkv) * d + d * nq + 3 * f * d
    params = shape.n_layers * layer + (vocab * d if head else 0)
    cached = sum(n - r for n, r in zip(seen_of, rows_of))  # positions read from the cache
    kv = shape.n_layers * 2 * nkv * e * (cached + rows)    # the rows' own keys and values are written
    flops = 2.0 * rows * params + shape.n_layers * 4.0 * nq * sum(r * n for r, n in zip(rows_of, seen_of))
    return params * e + rows * d * e + kv, flops


def work(case):
    bs, block, gen, jump = case["bs"], case["block"], case["gen"], case["jump"]
    if case["kind"] == "trajectory":
        # rank: one read, one write; noisy sequence: two reads, one write (a third pass over the ranks is not needed)
        return {"bytes": 4.0 * bs * gen * 4 + 12.0 * bs, "flops": 0.0}
    shape, lens = SHAPES[case["model"]], _lengths(case)
    if case["kind"] == "step":
        b, fl = _forward_work(shape, [block] * bs, [n + block for n in lens], True)
        return {"bytes": b, "flops": fl}
    total_b, total_f = _forward_work(shape, lens, lens, False)
    if case["kind"] in ("prefill", "refresh"):
        return {"bytes": total_b, "flops": total_f}
    if case["kind"] == "multiblock":
        rounds, done = -(-gen // jump), 0
        for r in range(rounds + 1):  # the last one over the last block's final tokens
            first = min(done // block, gen // block - 1) * block
            rows = min(case["active"] * block, gen - first) if r < rounds else block
            b, fl = _forward_work(shape, [rows] * bs, [n + first + rows for n in lens], r < rounds)
            total_b, total_f, done = total_b + b, total_f + fl, done + jump
        return {"bytes": total_b, "flops": total_f}
    for j in range(gen // block):
        seen = [n + (j + 1) * block for n in lens]
        for _ in range(-(-block // jump)):
            b, fl = _forward_work(shape, [block] * bs, seen, True)
            total_b, total_f = total_b + b, total_f + fl
        # the finished block's own forward can share the next one's pass over the weights
        b, fl = _forward_work(shape, [block] * bs, seen, False)
        total_b, total_f = total_b + (b if j == gen // block - 1 else 0), total_f + fl
        if case["refresh"] and (j + 1) % case["refresh"] == 0 and j + 1 < gen // block:
            b, fl = _forward_work(shape, seen, seen, False)
            total_b, total_f = total_b + b, total_f + fl
    return {"bytes": total_b, "flops": total_f}


def tolerance(case):
    """Tokens, positions and commit steps are whole numbers decided with wide margins: they have to be the same."""
    if case["kind"] == "trajectory":
        return "exact"
    if case["model"] == "tiny":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}  # 32-bit sums
    # Measured between schedules of the same forward (one launch or one kernel per matmul, split or whole K, attention on
    # either tensor-core path), whose fp32 sums differ in order and so round differently to bf16 at every storage point:
    if case["kind"] == "step":
        # confidence and entropy: 2.3e-5, at most 8e-5 of the root mean square; a sampled token among near-equals of a flat
        # distribution may be another one, whose probability (1e-3) then differs by as much
        return {"rel": 1e-3, "max": 1e-2, "differ": 0.0} if case["temperature"] > 0 else {"rel": 1e-4, "max": 4e-4, "differ": 0.0}
    # keys and values of the last layer: 0.25 %, at most 1.2 % of the root mean square
    return {"rel": 0.01, "max": 0.05, "differ": 0.0}


# ----------------------------------------------------------------------------- the same in 64 bits
def _forward64(shape, w, ids, segments):
    """The model over whole sequences in 64-bit floats: ids[b] [n], segments[b] [n] ascending; a row sees the rows of its own
    and earlier segments.  Returns the residual streams after the last layer and the last layer's keys and values [heads, n, d_head]."""
    f64 = torch.float64
    dh, hq, hkv, half = shape.d_head, shape.n_q_heads, shape.n_kv_heads, shape.d_head // 2
    cut = [len(i) for i in ids]
    x = w["tok_emb"][torch.cat(ids).long()].to(f64)
    inv = torch.tensor([float(shape.rope_theta) ** (-2.0 * k / dh) for k in range(half)], dtype=f64, device="cuda")
    ang = torch.cat([torch.arange(n, dtype=f64, device="cuda") for n in cut])[:, None] * inv
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]

    def normed(v):
        return v * torch.rsqrt(v.pow(2).mean(1, keepdim=True) + shape.rms_eps)

    def times(v, m):
        return v @ m.to(f64).t()

    def turned(v):
        a, b = v[..., :half], v[..., half:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    kv = None
    for m in w["layers"]:
        h = normed(x)
        q = turned(times(h, m["wq"]).view(-1, hq, dh))
        k = turned(times(h, m["wk"]).view(-1, hkv, dh))
        v = times(h, m["wv"]).view(-1, hkv, dh)
        kv = [(a.transpose(0, 1), b.transpose(0, 1)) for a, b in zip(k.split(cut), v.split(cut))]
        o = []
        for qb, (kb, vb), seg in zip(q.split(cut), kv, segments):
            hidden = seg[None, :] > seg[:, None]
            heads = []
            for g in range(hkv):
                per = hq // hkv
                sc = qb[:, g * per:(g + 1) * per].transpose(0, 1) @ kb[g].t() / math.sqrt(dh)
                heads.append(sc.masked_fill_(hidden, -math.inf).softmax(-1) @ vb[g])
            o.append(torch.cat(heads).transpose(0, 1).reshape(len(seg), hq * dh))
        x = x + times(torch.cat(o), m["wo"])
        h = normed(x)
        x = x + times(torch.nn.functional.silu(times(h, m["w_gate"])) * times(h, m["w_up"]), m["w_down"])
    return normed(x).split(cut), kv


def exact(case, seed):
    """What `run` returns, in 64 bits: keys and values, confidences and entropies (the tokens are whole numbers)."""
    if case["kind"] == "trajectory":
        return None
    shape, lens, bs, block = SHAPES[case["model"]], _lengths(case), case["bs"], case["block"]
    gen = torch.Generator("cuda")
    gen.manual_seed(seed + 1)
    prompts = torch.randint(0, shape.vocab - 2, (bs, case["p_max"]), device="cuda", generator=gen, dtype=torch.int32)
    ids = [prompts[b, :n] for b, n in enumerate(lens)]
    segments = [torch.zeros(n, dtype=torch.int64, device="cuda") for n in lens]
    w = _weights(shape, seed, case["jump"])
    if case["kind"] == "step":
        known = 1 + seed % case["jump"]
        rows = torch.full((bs, block), shape.mask_id, dtype=torch.int32, device="cuda")
        rows[:, :known] = torch.randint(0, shape.vocab - 2, (bs, known), device="cuda", generator=gen, dtype=torch.int32)
        x, _ = _forward64(shape, w, [torch.cat([a, b]) for a, b in zip(ids, rows)], [torch.cat([s, torch.ones_like(s[:1]).expand(block)]) for s in segments])
        head = w["lm_head"].to(torch.float64)
        conf, entropy = [], []
        for v in x:
            logits = v[-block:] @ head.t()
            logits[:, shape.mask_id] = -math.inf
            p = logits.softmax(-1)
            conf.append(p.max(-1).values)
            entropy.append(torch.special.entr(p).sum(-1))
        return None, None, None, None, None, (torch.cat(conf) if case["temperature"] == 0 else None), torch.cat(entropy)
    if case["gen"]:
        # the response copies the token `jump` positions back; a position sees the prompt, the blocks before its own and its own
        # (a refresh makes one segment of what is stored by then)
        joined = 0
        if case["refresh"]:
            joined = (case["gen"] // block - 1) // case["refresh"] * case["refresh"]
        after = torch.arange(case["gen"], device="cuda") // block + 1
        after[:joined * block] = 0
        for b in range(bs):
            last = ids[b][-case["jump"]:]
            ids[b] = torch.cat([ids[b], last.repeat(-(-case["gen"] // case["jump"]))[:case["gen"]]])
            segments[b] = torch.cat([segments[b], after])
    _, kv = _forward64(shape, w, ids, segments)
    stored = [torch.stack(pair) for pair in kv]
    return stored if not case["gen"] else [None, None] + stored
