"""The work whose speed is looked after: what a program that uses this framework has it do, through the public
calls of ``binding`` and ``engine``.  Model shapes are the presets of ``synth`` (random-init weights); batches,
contexts, numbers of draft tokens and prompt lengths cover what those presets, the benchmark and the tests use.

Kinds of a case
  tail        verify_from_logits: the vocabulary-wide accept / reject / resample step on supplied logits
  generate    Engine.generate of a small fp32 model: prompt pass, iterations, host polling
  iteration   Engine.spec_iteration: K draft steps and the verification pass that judges them
  verify      target_verify of supplied draft tokens and distributions
  decode      Engine.ar_step: the plain one-row decode step
  prefill     Engine.prefill: the prompt pass of the target and, where there is one, of the draft
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_04951_b200 import binding as B, engine, synth

KV_STD = 1.0            # cached keys and values of a random-init model are about unit normal
DRAFT_SEED = 7919       # the draft's weights are another model's


def _case(kind, model="llama-7b", batch=1, K=4, ctx=2048, temperature=1.0, **more):
    return dict(kind=kind, model=model, batch=batch, K=K, ctx=ctx, temperature=temperature, **more)


def _tail(batch, K, vocab, temperature, top_k, top_p, export):
    return dict(kind="tail", batch=batch, K=K, vocab=vocab, temperature=temperature, top_k=top_k, top_p=top_p, export=export)


def listed():
    named = [
        # one sequence's accept / resample step in a serving loop that runs the model elsewhere: the smallest call
        ("tail-b1", _tail(1, 4, 32000, 1.0, 0, 1.0, False)),
        # the same for a batch, under a top-k and top-p restriction, with the probability rows exported
        ("tail-restricted-b8", _tail(8, 5, 50304, 0.8, 50, 0.9, True)),
        # a whole generation of the fp32 GPT-2-like model: hundreds of tiny calls, latency and launches are everything
        ("generate-tiny", _case("generate", "tiny", K=4, ctx=32, iters=16)),
        # interactive use of a small model: one sequence, short context, a stand-alone draft model
        ("iteration-1.4b", _case("iteration", "neox-1.4b", K=5, ctx=211, temperature=0.8, fused=False)),
        # greedy decoding with a layer-skip draft and a long run of draft tokens (nine rows, head dimension 80)
        ("iteration-2.7b-greedy", _case("iteration", "neox-2.7b", K=8, ctx=519, temperature=0.0, fused=False)),
        # the benchmark's workload: eight sequences of ragged lengths around 2048 positions
        ("iteration-7b-b8", _case("iteration", batch=8, K=4, ctx=2100, fused=False)),
        # the pass the latency target is quoted on: one sequence, five rows
        ("verify-7b", _case("verify", K=4, ctx=2048)),
        # a long run of draft tokens on a long context: the far corner of the verification sweep
        ("verify-7b-k16-16k", _case("verify", K=16, ctx=16384)),
        # the largest model of the presets on a short context
        ("verify-12b", _case("verify", "neox-12b", K=5, ctx=163)),
        # autoregressive decoding of a batch, what speculation is compared with
        ("decode-7b-b8", _case("decode", batch=8, K=0, ctx=2100)),
        # the prompt pass of a batch of short requests through the 7B target and its stand-alone draft
        ("prefill-7b-b8", _case("prefill", batch=8, K=4, ctx=128)),
        # the prompt pass of a batch of long requests through target and layer-skip draft: the largest call
        ("prefill-2.7b-b8", _case("prefill", "neox-2.7b", batch=8, K=4, ctx=1023)),
    ]
    return [dict(c, name=n) for n, c in named]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tail", "generate", "iteration", "iteration", "verify", "verify", "decode", "prefill", "prefill"])
    t = rng.choice([0.0, 0.8, 1.0])
    if kind == "tail":
        return _tail(rng.randint(1, 12), rng.randint(0, 16), rng.choice([32000, 50304, _log_int(rng, 1000, 64000)]), t,
                     rng.choice([0, 0, 20, 50]), rng.choice([1.0, 1.0, 0.9, 0.95]), rng.random() < 0.5)
    if kind == "generate":
        return _case("generate", "tiny", batch=rng.randint(1, 4), K=rng.randint(1, 7), ctx=rng.randint(4, 64), temperature=t, iters=rng.randint(4, 16))
    model = rng.choice(["neox-1.4b", "neox-2.7b", "llama-7b", "llama-7b", "neox-12b"])
    if kind == "prefill":
        b = rng.choice([1, 1, 2, 4, 8])
        most = {"neox-1.4b": 2000 // b, "neox-2.7b": min(6000, 8184 // b), "llama-7b": 128, "neox-12b": 128}[model]
        return _case("prefill", model, batch=b, K=4, ctx=_log_int(rng, 12, most))
    b = rng.choice([1, 1, 1, 2, 3, 5, 8])
    most = min(16384, {"neox-1.4b": 24000, "neox-2.7b": 24000, "llama-7b": 17600, "neox-12b": 12000}[model] // b)
    ctx = _log_int(rng, 24, most)
    if kind == "decode":
        return _case("decode", model, batch=b, K=0, ctx=ctx, temperature=t)
    K = min(rng.choice([1, 2, 3, 4, 5, 6, 8, 11, 16]), 64 // b - 1)
    if kind == "verify":
        return _case("verify", model, batch=b, K=K, ctx=ctx, temperature=t)
    return _case("iteration", model, batch=b, K=K, ctx=ctx, temperature=t, fused=rng.random() < 0.25)


# ---- inputs ---------------------------------------------------------------------------------------
def _archs(case):
    p = synth.PRESETS[case["model"]]
    d = p["draft"]
    return p["target"], (p["target"].replace(n_layers=int(d.split(":")[1])) if isinstance(d, str) else d), isinstance(d, str)


def _weights(arch, gen, late_scale=1.0, late_from=0):
    """Random-init tensors in the library's order: matrices N(0, 1 / inputs), so that activations, keys, values and
    logits are of order one at every width; embeddings and vectors N(0, 0.02), gains 1 + N(0, 0.02)."""
    out = []
    for name in synth.tensor_names(arch):
        shape, base = synth.tensor_shape(arch, name), name.split(".")[-1]
        if shape is None:
            out.append(None)
            continue
        half = len(shape) == 2 and arch.dtype == synth.DT_BF16
        std = shape[-1] ** -0.5 if len(shape) == 2 and not base.endswith("_emb") else 0.02
        t = torch.empty(shape, dtype=torch.bfloat16 if half else torch.float32, device="cuda").normal_(0.0, std, generator=gen)
        if base.endswith("_g"):
            t += 1.0
        elif "." in name and base in ("w_o", "w_out", "b_o", "b_out") and int(name.split(".")[0][1:]) >= late_from and late_scale != 1.0:
            t *= late_scale
        out.append(t)
    return out


def _models(case, gen, want_draft=True):
    t_arch, d_arch, shared = _archs(case)
    # a layer-skip draft agrees with its target now and then only if the late layers change little
    late = dict(late_scale=0.2, late_from=d_arch.n_layers) if shared else {}
    target = B.Model(t_arch, _weights(t_arch, gen, **late))
    if not want_draft:
        return target, None
    return target, target.share_prefix(d_arch.n_layers) if shared else B.Model(d_arch, _weights(d_arch, gen))


def _spread(case):
    return max(1, case["ctx"] // 64) if case["batch"] > 1 else 0


def _lengths(case, seed):
    """Committed lengths of the sequences: ragged within a few positions where there are several."""
    b, n = case["batch"], case["ctx"]
    return (n - np.random.default_rng([seed, 5]).integers(0, _spread(case) + 1, size=b)).astype(np.int32)


def _fill(kv, lens, gen):
    kv.cache_view().normal_(0.0, KV_STD, generator=gen)
    B.kv_commit(kv, torch.from_numpy(lens).cuda())
    kv.lengths()


def _tokens(gen, vocab, *shape):
    return torch.randint(0, vocab, shape, generator=gen, device="cuda", dtype=torch.int32)


def _uniforms(gen, *shape, bits=24):
    """Uniforms on the grid k * 2^-24, k < 2^bits.  Those that draw a token from a model's row get 15 bits: where the
    row's running sum is still short, which token it is does not hang on the last bits of a sum over the vocabulary."""
    return torch.randint(0, 1 << bits, shape, generator=gen, device="cuda").float() * 2.0 ** -24


def _verify_uniforms(gen, b, K):
    return torch.cat([_uniforms(gen, b, K), _uniforms(gen, b, 1, bits=15)], dim=1)


def _restrict(p, top_k, top_p):
    """A draft distribution under the restriction that the target's gets (ties do not occur in these rows)."""
    s = p.sort(dim=-1, descending=True).values.double()
    if 0 < top_k < p.shape[-1]:
        s[..., top_k:] = 0.0
    if top_p < 1.0:
        s = torch.where(s.cumsum(-1) - s < top_p * s.sum(-1, keepdim=True), s, torch.zeros_like(s))
    low = torch.where(s > 0, s, torch.full_like(s, 2.0)).amin(-1, keepdim=True)
    p = torch.where(p.double() >= low, p, torch.zeros_like(p))
    return p / p.sum(-1, keepdim=True)


def _distributions(logits, temperature):
    if temperature > 0.0:
        return torch.softmax(logits / temperature, dim=-1)
    return torch.nn.functional.one_hot(logits.argmax(-1), logits.shape[-1]).float()


def _draw_from(q, gen):
    flat = q.reshape(-1, q.shape[-1])
    c = flat.double().cumsum(-1)
    u = torch.rand(flat.shape[0], 1, generator=gen, device="cuda", dtype=torch.float64) * c[:, -1:]
    return torch.searchsorted(c, u).clamp_(max=q.shape[-1] - 1).to(torch.int32).reshape(q.shape[:-1])


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    k, b, K = case["kind"], case["batch"], case["K"]
    s = dict(case=case)
    if k == "tail":
        V = case["vocab"]
        logits = torch.empty(b, K + 1, V, device="cuda").normal_(0.0, 2.0, generator=gen)
        s.update(logits=logits, u=_uniforms(gen, b, K + 1), rows=_tokens(gen, V, b, K + 1), q=None)
        if K:
            near = logits[:, :K] + torch.empty(b, K, V, device="cuda").normal_(0.0, 0.5, generator=gen)
            q = _distributions(near, case["temperature"])
            s["q"] = (_restrict(q, case["top_k"], case["top_p"]) if case["temperature"] > 0.0 else q).contiguous()
            s["rows"][:, 1:] = _draw_from(s["q"], gen)
        s.update(n_acc=torch.zeros(b, dtype=torch.int32, device="cuda"), nxt=torch.zeros(b, dtype=torch.int32, device="cuda"),
                 p=torch.empty(b, K + 1, V, device="cuda") if case["export"] else None,
                 scratch=torch.empty(B.verify_scratch_bytes(b, K), dtype=torch.uint8, device="cuda"))
        return s
    target, draft = _models(case, gen, want_draft=k in ("generate", "iteration", "prefill"))
    V = target.arch.vocab
    if k == "generate":
        it, P = case["iters"], case["ctx"]
        s["eng"] = engine.Engine(target, draft, b, min(target.arch.max_pos, P + (it + 2) * (K + 1)), K, case["temperature"], it * (K + 1))
        s["prompts"] = synth.gen_prompt(seed, b, P, V)
        u = np.stack([[synth.gen_uniforms(seed, q, i, 2 * K + 1) for i in range(it)] for q in range(b)])
        s["uniforms"] = lambda q, i: u[q, i]
        s["zero"] = torch.zeros(b, dtype=torch.int32, device="cuda")
    elif k == "prefill":
        s["eng"] = engine.Engine(target, draft, b, case["ctx"] + 1 + 8 * (K + 1), K, case["temperature"], 64)
        s["prompts"] = _tokens(gen, V, b, case["ctx"] + 1)
        s["zero"] = torch.zeros(b, dtype=torch.int32, device="cuda")
    elif k == "verify":
        lens = _lengths(case, seed)
        s["model"], s["kv"] = target, B.KV(target, b, case["ctx"] + 4 * (K + 1))
        _fill(s["kv"], lens, gen)
        s["ws"] = target.new_workspace(b, K + 1, s["kv"].max_len)
        s["q"] = _distributions(torch.empty(b, K, V, device="cuda").normal_(0.0, 1.3, generator=gen), case["temperature"]).contiguous()
        s["rows"] = _tokens(gen, V, b, K + 1)
        s["rows"][:, 1:] = _draw_from(s["q"], gen)
        s["u"] = _verify_uniforms(gen, b, K)
        s.update(n_acc=torch.zeros(b, dtype=torch.int32, device="cuda"), nxt=torch.zeros(b, dtype=torch.int32, device="cuda"))
    else:  # iteration, decode
        lens = _lengths(case, seed)
        eng = engine.Engine(target, draft, b, case["ctx"] + 4 * (K + 1), K, case["temperature"], 64)
        _fill(eng.tkv, lens, gen)
        pending = _tokens(gen, V, b)
        eng.rows[:, 0] = pending
        s.update(eng=eng, pending=pending)
        if k == "iteration":
            eng.fused_draft = case["fused"]
            # some sequences' drafts were all accepted the time before: those catch up two rows
            n_in = np.array([1 + (x == 1) for x in np.random.default_rng([seed, 6]).integers(0, 3, size=b)], np.int32)
            d_lens = np.maximum(lens - (n_in - 1), 0).astype(np.int32)
            _fill(eng.dkv, d_lens, gen)
            eng.draft_in.copy_(_tokens(gen, V, b, 2))
            eng.draft_in.scatter_(1, torch.from_numpy(n_in[:, None].astype(np.int64) - 1).cuda(), pending[:, None])
            eng.draft_n_in.copy_(torch.from_numpy(n_in))
            s.update(d_len=torch.from_numpy(d_lens).cuda(), u_draft=_uniforms(gen, b, K, bits=15), u=_verify_uniforms(gen, b, K))
        else:
            s.update(len=torch.from_numpy(lens).cuda(), u=_verify_uniforms(gen, b, 0))
    return s


# ---- one pass -------------------------------------------------------------------------------------
def _new_rows(kv, case):
    """The keys and values that a pass wrote (around them, where lengths differ, what was there)."""
    return kv.cache_view()[:, :, :, :, case["ctx"] - _spread(case):case["ctx"] + case["K"] + 1]


def run(state):
    case = state["case"]
    k, b, K = case["kind"], case["batch"], case["K"]
    if k == "tail":
        restricted = case["top_k"] > 0 or case["top_p"] < 1.0
        if restricted:
            B.set_sampling(case["top_k"], case["top_p"])
        B.verify_from_logits(state["logits"], K, state["rows"], state["q"], state["u"], case["temperature"], state["n_acc"], state["nxt"], 1,
                             state["p"], state["scratch"])
        if restricted:
            B.set_sampling(0, 1.0)
        return dict(n_accepted=state["n_acc"], next_token=state["nxt"], p=state["p"])
    if k == "verify":
        B.target_verify(state["model"], state["kv"], state["rows"], K, state["q"], state["u"], case["temperature"], state["n_acc"], state["nxt"], 1,
                        None, state["ws"])
        return dict(n_accepted=state["n_acc"], next_token=state["nxt"], logits=B.last_logits(state["model"], b, K + 1, state["ws"]),
                    kv=_new_rows(state["kv"], case))
    eng = state["eng"]
    if k in ("generate", "prefill"):
        # a new request on caches that are already there: cut them back, and tell the host's bound of the lengths
        B.kv_rollback(eng.tkv, state["zero"])
        B.kv_rollback(eng.dkv, state["zero"])
        eng.refresh_bounds()
        if k == "prefill":
            eng.prefill(state["prompts"])
            n = case["ctx"]
            return dict(kv=eng.tkv.cache_view()[:, :, :, :, :n], draft_kv=eng.dkv.cache_view()[:, :, :, :, :n])
        eng.generate(state["prompts"], 1 << 30, state["uniforms"], max_iters=case["iters"])
        n = case["ctx"] - 1 + case["iters"]  # committed for certain: the prompt and a token of each iteration
        return dict(tokens=eng.out_tokens, counts=eng.out_count, kv=eng.tkv.cache_view()[:, :, :, :, :n])
    if k == "decode":
        eng.ar_step(state["u"])
        B.kv_rollback(eng.tkv, state["len"])
        eng.rows[:, 0] = state["pending"]
    else:
        eng.spec_iteration(state["u_draft"], state["u"])
        B.kv_rollback(eng.dkv, state["d_len"])
    out = dict(next_token=eng.next_tok, logits=B.last_logits(eng.target, b, K + 1, eng.ws_t), kv=_new_rows(eng.tkv, case))
    if k == "iteration":
        out.update(n_accepted=eng.n_acc, drafts=eng.rows[:, 1:], q=eng.q)
    return out


# ---- what a pass cannot do without ------------------------------------------------------------------
def _pass(arch, b, rows, ctx, head=True):
    """A forward over b x rows rows after ctx positions: (bytes, flops) of matrices, cache and outputs, each once."""
    es = 2 if arch.dtype else 4
    d, F, L, R = arch.d_model, arch.d_ff, arch.n_layers, b * rows
    mats = L * (4 * d * d + arch.d_in * d + d * F)
    lm = arch.vocab * d if head else 0
    kv = 2 * L * d * es
    moved = (mats + lm) * es + R * d * es + b * ctx * kv + R * kv + (R * arch.vocab * 4 if head else 0)
    seen = b * (rows * ctx + rows * (rows + 1) // 2)
    return moved, 2 * R * (mats + lm) + 4 * d * L * seen


def work(case):
    k, b, K = case["kind"], case["batch"], case["K"]
    if k == "tail":
        V, rows = case["vocab"], b * (K + 1)
        return dict(bytes=4 * V * (rows + b * K + (rows if case["export"] else 0)), flops=10 * V * rows)
    t, d, _ = _archs(case)
    if k == "prefill":
        both = [_pass(a, b, case["ctx"], 0, head=False) for a in (t, d)]
    elif k == "generate":
        n = case["ctx"] + case["iters"] // 2
        each = [_pass(t, b, K + 1, n)] + [_pass(d, b, 1, n)] * K
        both = each * case["iters"] + [_pass(a, b, case["ctx"] - 1, 0, head=False) for a in (t, d)]
    else:
        both = [_pass(t, b, K + 1, case["ctx"])]
        if k == "iteration":
            both += [_pass(d, b, 1, case["ctx"])] * K
    q = b * K * t.vocab * 4 if k in ("verify", "iteration") else 0
    return dict(bytes=sum(m for m, _ in both) + q, flops=sum(f for _, f in both))


def tolerance(case):
    """fp32 and fp64 arithmetic on exact inputs, and bf16 only where the cache stores keys and values: passes differ by
    the order of fp32 sums, which now and then moves a stored key or value by one bf16 step.  Seen between two runs of
    the same passes: logits 8e-5, new keys and values 4e-4; 2e-3 where a prompt is fed in several passes, each of which
    attends to keys and values that the ones before it rounded."""
    if case["kind"] == "tail":
        return {"rel": 1e-5}
    if case["kind"] == "generate":
        return {"rel": 2e-5}
    return {"rel": 8e-3 if case["kind"] == "prefill" else 2e-3}
