"""Many-row prompt pass (tiled tcgen05 GEMMs + causal attention over the cache) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import decoder as od
from paper_2311_04951_b200 import binding as B, synth
from tests import gpu_util as gu
from tests.test_gpu_forward import ARCHS, gpu_logits

pytestmark = pytest.mark.gpu

BF16 = [n for n, a in ARCHS.items() if a.dtype == synth.DT_BF16]


@pytest.fixture(params=[2, 3], ids=["tc-attention-where-it-applies", "mma-attention"])
def many_row_mode(request):
    B.set_prefill_mode(request.param)
    yield
    B.set_prefill_mode(0)


def _cache_close(arch, got, ref):
    tol = gu.LOGIT_RTOL * np.abs(ref).max(axis=-1, keepdims=True) + gu.LOGIT_ATOL
    bad = np.argwhere(np.abs(got - ref) > tol)
    assert bad.shape[0] == 0, (bad[:8].tolist(), [(float(got[tuple(i)]), float(ref[tuple(i)])) for i in bad[:8]])


def _check_against_oracle(arch, omodel, model, kv, prompts, lens, S):
    Bn = prompts.shape[0]
    assert kv.status() == 0 and kv.lengths().tolist() == lens.tolist()
    rows = synth.gen_prompt(15, Bn, 3, arch.vocab)
    got = gpu_logits(model, kv, model.new_workspace(Bn, 3, S), rows, 2)
    cache = kv.cache_view().float().cpu().numpy()
    for b in range(Bn):
        oc = omodel.new_cache(S)
        oc.feed(prompts[b, :lens[b]], want_logits=False)
        gu.assert_logits_close(got[b], oc.feed(rows[b], advance=False))
        n = int(lens[b])
        _cache_close(arch, cache[:, b, :, :, :n], oc.kv[:, :, :, :n])


@pytest.mark.parametrize("name", BF16)
def test_many_row_prompt_pass_matches_oracle(name, many_row_mode):
    """One pass over ragged prompts: several 128-row GEMM tiles with a ragged last one, several 64-row attention
    tiles per sequence, a sequence that ends inside a tile, one that feeds a single token."""
    arch = ARCHS[name]
    ws_np = gu.scaled_weights(synth, arch, 3, 6.0)
    omodel = od.Model(arch, ws_np)
    model = B.Model(arch, B.upload_weights(arch, ws_np))
    P = 150
    if arch.pos == 0:
        P = arch.max_pos - 8
    S = P + 8
    Bn = 3
    lens = np.array([P, P - 67, 1], np.int32)
    prompts = synth.gen_prompt(31, Bn, P, arch.vocab)
    nbytes = model.prefill_workspace_bytes(Bn, P)
    assert nbytes > 0
    kv = B.KV(model, Bn, S)
    n0 = B.launch_count()
    B.kv_prefill(model, kv, torch.from_numpy(prompts).cuda(), torch.from_numpy(lens).cuda(), B.device_buffer(nbytes))
    # one pass: set-up, embedding, and per layer 4 GEMMs + norm(s) + append + attention + activation
    per_layer = 8 if arch.parallel_residual else 9
    assert B.launch_count() - n0 == 1 + 2 + per_layer * arch.n_layers + 1
    _check_against_oracle(arch, omodel, model, kv, prompts, lens, S)


@pytest.mark.parametrize("name", ["llama_bf16", "neox_bf16"])
def test_many_row_prompt_pass_in_several_passes_and_on_a_filled_cache(name, many_row_mode):
    """A workspace that holds only part of the prompt: equal passes, the later ones attending to what the earlier
    ones stored; then a second prompt call that continues the same sequences."""
    arch = ARCHS[name]
    ws_np = gu.scaled_weights(synth, arch, 3, 6.0)
    omodel = od.Model(arch, ws_np)
    model = B.Model(arch, B.upload_weights(arch, ws_np))
    Bn, P1, P2 = 2, 200, 45
    S = P1 + P2 + 8
    prompts = synth.gen_prompt(32, Bn, P1 + P2, arch.vocab)
    lens1 = np.array([P1, P1 - 90], np.int32)
    ws = B.device_buffer(model.prefill_workspace_bytes(Bn, 80))      # 200 tokens -> the largest power-of-two share that fits: four passes of 64 rows
    kv = B.KV(model, Bn, S)
    first = np.ascontiguousarray(prompts[:, :P1])
    B.kv_prefill(model, kv, torch.from_numpy(first).cuda(), torch.from_numpy(lens1).cuda(), ws)
    assert kv.status() == 0 and kv.lengths().tolist() == lens1.tolist()
    lens2 = np.array([P2, P2 - 4], np.int32)
    second = np.stack([prompts[b, lens1[b]:lens1[b] + P2] for b in range(Bn)])
    B.kv_prefill(model, kv, torch.from_numpy(np.ascontiguousarray(second)).cuda(), torch.from_numpy(lens2).cuda(), ws)
    total = lens1 + lens2
    _check_against_oracle(arch, omodel, model, kv, prompts, total, S)


def test_many_row_form_is_taken_from_256_rows_and_equals_the_chunked_form():
    """Default mode: 2 x 130 rows take the many-row form (fewer launches than chunks), 2 x 100 do not; both forms
    leave the same cache up to rounding."""
    arch = ARCHS["llama_bf16"]
    ws_np = gu.scaled_weights(synth, arch, 3, 6.0)
    model = B.Model(arch, B.upload_weights(arch, ws_np))
    Bn, S = 2, 160
    C = min(B.MAX_ROWS_PER_SEQ, B.MAX_ROWS // Bn)
    caches = {}
    for P in (130, 100):
        prompts = torch.from_numpy(synth.gen_prompt(33, Bn, P, arch.vocab)).cuda()
        lens = torch.full((Bn,), P, dtype=torch.int32, device="cuda")
        big = B.device_buffer(max(model.prefill_workspace_bytes(Bn, P), model.workspace_bytes(Bn, C, S)))
        for mode in (0, 1):
            B.set_prefill_mode(mode)
            try:
                kv = B.KV(model, Bn, S)
                n0 = B.launch_count()
                B.kv_prefill(model, kv, prompts, lens, big)
                caches[(P, mode)] = (kv.cache_view().float().cpu().numpy()[..., :P, :], B.launch_count() - n0)
                assert kv.status() == 0 and kv.lengths().tolist() == [P] * Bn
            finally:
                B.set_prefill_mode(0)
    chunks = lambda P: -(-P // C)
    assert caches[(130, 1)][1] == 3 * chunks(130) and caches[(100, 0)][1] == 3 * chunks(100)
    assert caches[(130, 0)][1] == 1 + 2 + 9 * arch.n_layers + 1
    _cache_close(arch, caches[(130, 0)][0], caches[(130, 1)][0])


def test_prompt_longer_than_the_cache_is_refused(many_row_mode):
    arch = ARCHS["neox_bf16"]
    model = B.Model(arch, B.upload_weights(arch, gu.scaled_weights(synth, arch, 3, 6.0)))
    kv = B.KV(model, 2, 64)
    prompts = torch.from_numpy(synth.gen_prompt(34, 2, 80, arch.vocab)).cuda()
    lens = torch.full((2,), 80, dtype=torch.int32, device="cuda")
    with pytest.raises(B.SsdError):
        B.kv_prefill(model, kv, prompts, lens, B.device_buffer(model.prefill_workspace_bytes(2, 80)))
    assert kv.lengths().tolist() == [0, 0]


def test_many_row_prompt_pass_is_run_to_run_identical():
    """Nothing in the many-row pass depends on an order of arrival: the projections own their output tiles and a query
    row's softmax and output belong to two threads that exchange one maximum per chunk.  Repeated passes over the same prompts must agree bit for bit (the
    tensor-core attention runs its warps up to a chunk apart; with several chunks per row tile and many CTAs a
    hand-over that miscounts shows up as other bits within a few passes)."""
    arch = synth.llama_like(2, 4096, 32, 512, 512)
    model = B.Model(arch, B.upload_weights(arch, synth.gen_weights(arch, 31)))
    Bn, P = 8, 1000
    dev = "cuda"
    kv = B.KV(model, Bn, P)
    prompts = torch.from_numpy(synth.gen_prompt(32, Bn, P, arch.vocab)).to(dev)
    n = torch.full((Bn,), P, dtype=torch.int32, device=dev)
    zero = torch.zeros(Bn, dtype=torch.int32, device=dev)
    ws = B.device_buffer(model.prefill_workspace_bytes(Bn, P))
    ref = None
    for _ in range(40):
        B.kv_rollback(kv, zero)
        kv.lengths()
        B.kv_prefill(model, kv, prompts, n, ws)
        got = kv.cache_view()
        if ref is None:
            ref = got.clone()
        else:
            assert torch.equal(got, ref)
    assert kv.status() == 0


@pytest.mark.parametrize("name", ["llama_bf16", "neox_bf16_h80"])
def test_layer_skip_draft_takes_the_many_row_form(name, many_row_mode):
    """A draft that shares its target's first layers has the target's many-row pass: its cache equals those layers of
    the target's cache bit for bit (the same kernels on the same tensors)."""
    arch = ARCHS[name]
    model = B.Model(arch, B.upload_weights(arch, gu.scaled_weights(synth, arch, 3, 6.0)))
    draft = model.share_prefix(arch.n_layers - 1)
    Bn, P = 2, 140
    assert draft.prefill_workspace_bytes(Bn, P) == model.prefill_workspace_bytes(Bn, P) > 0
    prompts = torch.from_numpy(synth.gen_prompt(33, Bn, P, arch.vocab)).to("cuda")
    n = torch.tensor([P, P - 50], dtype=torch.int32, device="cuda")
    caches = []
    for m in (model, draft):
        kv = B.KV(m, Bn, P + 4)
        B.kv_prefill(m, kv, prompts, n, B.device_buffer(m.prefill_workspace_bytes(Bn, P)))
        assert kv.status() == 0 and kv.lengths().tolist() == n.tolist()
        caches.append(kv.cache_view().clone())
    assert torch.equal(caches[0][:arch.n_layers - 1], caches[1])


def _odd(arch, **kw):
    return arch.replace(dtype=synth.DT_BF16, **kw)


# head dims of one and two 64-column panels with and without a remainder; rotary widths whose halves are not whole 16-byte
# pieces; MLP widths that end inside a 128- or 256-column weight tile, and a SwiGLU tile that reaches past both halves
ODD = {
    "head16-rot12-gelu200": _odd(synth.neox_like(2, 144, 9, 200, 300), rotary_dim=12),
    "head48-swiglu136": _odd(synth.llama_like(2, 144, 3, 136, 300)),
    "head80-rot20-gelu264": _odd(synth.neox_like(2, 160, 2, 264, 300), rotary_dim=20),
    "head96-rot24-gelu128": _odd(synth.neox_like(2, 192, 2, 128, 300), rotary_dim=24),
    "head112-swiglu392": _odd(synth.llama_like(2, 224, 2, 392, 300)),
}


@pytest.mark.parametrize("name", list(ODD))
@pytest.mark.parametrize("P", [127, 129, 257])
def test_many_row_prompt_pass_at_odd_head_and_mlp_widths(name, P, many_row_mode):
    """Around the 128-position chunk and the 128-row tile, over a cache that holds NaNs wherever nothing was stored (a position
    that no row sees must not reach the output, not even times zero)."""
    arch = ODD[name]
    ws_np = gu.scaled_weights(synth, arch, 3, 6.0)
    model = B.Model(arch, B.upload_weights(arch, ws_np))
    S, lens = P + 8, np.array([P, P - 63], np.int32)
    prompts = synth.gen_prompt(35, 2, P, arch.vocab)
    kv = B.KV(model, 2, S)
    kv.cache_view().fill_(float("nan"))
    B.kv_prefill(model, kv, torch.from_numpy(prompts).cuda(), torch.from_numpy(lens).cuda(),
                 B.device_buffer(model.prefill_workspace_bytes(2, P)))
    _check_against_oracle(arch, od.Model(arch, ws_np), model, kv, prompts, lens, S)


@pytest.mark.parametrize("name,P", [("llama_bf16", 140), ("neox_bf16_h80", 140), ("neox_bf16", 21), ("gpt2_f32", 17), ("gpt2_bf16", 1)])
def test_prompt_pass_of_a_target_and_its_layer_skip_draft(name, P):
    """The draft's cache after the common pass is the one of a pass of its own: taken over from the target's (bit for bit) while
    both are empty, computed when they are not (the few-row projections add their partial sums in no fixed order, so two
    passes agree to rounding)."""
    arch = ARCHS[name]
    target = B.Model(arch, B.upload_weights(arch, gu.scaled_weights(synth, arch, 3, 6.0)))
    draft = target.share_prefix(arch.n_layers - 1)
    Bn, S, C = 3, 2 * P + 4, min(B.MAX_ROWS_PER_SEQ, B.MAX_ROWS // 3)
    sizes = {m: max(m.prefill_workspace_bytes(Bn, P), m.workspace_bytes(Bn, C, S)) for m in (target, draft)}
    ws = {m: B.device_buffer(n) for m, n in sizes.items()}
    pair = {target: B.KV(target, Bn, S), draft: B.KV(draft, Bn, S + 12)}
    alone = {target: B.KV(target, Bn, S), draft: B.KV(draft, Bn, S + 12)}
    for seed in (36, 37):   # empty caches, then filled ones
        prompts = torch.from_numpy(synth.gen_prompt(seed, Bn, P, arch.vocab)).cuda()
        n = torch.tensor([P, max(P - 9, 1), 1], dtype=torch.int32, device="cuda")
        n0 = B.launch_count()
        B.kv_prefill_pair(target, pair[target], draft, pair[draft], prompts, n, ws[target], ws[draft])
        n1 = B.launch_count()
        for m in (target, draft):
            B.kv_prefill(m, alone[m], prompts, n, ws[m])
        if P > 1:
            assert (n1 - n0 < B.launch_count() - n1) == (seed == 36)
        for m in (target, draft):
            assert pair[m].status() == 0 and pair[m].lengths().tolist() == alone[m].lengths().tolist()
            got, ref = pair[m].cache_view(), alone[m].cache_view()
            for b, v in enumerate(alone[m].lengths().tolist()):
                _cache_close(arch, got[:, b, :, :, :v].float().cpu().numpy(), ref[:, b, :, :, :v].float().cpu().numpy())
                if seed == 36:
                    assert torch.equal(pair[draft].cache_view()[:, b, :, :, :v], pair[target].cache_view()[:-1, b, :, :, :v])


def test_prompt_pass_of_a_target_and_a_draft_of_its_own():
    arch = ARCHS["llama_bf16"]
    models = [B.Model(arch, B.upload_weights(arch, gu.scaled_weights(synth, arch, s, 6.0))) for s in (3, 4)]
    prompts = torch.from_numpy(synth.gen_prompt(38, 2, 20, arch.vocab)).cuda()
    n = torch.tensor([20, 7], dtype=torch.int32, device="cuda")
    ws = B.device_buffer(models[0].workspace_bytes(2, 8, 24))
    pair, alone = [[B.KV(m, 2, 24) for m in models] for _ in range(2)]
    B.kv_prefill_pair(models[0], pair[0], models[1], pair[1], prompts, n, ws, ws)
    for m, kv, got in zip(models, alone, pair):
        B.kv_prefill(m, kv, prompts, n, ws)
        assert got.lengths().tolist() == kv.lengths().tolist() == [20, 7]
        _cache_close(arch, *(k.cache_view()[:, 0, :, :, :20].float().cpu().numpy() for k in (got, kv)))


def _layer_skip_pair():
    arch = synth.llama_like(3, 256, 4, 512, 512)
    target = B.Model(arch, B.upload_weights(arch, gu.scaled_weights(synth, arch, 51, 6.0)))
    return arch, target, target.share_prefix(1)


def _prompt(seed, n, vocab):
    return torch.from_numpy(synth.gen_prompt(seed, 2, n, vocab)).cuda(), torch.full((2,), n, dtype=torch.int32, device="cuda")


def _rows_close(kv, ref, n):
    got, want = (k.cache_view()[..., :n, :].float() for k in (kv, ref))
    assert ((got - want).abs() <= gu.LOGIT_ATOL + gu.LOGIT_RTOL * want.abs().amax(-1, keepdim=True)).all()


def test_prompt_pair_after_a_slab_copy_does_not_take_the_cache_for_an_empty_one():
    """Lengths that a copy of another cache's slab brought (no kernel reported them) and kv_lengths has read: the draft's
    prompt is computed, not taken over from a target cache that holds more than it."""
    arch, target, draft = _layer_skip_pair()
    S = 96
    ws_t, ws_d = target.new_workspace(2, 8, S), draft.new_workspace(2, 8, S)
    first, second = _prompt(1, 20, arch.vocab), _prompt(2, 12, arch.vocab)
    full, tkv, dkv, alone = B.KV(target, 2, S), B.KV(target, 2, S), B.KV(draft, 2, S), B.KV(draft, 2, S)
    B.kv_prefill(target, full, *first, ws_t)
    zero = torch.zeros(2, dtype=torch.int32, device="cuda")
    B.kv_rollback(tkv, zero)
    B.kv_rollback(dkv, zero)
    torch.cuda.synchronize()
    tkv.buf.copy_(full.buf)
    assert tkv.lengths().tolist() == [20, 20] and dkv.lengths().tolist() == [0, 0]
    B.kv_prefill_pair(target, tkv, draft, dkv, *second, ws_t, ws_d)
    assert tkv.lengths().tolist() == [32, 32] and dkv.lengths().tolist() == [12, 12]
    assert tkv.status() == 0 and dkv.status() == 0
    B.kv_prefill(draft, alone, *second, ws_d)
    _rows_close(dkv, alone, 12)


def test_prompt_pair_over_a_slab_written_behind_the_library_is_refused():
    """The same copy without kv_lengths: the host's bound still says empty; the device sees that it is not."""
    arch, target, draft = _layer_skip_pair()
    S = 96
    ws_t, ws_d = target.new_workspace(2, 8, S), draft.new_workspace(2, 8, S)
    full, tkv, dkv = B.KV(target, 2, S), B.KV(target, 2, S), B.KV(draft, 2, S)
    B.kv_prefill(target, full, *_prompt(1, 20, arch.vocab), ws_t)
    tkv.buf.copy_(full.buf)
    B.kv_prefill_pair(target, tkv, draft, dkv, *_prompt(2, 12, arch.vocab), ws_t, ws_d)
    assert tkv.lengths().tolist() == [32, 32] and tkv.status() == 0
    assert dkv.status() == -1 and dkv.lengths().tolist() == [0, 0]


def test_recorded_prompt_pair_extends_both_caches_at_every_replay():
    """A pair call recorded on empty caches and replayed twice: the second replay's prompt follows the first one's in both."""
    arch, target, draft = _layer_skip_pair()
    S, n = 96, 12
    ws_t, ws_d = target.new_workspace(2, 8, S), draft.new_workspace(2, 8, S)
    prompt = _prompt(3, n, arch.vocab)
    tkv, dkv, alone = B.KV(target, 2, S), B.KV(draft, 2, S), B.KV(draft, 2, S)
    for _ in range(2):
        B.kv_prefill(draft, alone, *prompt, ws_d)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.kv_prefill_pair(target, tkv, draft, dkv, *prompt, ws_t, ws_d)
    graph.replay()
    graph.replay()
    assert tkv.lengths().tolist() == dkv.lengths().tolist() == [2 * n, 2 * n]
    assert tkv.status() == 0 and dkv.status() == 0
    _rows_close(dkv, alone, 2 * n)
