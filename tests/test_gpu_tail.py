"""GPU parity of the vocabulary-wide tail (softmax, accept scan, residual resample, bonus draw)
on supplied logits, draft rows and uniforms, through the C ABI (verify_from_logits)."""
import numpy as np
import pytest
import torch

from oracle import sampling as osamp
from paper_2311_04951_b200 import binding as B, synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def run_tail(logits, rows, q, u, T, want_p=True):
    Bn, M, V = logits.shape
    K = M - 1
    dev = "cuda"
    lg = torch.from_numpy(logits).to(dev)
    n_acc = torch.full((Bn,), -7, dtype=torch.int32, device=dev)
    nxt = torch.full((Bn,), -7, dtype=torch.int32, device=dev)
    p = torch.zeros(Bn, M, V, dtype=torch.float32, device=dev) if want_p else None
    scratch = torch.empty(B.verify_scratch_bytes(Bn, K), dtype=torch.uint8, device=dev)
    B.verify_from_logits(lg, K, torch.from_numpy(rows).to(dev), None if K == 0 else torch.from_numpy(q).to(dev),
                         torch.from_numpy(u).to(dev), T, n_acc, nxt, 1, p, scratch)
    torch.cuda.synchronize()
    return n_acc.cpu().numpy(), nxt.cpu().numpy(), (p.cpu().numpy() if want_p else None)


def make_case(seed, Bn, K, V, T, corr):
    """Logits ~ N(0, 1.5); draft rows either Dirichlet(0.1) (far from p) or a perturbed copy of p
    (acceptance non-trivial); draft tokens drawn from q."""
    logits = synth.gen_logits(seed, Bn * (K + 1), V, 1.5).reshape(Bn, K + 1, V)
    if corr:
        noise = synth.gen_logits(seed + 100, Bn * K, V, 0.7).reshape(Bn, K, V)
        ql = logits[:, :K] + noise
        q = np.stack([[osamp.softmax_t(ql[b, i], T if T > 0 else 1.0) for i in range(K)] for b in range(Bn)]) \
            if K else np.zeros((Bn, 0, V), np.float32)
    else:
        q = synth.gen_dirichlet_rows(seed + 1, Bn * K, V).reshape(Bn, K, V) if K else np.zeros((Bn, 0, V), np.float32)
    toks = synth.draw_tokens_from_rows(seed + 2, q.reshape(Bn * K, V)).reshape(Bn, K) if K else np.zeros((Bn, 0), np.int32)
    if T == 0 and K:  # greedy drafts propose one-hot rows
        hot = np.zeros_like(q)
        for b in range(Bn):
            for i in range(K):
                # half of the rows agree with the target argmax so that acceptance varies
                t = int(np.argmax(logits[b, i])) if (b + i) % 2 == 0 else int(toks[b, i])
                toks[b, i] = t
                hot[b, i, t] = 1
        q = hot
    rows = np.concatenate([np.zeros((Bn, 1), np.int32), toks.astype(np.int32)], axis=1)
    u = np.stack([synth.gen_uniforms(seed + 3, b, 0, K + 1) for b in range(Bn)])
    return logits, rows, q.astype(np.float32), u


@pytest.mark.parametrize("V", [1000, 32000, 50304])
@pytest.mark.parametrize("K,Bn", [(0, 1), (1, 2), (4, 1), (8, 3), (16, 1)])
@pytest.mark.parametrize("T,corr", [(1.0, False), (0.8, True), (0.0, True)])
def test_tail_matches_oracle(V, K, Bn, T, corr):
    logits, rows, q, u = make_case(1000 + V % 97 + K, Bn, K, V, T, corr)
    n_acc, nxt, p = run_tail(logits, rows, q, u, T)
    exact = 0
    for b in range(Bn):
        p_ref = np.stack([osamp.softmax_t(logits[b, i], T) for i in range(K + 1)])
        assert np.abs(p[b] - p_ref).max() <= gu.P_ATOL                      # layer A
        assert abs(p[b].sum(axis=1) - 1).max() < 1e-4
        exact += gu.check_decisions_on_own_rows(p[b], q[b], rows[b, 1:], u[b, :K], u[b, K], int(n_acc[b]), int(nxt[b]))
        # and against the oracle end to end, unless a decision is within tolerance of its threshold
        a_ref, y_ref = osamp.accept_resample(p_ref, q[b], rows[b, 1:], u[b, :K], u[b, K])
        if (a_ref, y_ref) != (int(n_acc[b]), int(nxt[b])):
            i = min(a_ref, int(n_acc[b]))
            if a_ref != int(n_acc[b]):
                x = rows[b, 1 + i]
                assert abs(float(p_ref[i, x]) - float(np.float32(u[b, i]) * q[b, i, x])) <= gu.P_ATOL + 4e-2 * p_ref[i, x]
    assert exact >= Bn - 1


def test_acceptance_varies_and_all_branches_are_hit():
    """Over many seeded cases every accepted count 0..K occurs (rejection at each row and the bonus
    branch), so the parity above covers all paths."""
    K, V, seen = 3, 2000, set()
    for seed in range(12):
        logits, rows, q, u = make_case(50 + seed, 4, K, V, 1.0, True)
        n_acc, nxt, _ = run_tail(logits, rows, q, u, 1.0, want_p=False)
        for b in range(4):
            p_ref = np.stack([osamp.softmax_t(logits[b, i], 1.0) for i in range(K + 1)])
            a_ref, y_ref = osamp.accept_resample(p_ref, q[b], rows[b, 1:], u[b, :K], u[b, K])
            seen.add(a_ref)
            if (a_ref, y_ref) != (int(n_acc[b]), int(nxt[b])):
                assert a_ref == int(n_acc[b])   # a token may differ only at a CDF step of near-equal sums
    assert seen == {0, 1, 2, 3}


def test_degenerate_rows():
    V, K = 512, 2
    logits = np.zeros((1, K + 1, V), np.float32)
    logits[0, :, 7] = 50.0                               # p is (numerically) one-hot at 7
    q = np.zeros((1, K, V), np.float32)
    q[0, 0, 7] = 1.0                                     # q == p -> accept
    q[0, 1, 9] = 1.0                                     # draft certain of a token the target excludes
    rows = np.array([[0, 7, 9]], np.int32)
    u = np.array([[0.5, 0.5, 0.3]], np.float32)
    n_acc, nxt, p = run_tail(logits, rows, q, u, 1.0)
    assert n_acc[0] == 1 and nxt[0] == 7                 # rejected at row 2, residual = p -> 7
    # q(x~) = 0 < p(x~): accepted even for u close to 1
    q2 = q.copy(); q2[0, 0] = 0; q2[0, 0, 3] = 1.0
    n_acc, nxt, _ = run_tail(logits, np.array([[0, 7, 7]], np.int32), q2, np.array([[0.999, 0.999, 0.1]], np.float32), 1.0)
    assert n_acc[0] == 2 and nxt[0] == 7
    # ties in greedy mode: lowest index wins
    lg = np.zeros((1, 1, V), np.float32); lg[0, 0, [5, 400]] = 3.0
    n_acc, nxt, p = run_tail(lg, np.zeros((1, 1), np.int32), np.zeros((1, 0, V), np.float32), np.array([[0.7]], np.float32), 0.0)
    assert nxt[0] == 5 and p[0, 0, 5] == 1.0 and p[0, 0].sum() == 1.0


def test_argument_errors_are_reported_on_the_host():
    dev = "cuda"
    lg = torch.zeros(1, 2, 128, device=dev)
    z = torch.zeros(4, dtype=torch.int32, device=dev)
    f = torch.zeros(256, device=dev)
    sc = torch.empty(B.verify_scratch_bytes(1, 1), dtype=torch.uint8, device=dev)
    with pytest.raises(B.SsdError) as e:
        B.verify_from_logits(lg, 1, z, None, f, 1.0, z, z, 1, None, sc)     # K > 0 without q
    assert e.value.code == -1
    with pytest.raises(B.SsdError) as e:
        B.verify_from_logits(lg, 1, z, f, f, 1.0, z, z, 1, None, sc[:8])    # scratch too small
    assert e.value.code == -3
    with pytest.raises(B.SsdError):
        B.verify_from_logits(lg, 1, z, f, f, -1.0, z, z, 1, None, sc)       # negative temperature


@pytest.mark.parametrize("V", [1000, 32000, 50304])
@pytest.mark.parametrize("top_k,top_p", [(50, 1.0), (0, 0.9), (40, 0.7), (1, 1.0), (0, 0.2), (100000, 0.999)])
def test_restricted_tail_matches_oracle(V, top_k, top_p):
    """top-k / top-p restriction inside the tail: the p rows the decisions use equal the oracle's restricted
    rows (same kept set unless a token sits at the nucleus boundary within rounding of the running sum), and
    the decisions follow the oracle's rule on those rows.  q is restricted the same way on the host side of
    the test, as a draft that runs under the same setting would deliver it."""
    T, K, Bn = 0.9, 4, 2
    logits, rows, q, u = make_case(2000 + V % 89 + top_k % 7, Bn, K, V, T, True)
    std = 3.0 if V > 1000 else 1.5          # peakier rows: a nucleus of tens, not thousands, of tokens
    logits = (logits * np.float32(std / 1.5)).astype(np.float32)
    q = np.stack([[osamp.filter_top_k_top_p(q[b, i], top_k, top_p) for i in range(K)] for b in range(Bn)])
    toks = synth.draw_tokens_from_rows(77, q.reshape(Bn * K, V)).reshape(Bn, K)
    rows[:, 1:] = toks
    B.set_sampling(top_k, top_p)
    try:
        n_acc, nxt, p = run_tail(logits, rows, q, u, T)
    finally:
        B.set_sampling(0, 1.0)
    for b in range(Bn):
        for i in range(K + 1):
            raw = osamp.softmax_t(logits[b, i], T)
            ref = osamp.filter_top_k_top_p(raw, top_k, top_p)
            got = p[b, i]
            same = (got > 0) == (ref > 0)
            if not same.all():
                # only tokens whose probability equals the threshold up to rounding of the running sums may differ
                thr = min(raw[got > 0].min(), raw[ref > 0].min())
                odd = raw[~same]
                assert (np.abs(odd - thr) <= 1e-6 * max(thr, 1e-30) + 1e-12).all() or \
                    abs(raw[got > 0].astype(np.float64).sum() - raw[ref > 0].astype(np.float64).sum()) <= 2e-6
            else:
                assert np.abs(got - ref).max() <= gu.P_ATOL
                assert abs(float(got.astype(np.float64).sum()) - 1.0) < 1e-5
        gu.check_decisions_on_own_rows(p[b], q[b], rows[b, 1:], u[b, :K], u[b, K], int(n_acc[b]), int(nxt[b]))
        assert p[b, int(n_acc[b])][int(nxt[b])] > 0       # the emitted token lies inside the restricted target
    if top_k == 1:
        assert ((p > 0).sum(axis=2) == 1).all()


def test_draft_and_verify_under_a_restriction_follow_the_oracle_loop():
    """Whole speculative iterations with top-k / top-p set (fp32 model, so the two sides agree to rounding):
    the draft's exported q rows, its tokens, the accepted counts and the target's tokens equal the oracle's
    loop run with the same restriction."""
    from oracle import decoder as od, spec as ospec
    from paper_2311_04951_b200 import engine
    arch = synth.gpt2_like(3, 128, 4, 256, 400, 160)
    ws = gu.scaled_weights(synth, arch, 21, 7.0)
    d_arch, d_ws = synth.prefix_draft(arch, ws, 1)
    tgt = B.Model(arch, B.upload_weights(arch, ws))
    K, T, n_new, top_k, top_p = 3, 0.9, 40, 12, 0.85
    prompt = synth.gen_prompt(22, 1, 12, arch.vocab)
    ref = ospec.speculative_generate(od.Model(arch, ws), od.Model(d_arch, d_ws), prompt[0], n_new, K, T,
                                     lambda it: synth.gen_uniforms(23, 0, it, 2 * K + 1), 160, keep_trace=True,
                                     top_k=top_k, top_p=top_p)
    B.set_sampling(top_k, top_p)
    try:
        eng = engine.Engine(tgt, tgt.share_prefix(1), 1, 160, K, T, 128)
        res = gu.lockstep(eng, synth, prompt[0], ref["iterations"], K, 23, ref["trace"])
    finally:
        B.set_sampling(0, 1.0)
    assert eng.tkv.status() == 0 and eng.dkv.status() == 0
    assert res["identical"] == res["iterations"] == ref["iterations"] and res["excused"] == 0
    assert max(int((t["q"][0] > 0).sum()) for t in ref["trace"]) <= top_k     # the restriction was active
    n_out = int(eng.out_count.cpu()[0])
    assert eng.out_tokens.cpu().numpy()[0, :n_out].tolist() == ref["all_tokens"][len(prompt[0]):]


@pytest.mark.parametrize("top_k,top_p", [(0, 1.0), (37, 0.9), (0, 0.9)])
@pytest.mark.parametrize("V", [33, 255, 8193, 65535, 65537, 131100])
def test_tail_at_the_edges_of_the_row_pieces(V, top_k, top_p):
    """A cluster's 256 warps own pieces of whole 32-entry lane rows and hold 256 entries at a time: rows shorter than one
    piece per warp, one entry past a whole number of lane rows, and (from 65537 entries) pieces read in two steps; under a
    restriction, rows whose probabilities fit the two CTAs' shared memory and (from about 88000 entries) do not; with equal
    values at the threshold, a flat row (one bin of the search), a row of two values and one with a far tail."""
    T, K, Bn = 1.0, 3, 2
    logits, rows, q, u = make_case(3000 + V, Bn, K, V, T, True)
    logits[0, 1] = 0.25
    logits[1, 0] = np.where(np.arange(V) % 3 == 0, 1.0, -30.0)
    logits[1, 2] *= 20.0
    q = np.stack([[osamp.filter_top_k_top_p(q[b, i], top_k, top_p) for i in range(K)] for b in range(Bn)])
    rows[:, 1:] = synth.draw_tokens_from_rows(78, q.reshape(Bn * K, V)).reshape(Bn, K)
    B.set_sampling(top_k, top_p)
    try:
        n_acc, nxt, p = run_tail(logits, rows, q, u, T)
    finally:
        B.set_sampling(0, 1.0)
    for b in range(Bn):
        for i in range(K + 1):
            raw = osamp.softmax_t(logits[b, i], T)
            ref = osamp.filter_top_k_top_p(raw, top_k, top_p)
            odd = raw[(p[b, i] > 0) != (ref > 0)]
            if odd.size:      # only values at the nucleus boundary, within the rounding of the running sums
                assert np.ptp(odd) <= 1e-6 * odd.max()
            else:
                assert np.abs(p[b, i] - ref).max() <= gu.P_ATOL
            assert abs(float(p[b, i].astype(np.float64).sum()) - 1.0) < 1e-5
        gu.check_decisions_on_own_rows(p[b], q[b], rows[b, 1:], u[b, :K], u[b, K], int(n_acc[b]), int(nxt[b]))


def check_restricted_row(got, logits, T, top_k, top_p, exact):
    """A restricted row of the kernel against the oracle's: equal logits have bit-equal probabilities, so a tie group stays or goes
    as a whole; the kept set is the oracle's but for groups at the threshold that rounding may move (`exact`: not even those);
    the row sums to 1; and a kept value is the oracle's probability over the mass of the kernel's own kept set.  Relative
    3e-5 there: an exponent of up to 70 carries two fp32 roundings of 6e-8 (8e-6) and that of 1 / T (4e-6), beside those
    of exp, two divisions and the row's sums (1e-6); tokens below 1e-30 of the row are compared as zeros."""
    raw = osamp.softmax_t(logits, T)
    ref = osamp.filter_top_k_top_p(raw, top_k, top_p)
    order = np.argsort(logits, kind="stable")
    tied = logits[order][1:] == logits[order][:-1]
    assert (got[order][1:][tied] == got[order][:-1][tied]).all()
    visible = raw > 1e-30
    kept, kept_ref = (got > 0) & visible, (ref > 0) & visible
    odd = raw[kept != kept_ref]
    if odd.size:
        assert not exact
        # other logits whose probability is the k-th largest's to rounding, or one group where the nucleus' running sum ends to rounding
        at_k = np.partition(logits, -top_k)[-top_k]
        t_k = raw[logits == at_k][0]
        mass = raw[raw >= t_k].astype(np.float64).sum()
        ends = [raw[raw > odd.min()].astype(np.float64).sum(), raw[raw >= odd.max()].astype(np.float64).sum()]
        near_k = (np.abs(odd - t_k) <= 1e-6 * t_k).all() and (logits[kept != kept_ref] != at_k).all()
        assert np.ptp(odd) <= 1e-6 * odd.max() and (near_k or min(abs(c - float(np.float32(top_p)) * mass) for c in ends) <= 1e-6 * mass)
    assert abs(float(got.astype(np.float64).sum()) - 1.0) < 1e-5
    own = raw[kept].astype(np.float64)
    assert (np.abs(got[kept] - own / own.sum()) <= 3e-5 * own / own.sum()).all()


@pytest.mark.parametrize("top_k", [1, 50, 96, 97])  # the last k of the picked form, the first of the histograms
@pytest.mark.parametrize("V", [130, 1025, 32000])
def test_few_kept_tokens_are_picked_or_searched_alike(V, top_k):
    """Up to 96 kept tokens are picked among those that reach a bound; rows that give no usable bound or too many candidates
    (a constant row, more than 256 equal maxima, fewer finite entries than tokens to keep, the kept ones in one warp's piece)
    take the histograms as every row does beyond 96.  All follow the oracle's restriction of the row's probabilities, wherever
    the logits lie, ties at the threshold included."""
    T, K, Bn, top_p = 0.7, 4, 2, 0.9
    logits, rows, q, u = make_case(4000 + V, Bn, K, V, T, True)
    logits[0, 0] -= 100
    logits[0, 1] = 0.25
    logits[0, 2] = np.round(logits[0, 2] * 4) / 4                  # ties everywhere
    logits[0, 3, :min(V, 300)] = logits[0, 3].max() + 1            # more equal maxima than candidates
    logits[1, 0, 60:] = -np.inf                                    # fewer finite entries than tokens to keep
    logits[1, 1, :min(V - 1, 50)] += 40                            # the kept ones in one warp's piece
    logits[1, 2] *= 50
    logits[1, 3] += 300
    logits[0, 4, np.arange(V) % 3 > 0] = -np.inf                   # gaps
    logits[1, 4, 97:] = -np.inf                                    # just enough finite entries
    q = np.stack([[osamp.filter_top_k_top_p(q[b, i], top_k, top_p) for i in range(K)] for b in range(Bn)])
    rows[:, 1:] = synth.draw_tokens_from_rows(79, q.reshape(Bn * K, V)).reshape(Bn, K)
    B.set_sampling(top_k, top_p)
    try:
        n_acc, nxt, p = run_tail(logits, rows, q, u, T)
    finally:
        B.set_sampling(0, 1.0)
    for b in range(Bn):
        for i in range(K + 1):
            check_restricted_row(p[b, i], logits[b, i], T, top_k, top_p, exact=(b, i) in ((0, 1), (0, 3)))
        gu.check_decisions_on_own_rows(p[b], q[b], rows[b, 1:], u[b, :K], u[b, K], int(n_acc[b]), int(nxt[b]))


def test_picked_rows_cost_the_same_wherever_the_logits_lie():
    """The candidate bound does not hang on the logits' absolute size: rows around 300 gave more than 256 candidates each, went the
    general way after all and took twice the time of rows around 0."""
    Bn, K, V, T, top_k = 8, 5, 32000, 0.8, 50
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    base = torch.empty(Bn, K + 1, V, device="cuda").normal_(0.0, 2.0, generator=gen)
    q = torch.softmax(base[:, :K], -1).contiguous()
    rows, u = torch.zeros(Bn, K + 1, dtype=torch.int32, device="cuda"), torch.full((Bn, K + 1), 0.5, device="cuda")
    n_acc, nxt = torch.zeros(Bn, dtype=torch.int32, device="cuda"), torch.zeros(Bn, dtype=torch.int32, device="cuda")
    scratch = torch.empty(B.verify_scratch_bytes(Bn, K), dtype=torch.uint8, device="cuda")

    def best(logits):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ms = []
        for _ in range(8):
            ev[0].record()
            for _ in range(20):
                B.verify_from_logits(logits, K, rows, q, u, T, n_acc, nxt, 1, None, scratch)
            ev[1].record()
            torch.cuda.synchronize()
            ms.append(ev[0].elapsed_time(ev[1]))
        return min(ms)

    B.set_sampling(top_k, 0.9)
    try:
        near = best(base)
        assert max(best(base + 300.0), best(base - 100.0)) <= 1.4 * near
    finally:
        B.set_sampling(0, 1.0)


@pytest.mark.parametrize("top_k", [0, 37])
@pytest.mark.parametrize("V", [33, 8193, 32000, 65537])
@pytest.mark.parametrize("u_draw", [1.0, float("nan"), float("inf"), -0.25, 1.0 - 2.0 ** -24, 0.0])
def test_every_uniform_draws_a_token(u_draw, V, top_k):
    """A uniform outside [0, 1) - a float64 one close to 1 rounds to 1.0 - still writes a token: the last index with weight > 0
    from 1 on and for a NaN, the first one below 0; in the residual draw (sequence 0) and in the bonus draw (sequence 1).
    The end of the row weighs nothing."""
    K = 1
    logits = synth.gen_logits(91 + V, 2 * (K + 1), V, 1.5).reshape(2, K + 1, V)
    logits[:, :, V - V // 3:] = -np.inf
    q = np.stack([osamp.filter_top_k_top_p(osamp.softmax_t(synth.gen_logits(92 + b, 1, V, 1.5)[0], 1.0), top_k) for b in range(2)])[:, None]
    p_ref = np.stack([osamp.filter_top_k_top_p(osamp.softmax_t(logits[b, 0], 1.0), top_k) for b in range(2)])
    x = [int(np.argmax(q[0, 0])), int(np.argmax(p_ref[1]))]
    u = np.array([[2.0 * p_ref[0, x[0]] / q[0, 0, x[0]] + 1.0, u_draw], [0.0, u_draw]], np.float32)  # refused; accepted
    B.set_sampling(top_k, 1.0)
    try:
        n_acc, nxt, p = run_tail(logits, np.array([[0, x[0]], [0, x[1]]], np.int32), q, u, 1.0)
    finally:
        B.set_sampling(0, 1.0)
    assert n_acc.tolist() == [0, 1]
    for b, w in ((0, osamp.residual(p[0, 0], q[0, 0])), (1, p[1, 1])):
        live = np.nonzero(w > 0)[0]
        if not u_draw < 1.0:
            assert nxt[b] == live[-1]
        elif u_draw <= 0.0:
            assert nxt[b] == live[0]
        else:
            assert w[nxt[b]] > 0 and w[nxt[b]:].astype(np.float64).sum() >= 0.5 * 2.0 ** -24 * w.astype(np.float64).sum()


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("u", [1.0, float("nan")])
def test_a_draft_step_draws_a_token_for_a_uniform_of_one(u, fused):
    """As above for the draft's draw, in the stand-alone tail and in the one inside the forward kernel."""
    arch = synth.neox_like(2, 128, 4, 256, 640)
    m = B.Model(arch, B.upload_weights(arch, gu.scaled_weights(synth, arch, 21, 7.0)))
    kv, ws = B.KV(m, 1, 16), m.new_workspace(1, 1, 16)
    tok = torch.full((1, 1), -7, dtype=torch.int32, device="cuda")
    q = torch.zeros(1, 1, arch.vocab, device="cuda")
    x, uu = torch.tensor([[5]], dtype=torch.int32, device="cuda"), torch.tensor([[u]], device="cuda")
    if fused:
        B.draft_steps(m, kv, 1, x, 1, 1, None, 1.0, uu, 1, tok, 1, q, arch.vocab, ws)
    else:
        B.draft_step(m, kv, x, 1, 1, None, 1.0, uu, 1, tok, 1, q, arch.vocab, ws)
    assert int(tok.item()) == int(torch.nonzero(q[0, 0] > 0).max()) and kv.status() == 0


@pytest.mark.parametrize("top_k", [0, 50])
@pytest.mark.parametrize("V,n_bad", [(8192, 32), (8192, 256), (32000, 512), (66000, 1056)])
def test_a_run_of_nans_makes_the_whole_row_not_a_number(V, n_bad, top_k):
    """NaN logits that fill a whole warp's piece of the row (which then has no maximum) reach the row's sum like single ones:
    every probability of the row is NaN, its draft token is refused and the token of the largest finite logit is emitted; the
    neighbouring sequence is not touched."""
    logits, rows, q, u = make_case(4000 + V, 2, 1, V, 1.0, True)
    q = np.stack([osamp.filter_top_k_top_p(q[b, 0], top_k) for b in range(2)])[:, None]
    rows[:, 1] = [int(np.argmax(q[b, 0])) for b in range(2)]
    bad = np.zeros(V, bool)
    bad[n_bad * 3:n_bad * 4] = True
    logits[0, :, bad] = np.nan
    B.set_sampling(top_k, 1.0)
    try:
        n_acc, nxt, p = run_tail(logits, rows, q, u, 1.0)
    finally:
        B.set_sampling(0, 1.0)
    assert np.isnan(p[0]).all() and n_acc[0] == 0
    assert nxt[0] == int(np.argmax(np.where(bad, -np.inf, logits[0, 0])))
    assert np.isfinite(p[1]).all()
    gu.check_decisions_on_own_rows(p[1], q[1], rows[1, 1:], u[1, :1], u[1, 1], int(n_acc[1]), int(nxt[1]))


@pytest.mark.parametrize("T", [0.0, 0.8])
@pytest.mark.parametrize("V,Bn,K,want_p", [
    (1000, 1, 4, True), (8192, 1, 31, True), (8193, 4, 31, True), (32769, 2, 12, True), (50304, 1, 8, False), (50304, 9, 16, True),
    (65537, 2, 7, False), (131100, 3, 5, True),
])
def test_rows_in_clusters_of_their_own_give_the_same_bits(V, Bn, K, want_p, T):
    """The same verification with its rows walked by one cluster (the entry point without scratch always does) and, from some
    number of rows on, with a cluster per row in a launch before: equal decisions and p rows, bit for bit."""
    logits, rows, q, u = make_case(5000 + V, Bn, K, V, T, True)
    n0 = B.launch_count()
    n_acc, nxt, p = run_tail(logits, rows, q, u, T, want_p)
    launches = B.launch_count() - n0
    dev = "cuda"
    out = [torch.full((Bn,), -7, dtype=torch.int32, device=dev) for _ in range(2)]
    p1 = torch.zeros(Bn, K + 1, V, device=dev) if want_p else None
    B.verify_from_logits_noalloc(torch.from_numpy(logits).to(dev), K, torch.from_numpy(rows).to(dev),
                                 torch.from_numpy(q).to(dev), torch.from_numpy(u).to(dev), T, out[0], out[1], 1, p1)
    assert launches == (1 if (V, Bn) in ((1000, 1), (50304, 9)) or T == 0.0 and V in (8193, 50304, 65537) else 2)
    assert out[0].cpu().numpy().tolist() == n_acc.tolist() and out[1].cpu().numpy().tolist() == nxt.tolist()
    if want_p:
        assert np.array_equal(p1.cpu().numpy(), p)
