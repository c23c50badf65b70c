"""GPU parity of temperature-1 drafting (Algorithm 1 with Decode = a draw from
the softmax by the Gumbel-max rule) against the oracle.

Both sides draw the same Philox4x32-10 uniforms, so a device token must be
the oracle's argmax of the keys l + g at every position, except where the
oracle's top-2 key gap is a near-tie (then within the tie tolerance of the
maximum key); the drafted prefix is re-checked in the oracle's forced mode.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2607_07409_gb300 as dels
from parity import LP_TOL_BF16, LP_TOL_F32, check_draft, record
from test_gpu_parity import DEV, SMALL, _oracle_head, _with_table, _learned_weights

pytestmark = pytest.mark.gpu


def _sampled(name, seed=17, step=3, weights="learned"):
    w = synth.stress(SMALL[name])
    d = synth.make_inputs(w, device=DEV, target=False)
    if name == "gru_b64":
        d = _with_table(w, d)
    a, b = _learned_weights(w.n) if weights == "learned" else ([w.weight] * w.n, [w.weight] * w.n)
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
    tok, lp, gap, state = dr.sample(d["long"], prior, a, b, seed, step)
    torch.cuda.synchronize()
    assert dr.status() == 0
    W = {k: v for k, v in W.items() if k != "input_table"}
    return w, d, W, a, b, tok.cpu().numpy(), lp.cpu().numpy(), gap.cpu().numpy(), state


@pytest.mark.parametrize("name,seed,step", [("gru", 17, 3), ("gru_b64", 17, 3), ("gru_b100", 17, 3), ("mlp2", 17, 3),
                                            ("xfmr", 17, 3),
                                            ("markov", 17, 3), ("gru_f32", 17, 3), ("tiny", 17, 3),
                                            ("gru", 0xFEDCBA9876543210, 2 ** 32 - 1)])
def test_sampled_draft_matches_oracle(name, seed, step):
    """Every head; the last case puts both halves of the key and the whole
    step word of the counter to use."""
    w, d, W, a, b, tok, lp, gap, state = _sampled(name, seed, step)
    tol = LP_TOL_F32 if w.head.wdtype == "f32" else LP_TOL_BF16
    info = check_draft(tok, lp, gap, _oracle_head(w, W), d["long"].cpu(), oracle.log_prior(d["counts"]),
                       np.array(a), np.array(b), tol, sample=(seed, step))
    # the LSE of every fused row, kept for the verification
    lse = state[: w.B * w.n * 4].view(torch.float32).view(w.B, w.n).cpu().numpy()
    np.testing.assert_allclose(lse, info["ref"].lse, rtol=0, atol=tol * 4)
    print(name, record(f"sampled draft {name}", info))


@pytest.mark.parametrize("B,r,ldt", [(32, 384, "bf16"), (33, 768, "f32"), (64, 512, "bf16"), (40, 896, "bf16"),
                                     (9, 400, "bf16"), (32, 576, "f32"), (1, 512, "bf16"), (96, 512, "f32"),
                                     (128, 256, "f32")])
def test_sampled_draft_staged_activation_edges(B, r, ldt):
    """Both sides of the lines between copied and packed activations, and
    float32 logit tiles that leave no room for resident ones."""
    w = synth.stress(synth.Workload("staged", B=B, n=3, V=24008, logit_dtype=ldt,
                                    head=synth.HeadSpec("markov", "bf16", 0, 0, r), weight=0.5, seed=B))
    d = synth.make_inputs(w, device=DEV, target=False)
    a, b = _learned_weights(w.n)
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
    tok, lp, gap, _ = dr.sample(d["long"], dels.dels_prior_from_counts(d["counts"]).to(DEV), a, b, 17, 3)
    torch.cuda.synchronize()
    assert dr.status() == 0
    check_draft(tok.cpu().numpy(), lp.cpu().numpy(), gap.cpu().numpy(), _oracle_head(w, W), d["long"].cpu(),
                oracle.log_prior(d["counts"]), np.array(a), np.array(b), LP_TOL_BF16, sample=(17, 3))


@pytest.mark.parametrize("layers,B,V", [(2, 3, 1024), (2, 9, 1024), (1, 3, 1024), (2, 9, 4096)])
def test_sampled_f32_mlp_merged_in_its_first_product(layers, B, V):
    """A float32 MLP's first product decodes the position before it, and keeps
    that position's feature: two layers with few records (the fused launch),
    one layer and many records (a merge launch of its own)."""
    spec = synth.HeadSpec("mlp", "f32", 32, 100, 100, window=3, n_layers=layers)
    w = synth.stress(synth.Workload("f32_mlp", B=B, n=5, V=V, logit_dtype="f32", head=spec, weight=0.5, seed=B))
    d = synth.make_inputs(w, device=DEV, target=False)
    a, b = _learned_weights(w.n)
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
    tok, lp, gap, state = dr.sample(d["long"], prior, a, b, 23, 7)
    torch.cuda.synchronize()
    assert dr.status() == 0
    tok, lp, gap = tok.cpu().numpy(), lp.cpu().numpy(), gap.cpu().numpy()
    check_draft(tok, lp, gap, _oracle_head(w, W), d["long"].cpu(), oracle.log_prior(d["counts"]), np.array(a),
                np.array(b), LP_TOL_F32, sample=(23, 7))
    # the kept features, through the verification that rebuilds q from them
    target = synth.make_target_logits(w, d["long"], device=DEV)
    acc, bonus, bgap, st = _verify_raw(w, d, W, a, b, tok, lp, state, target, prior)
    assert st == 0
    _check_verify(w, d, W, a, b, tok, acc, bonus, bgap, target, 23, 7, LP_TOL_F32)


@pytest.mark.parametrize("offset", [1, 2])
def test_sampled_verify_unaligned_f32_weights(offset):
    """A float32 W_vocab off its 16-byte boundary gives the results of an aligned one."""
    w, d, W, a, b, tok, lp, gap, state = _sampled("gru_f32", 23, 7)
    target = synth.make_target_logits(w, d["long"], device=DEV)
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    one = _verify_raw(w, d, W, a, b, tok, lp, state, target, prior)
    wv = W["w_vocab"]
    shifted = torch.empty(wv.numel() + 4, device=DEV)[offset:offset + wv.numel()].view_as(wv)
    shifted.copy_(wv)
    two = _verify_raw(w, d, dict(W, w_vocab=shifted), a, b, tok, lp, state, target, prior)
    assert one[3] == 0 and two[3] == 0
    for x, y in zip(one, two):
        np.testing.assert_array_equal(x, y)


def test_sampled_calls_reject_a_step_outside_the_counter_word():
    w = synth.stress(SMALL["gru"])
    d = synth.make_inputs(w, device=DEV, target=False)
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
    with pytest.raises(dels.DelsError) as e:
        dr.sample(d["long"], prior, [0.3] * w.n, [0.3] * w.n, 1, 2 ** 32)
    assert e.value.code == dels.DELS_ERR_BAD_SHAPE


def test_sampled_draft_depends_on_seed_and_step_only():
    w, d, W, a, b, tok1, lp1, _, _ = _sampled("gru", 5, 9)
    _, _, _, _, _, tok2, lp2, _, _ = _sampled("gru", 5, 9)
    np.testing.assert_array_equal(tok1, tok2)
    np.testing.assert_array_equal(lp1, lp2)
    _, _, _, _, _, tok3, _, _, _ = _sampled("gru", 5, 10)
    _, _, _, _, _, tok4, _, _, _ = _sampled("gru", 6, 9)
    assert not np.array_equal(tok1, tok3) and not np.array_equal(tok1, tok4)


def test_sampled_draft_first_token_frequencies_follow_the_softmax():
    """x_0 over many steps: empirical frequencies against softmax(l_L^(0)) of a
    small, flat row (every token has mass)."""
    from scipy.stats import chisquare
    V, B = 16, 64
    w = synth.Workload("flat", B=B, n=1, V=V, logit_dtype="f32",
                       head=synth.HeadSpec("markov", "f32", 0, 0, 16), weight=0.0, seed=3)
    d = synth.make_inputs(w, device=DEV, target=False)
    row = torch.linspace(-1.0, 1.0, V, device=DEV)
    long = row.expand(B, 1, V).contiguous()
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    dr = dels.Drafter(w.head, W, B, 1, V)
    prior = torch.zeros(V, device=DEV)
    counts = np.zeros(V)
    for step in range(40):
        tok, _, _, _ = dr.sample(long, prior, [0.0], [0.0], 99, step)
        counts += np.bincount(tok.cpu().numpy().ravel(), minlength=V)
    p = torch.softmax(row.double(), 0).cpu().numpy()
    assert chisquare(counts, counts.sum() * p).pvalue > 1e-3


# ------------------------------------------------ speculative-sampling verification

def _verify(w, d, W, a, b, tok, lp, state, target, seed, step):
    head = dels.make_head(w.head, W)
    tdt = dels.dtype_code(target)
    nbytes = dels.dels_verify_sampled_workspace_bytes(head, w.B, w.n, w.V, tdt)
    assert nbytes > 0
    ws = torch.zeros(nbytes, dtype=torch.uint8, device=DEV)
    acc = torch.full((w.B,), -5, dtype=torch.int32, device=DEV)
    bonus = torch.full((w.B,), -5, dtype=torch.int32, device=DEV)
    bgap = torch.empty(w.B, dtype=torch.float32, device=DEV)
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    r = dels.dels_verify_block_sampled(head, torch.as_tensor(tok, device=DEV), torch.as_tensor(lp, device=DEV), state,
                                       d["long"], dels.dtype_code(d["long"]), prior, a, b, target, tdt, w.B, w.n, w.V,
                                       seed, step, acc, bonus, bgap, ws, nbytes)
    assert r == 0, dels.dels_status_string(r)
    torch.cuda.synchronize()
    assert dels.dels_read_status(ws) == 0
    return acc.cpu().numpy(), bonus.cpu().numpy(), bgap.cpu().numpy()


def _check_verify(w, d, W, a, b, tok, acc, bonus, bgap, target, seed, step, lp_tol):
    """Accepted lengths and bonus tokens against the oracle run on the device's
    drafted tokens (the oracle rebuilds q from its own fused rows)."""
    ref = oracle.draft_block(_oracle_head(w, W), d["long"].cpu(), oracle.log_prior(d["counts"]), np.array(a),
                             np.array(b), forced=tok, sample=(seed, step), keep_fused=True)
    r_acc, r_bonus, info = oracle.verify_sampled(tok, ref.fused, target.cpu(), seed, step)
    # a test whose ratio p/q lies within the logprob tolerance of its uniform may go either way
    close = info["margin"] < 8 * lp_tol
    same_acc = acc == r_acc
    assert np.all(same_acc | close), (acc, r_acc, info["margin"])
    ok = same_acc & ~close
    # the bonus draw: identical unless the oracle's key gap is a near-tie
    tie = info["bonus_gap"] < 0.05
    bad = ok & (bonus != r_bonus) & ~tie
    assert not bad.any(), (bonus[bad], r_bonus[bad], info["bonus_gap"][bad])
    fin = ok & (bonus == r_bonus) & np.isfinite(info["bonus_gap"])
    return dict(requests=int(len(acc)), close=int(close.sum()), ties=int((ok & tie).sum()),
                accept=acc.tolist(), gap_err=float(np.abs(bgap[fin] - info["bonus_gap"][fin]).max(initial=0)))


@pytest.mark.parametrize("name", ["gru", "gru_b64", "mlp2", "xfmr", "markov", "gru_f32", "tiny"])
def test_sampled_verify_matches_oracle(name):
    seed, step = 23, 7
    w, d, W, a, b, tok, lp, gap, state = _sampled(name, seed, step)
    target = synth.make_target_logits(w, d["long"], device=DEV)
    acc, bonus, bgap = _verify(w, d, W, a, b, tok, lp, state, target, seed, step)
    tol = LP_TOL_F32 if w.head.wdtype == "f32" else LP_TOL_BF16
    info = _check_verify(w, d, W, a, b, tok, acc, bonus, bgap, target, seed, step, tol)
    print(name, info)
    assert np.all((acc >= 0) & (acc <= w.n)) and np.all((bonus >= 0) & (bonus < w.V))


def _verify_raw(w, d, W, a, b, tok, lp, state, target, prior):
    """One verification call (seed 23, step 7): outputs and device status."""
    head = dels.make_head(w.head, W)
    tdt = dels.dtype_code(target)
    nbytes = dels.dels_verify_sampled_workspace_bytes(head, w.B, w.n, w.V, tdt)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device=DEV)
    acc, bonus = (torch.full((w.B,), -5, dtype=torch.int32, device=DEV) for _ in range(2))
    bgap = torch.empty(w.B, dtype=torch.float32, device=DEV)
    r = dels.dels_verify_block_sampled(head, torch.as_tensor(tok, device=DEV), torch.as_tensor(lp, device=DEV), state,
                                       d["long"], dels.dtype_code(d["long"]), prior, a, b, target, tdt, w.B, w.n, w.V,
                                       23, 7, acc, bonus, bgap, ws, nbytes)
    assert r == 0, dels.dels_status_string(r)
    return acc.cpu().numpy(), bonus.cpu().numpy(), bgap.cpu().numpy(), dels.dels_read_status(ws)


@pytest.mark.parametrize("name", ["gru", "gru_f32"])
@pytest.mark.parametrize("target_dtype", [torch.float32, torch.bfloat16])
def test_sampled_verify_unaligned_prior_takes_the_element_path(name, target_dtype):
    """A prior off its 16-byte boundary (the residual's element loads) gives
    the results of an aligned one (its 16-byte loads) bit for bit, for both
    target types and both draft-logit types."""
    w, d, W, a, b, tok, lp, gap, state = _sampled(name, 23, 7)
    target = synth.make_target_logits(w, d["long"], device=DEV).to(target_dtype)
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    shifted = torch.empty(w.V + 4, device=DEV)[1:w.V + 1]
    shifted.copy_(prior)
    one = _verify_raw(w, d, W, a, b, tok, lp, state, target, prior)
    two = _verify_raw(w, d, W, a, b, tok, lp, state, target, shifted)
    assert one[3] == 0 and two[3] == 0
    for x, y in zip(one, two):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("target_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("what", ["nan", "nan_first", "inf", "masked", "masked_row"])
def test_sampled_verify_nonfinite_target_rows(target_dtype, what):
    """A NaN, a +inf or an all -inf target row sets the status; a row with
    masked (-inf) entries does not and keeps its LSE."""
    w, d, W, a, b, tok, lp, gap, state = _sampled("gru", 23, 7)
    target = synth.make_target_logits(w, d["long"], device=DEV).to(target_dtype)
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    if what == "nan":
        target[1, 2, w.V - 3] = float("nan")
    elif what == "nan_first":                 # in a group with nothing finite, before anything else
        target[1, 2, :8] = float("-inf")
        target[1, 2, 1] = float("nan")
    elif what == "inf":
        target[1, 2, 9] = float("inf")
    elif what == "masked_row":
        target[1, 2] = float("-inf")
    else:
        target[:, :, ::3] = float("-inf")
    acc, bonus, bgap, st = _verify_raw(w, d, W, a, b, tok, lp, state, target, prior)
    if what == "masked":
        assert st == 0
        info = _check_verify(w, d, W, a, b, tok, acc, bonus, bgap, target, 23, 7, LP_TOL_BF16)
        assert info["requests"] == w.B
    else:
        assert st & dels.DELS_STATUS_NONFINITE


def test_sampled_verify_of_every_request_that_a_counter_holds():
    """65536 requests and a float32 width whose products take one request per
    CTA: more groups than a launch has rows of CTAs."""
    B, n, V, R = 65536, 1, 8, 12292
    w = synth.Workload("many", B=B, n=n, V=V, logit_dtype="f32", head=synth.HeadSpec("markov", "f32", 0, 0, R),
                       weight=1.0, seed=3)
    W = {"emb": torch.zeros(V, R, device=DEV), "w_vocab": torch.zeros(V, R, device=DEV)}
    state = torch.zeros(B * n * (R + 1) * 4 + 4096, dtype=torch.uint8, device=DEV)   # every q and input zero
    tok = torch.zeros(B, n, dtype=torch.int32, device=DEV)
    lp = torch.full((B, n), -60.0, device=DEV)                                       # p / q large: accepted
    lp[1::2] = 60.0                                                                  # rejected
    rows = torch.zeros(B, n, V, device=DEV)
    target = torch.zeros(B, n + 1, V, device=DEV)
    acc, bonus, bgap, st = _verify_raw(w, {"long": rows}, W, [0.0], [0.0], tok, lp, state, target,
                                       torch.zeros(V, device=DEV))
    assert st == 0 and np.array_equal(acc, 1 - np.arange(B) % 2) and np.all((bonus >= 0) & (bonus < V))


def test_calls_from_several_host_threads():
    """Blocks drafted and verified by threads with streams and workspaces of
    their own, all at once, equal the same calls made one after another."""
    import threading
    names = ["gru", "gru_f32", "markov", "gru_b64"]
    jobs = []
    for name in names:
        w = synth.stress(SMALL[name])
        d = synth.make_inputs(w, device=DEV, target=False)
        W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
        a, b = _learned_weights(w.n)
        jobs.append((w, d, W, a, b, dels.dels_prior_from_counts(d["counts"]).to(DEV),
                     synth.make_target_logits(w, d["long"], device=DEV)))

    def one(job, rounds):
        w, d, W, a, b, prior, target = job
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(rounds):
                dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
                tok, lp, gap, state = dr.sample(d["long"], prior, a, b, 23, 7)
                acc, bonus, bgap, st = _verify_raw(w, d, W, a, b, tok, lp, state, target, prior)
            torch.cuda.current_stream().synchronize()
            return [x.cpu().numpy() for x in (tok, lp, gap)] + [acc, bonus, bgap, np.array([st, dr.status()])]

    torch.cuda.synchronize()
    want = [one(j, 1) for j in jobs]
    got = [None] * len(jobs)

    def run(i):
        got[i] = one(jobs[i], 8)

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for x, y in zip(got, want):
        for u, v in zip(x, y):
            np.testing.assert_array_equal(u, v)


def test_sampled_verify_right_behind_the_launch_that_writes_its_weights():
    """W_vocab of a float32 head written by a launch that lets its successors
    start early (an input table, 48 wide): the verification called right behind
    it reads the new weights."""
    V, R, B, n = 100000, 48, 2, 3
    g = torch.Generator(device=DEV).manual_seed(4)
    gru = synth.HeadSpec("gru", "bf16", 4096, R // 3, 16)
    E = torch.randn(V, 4096, generator=g, device=DEV).to(torch.bfloat16)
    Wih = torch.randn(R, 4096, generator=g, device=DEV).to(torch.bfloat16) / 64
    maker = dels.make_head(gru, {"emb": E, "w_ih": Wih, "w_vocab": E})
    G = torch.empty(V, R, device=DEV)
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)

    def write_weights():
        assert dels.dels_gru_build_input_table(maker, V, G, V * R * 4, ws, 256) == 0

    write_weights()
    w = synth.Workload("behind", B=B, n=n, V=V, logit_dtype="f32", head=synth.HeadSpec("markov", "f32", 0, 0, R),
                       weight=1.0, seed=3)
    W = {"emb": torch.randn(V, R, generator=g, device=DEV) * 0.3, "w_vocab": G}
    d = {"long": torch.randn(B, n, V, generator=g, device=DEV) * 2}
    prior = torch.full((V,), -float(np.log(V)), device=DEV)
    a = b = [1.0] * n
    dr = dels.Drafter(w.head, W, B, n, V)
    tok, lp, gap, state = dr.sample(d["long"], prior, a, b, 23, 7)
    lp = lp + torch.tensor([-50.0, 50.0, 0.0], device=DEV)       # accepted, then rejected: q is rebuilt from W_vocab
    target = torch.randn(B, n + 1, V, generator=g, device=DEV) * 2
    head = dels.make_head(w.head, W)
    nbytes = dels.dels_verify_sampled_workspace_bytes(head, B, n, V, dels.DELS_F32)
    vws = torch.zeros(nbytes, dtype=torch.uint8, device=DEV)
    acc, bonus = (torch.empty(B, dtype=torch.int32, device=DEV) for _ in range(2))
    bgap = torch.empty(B, dtype=torch.float32, device=DEV)

    def verify():                                 # no launch but the library's in between
        assert dels.dels_verify_block_sampled(head, tok, lp, state, d["long"], dels.DELS_F32, prior, a, b, target,
                                              dels.DELS_F32, B, n, V, 23, 7, acc, bonus, bgap, vws, nbytes) == 0

    def results():
        assert dels.dels_read_status(vws) == 0
        return acc.tolist(), bonus.tolist(), bgap.tolist()

    verify()
    want = results()
    assert want[0] == [1] * B
    for _ in range(5):
        G.fill_(3.0)
        torch.cuda.synchronize()
        write_weights()
        verify()
        assert results() == want


@pytest.mark.parametrize("mask", ["lowest", -1e30, -1e9])
@pytest.mark.parametrize("target_dtype", [torch.float32, torch.bfloat16])
def test_sampled_rows_masked_by_a_finite_value(target_dtype, mask):
    """Draft and target rows whose leading half, and nearly all of one row, hold
    a finite mask."""
    w = synth.stress(SMALL["gru"])
    d = synth.make_inputs(w, device=DEV, target=False)
    value = torch.finfo(torch.bfloat16).min if mask == "lowest" else mask
    d["long"][:, :, : w.V // 2] = value
    a, b = _learned_weights(w.n)
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
    tok, lp, gap, state = dr.sample(d["long"], prior, a, b, 23, 7)
    torch.cuda.synchronize()
    assert dr.status() == 0
    tok, lp, gap = tok.cpu().numpy(), lp.cpu().numpy(), gap.cpu().numpy()
    check_draft(tok, lp, gap, _oracle_head(w, W), d["long"].cpu(), oracle.log_prior(d["counts"]), np.array(a),
                np.array(b), LP_TOL_BF16, sample=(23, 7))
    target = synth.make_target_logits(w, d["long"], device=DEV).to(target_dtype)
    target[:, :, : w.V // 2] = torch.finfo(target_dtype).min if mask == "lowest" else mask
    target[1, 2, : w.V - 9] = value
    acc, bonus, bgap, st = _verify_raw(w, d, W, a, b, tok, lp, state, target, prior)
    assert st == 0
    info = _check_verify(w, d, W, a, b, tok, acc, bonus, bgap, target, 23, 7, LP_TOL_BF16)
    assert info["requests"] == w.B


@pytest.mark.parametrize("target_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [72, 20000])
def test_sampled_verify_denormal_residual(target_dtype, V):
    """A residual whose every weight is a denormal float32 is drawn from, not
    taken for zero: p and q agree on token 0 and only token 5 has p > q, by
    e^-90 (a draft log-probability set far too high rejects token 0)."""
    w = synth.stress(synth.Workload("denormal", B=2, n=1, V=V, logit_dtype="f32",
                                    head=synth.HeadSpec("markov", "bf16", 0, 0, 64), weight=0.5, seed=3))
    d = synth.make_inputs(w, device=DEV, target=False)
    d["long"].fill_(-200.0)
    d["long"][:, :, 0] = 0.0
    W = {k[5:]: v for k, v in d.items() if k.startswith("head.")}
    prior = dels.dels_prior_from_counts(d["counts"]).to(DEV)
    dr = dels.Drafter(w.head, W, w.B, w.n, w.V)
    tok, lp, gap, state = dr.sample(d["long"], prior, [0.0], [0.0], 23, 7)
    assert tok.tolist() == [[0], [0]]
    target = torch.full((w.B, 2, V), -200.0, device=DEV)
    target[:, :, 0] = 0.0
    target[:, :, 5] = -90.0
    acc, bonus, bgap, st = _verify_raw(w, d, W, [0.0], [0.0], tok, lp + 60.0, state, target.to(target_dtype), prior)
    assert st == 0 and acc.tolist() == [0, 0]
    assert bonus.tolist() == [5, 5] and np.all(np.isinf(bgap))


@pytest.mark.parametrize("name", ["gru", "markov", "tiny"])
def test_sampled_verify_rejection_at_position_zero(name):
    """The target rules out every x_0 (p_0(x_0) = 0): every request rejects at
    0 and its bonus comes from the residual of softmax(l_L^(0)), never x_0."""
    seed, step = 31, 2
    w, d, W, a, b, tok, lp, gap, state = _sampled(name, seed, step)
    target = synth.make_target_logits(w, d["long"], device=DEV).clone()
    for bb in range(w.B):
        target[bb, 0, int(tok[bb, 0])] = float("-inf")
    acc, bonus, bgap = _verify(w, d, W, a, b, tok, lp, state, target, seed, step)
    assert np.all(acc == 0) and np.all(bonus != tok[:, 0])
    tol = LP_TOL_F32 if w.head.wdtype == "f32" else LP_TOL_BF16
    print(name, _check_verify(w, d, W, a, b, tok, acc, bonus, bgap, target, seed, step, tol))


def test_gumbel_transform_error_over_every_uniform():
    """The device's g = -ln(-ln u) for every one of the 2^23 uniforms a Philox
    word can give (u = (2k + 1) 2^-24), against the float64 transform: the
    largest absolute error stays below 4e-6 (the exponential variate E = -ln u
    carries a relative error of ~1.5e-6 at most, which g inherits as an
    absolute error, plus the fast outer logarithm's)."""
    k = torch.arange(1 << 23, dtype=torch.int64)
    w = k << 9                                   # the word's top 23 bits select k
    bits = torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32).to(DEV)   # same 32 bits, as int32
    g = torch.empty(1 << 23, dtype=torch.float32, device=DEV)
    assert dels.dels_selftest_gumbel(bits, g, 1 << 23) == 0
    torch.cuda.synchronize()
    u = (2.0 * np.arange(1 << 23, dtype=np.float64) + 1.0) / 2.0 ** 24
    exact = -np.log(-np.log(u))
    err = np.abs(g.cpu().numpy().astype(np.float64) - exact)
    worst = int(np.argmax(err))
    print(f"gumbel transform: max |error| {err[worst]:.3g} at u = {u[worst]:.9f}, mean {err.mean():.3g}")
    assert err[worst] < 4e-6
    assert dels.dels_selftest_gumbel(bits, g, -1) == dels.DELS_ERR_BAD_SHAPE
    assert dels.dels_selftest_gumbel(None, g, 1) == dels.DELS_ERR_NULL_POINTER
