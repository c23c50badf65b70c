"""GPU parity of the device unigram-prior estimation (Appendix A) against the oracle.

Counts and tallies are integers and must match bit for bit. The log prior is
evaluated in float64 on both sides and stored as float32 by the device, so
each entry must lie within one float32 spacing of the oracle's fp64 value.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2607_07409_gb300 as dels

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _ws(V, N):
    n = dels.dels_prior_workspace_bytes(V, N)
    assert n > 0
    return torch.zeros(n, dtype=torch.uint8, device=DEV), n


def _check_log_prior(got, counts, lam):
    ref = oracle.log_prior(counts, lam)
    ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    err = np.abs(got.cpu().numpy().astype(np.float64) - ref)
    assert np.all(err <= ulp), f"max error {err.max()} ulp {ulp[np.argmax(err)]}"


def _estimate(tok, mask, V, lam=1.0):
    out, counts, tally = dels.estimate_prior(tok, mask, V, lam)
    torch.cuda.synchronize()
    return out, counts.cpu().numpy(), tally.cpu().numpy()


def _corpus(V, N, seed, bad=0):
    tok, mask = synth.make_corpus(V, N, seed)
    if bad:
        g = torch.Generator().manual_seed(seed)
        where = torch.randperm(N, generator=g)[:bad]
        tok[where] = torch.tensor([-1, V, V + 7, -(2 ** 31)], dtype=torch.int32).repeat(bad)[:bad]
        mask[where] = 1
    return tok, mask


@pytest.mark.parametrize("V,N,seed,lam", [
    (1000, 100003, 1, 1.0),        # ragged tail after the vector range
    (151936, 1 << 20, 2, 1.0),
    (32000, 511, 3, 0.5),          # shorter than one warp step: all scalar
    (7, 4096, 4, 2.0),             # tiny vocabulary: every id hot
])
def test_estimate_matches_oracle(V, N, seed, lam):
    tok, mask = _corpus(V, N, seed)
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V, lam)
    np.testing.assert_array_equal(c, c_ref)
    assert tally.tolist() == [n_in, n_out]
    _check_log_prior(out, c_ref, lam)


def test_out_of_range_ids_are_tallied_and_flagged():
    V, N = 5000, 70001
    tok, mask = _corpus(V, N, 5, bad=37)
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    assert n_out == 37
    ws, nbytes = _ws(V, N)
    out = torch.empty(V, dtype=torch.float32, device=DEV)
    counts = torch.empty(V, dtype=torch.int64, device=DEV)
    tally = torch.empty(2, dtype=torch.int64, device=DEV)
    r = dels.dels_prior_estimate(tok.to(DEV), mask.to(DEV), N, V, 1.0, out, counts, tally, ws, nbytes)
    assert r == 0
    assert dels.dels_read_status(ws) == dels.DELS_STATUS_BAD_TOKEN
    np.testing.assert_array_equal(counts.cpu().numpy(), c_ref)
    assert tally.cpu().tolist() == [n_in, n_out]
    _check_log_prior(out, c_ref, 1.0)


@pytest.mark.parametrize("tok_off,mask_off", [(1, 1), (2, 2), (3, 3), (1, 0), (0, 3), (2, 1)])
def test_unaligned_corpus_pieces(tok_off, mask_off):
    """Offsets into a larger corpus: equal offsets keep a vector range, others go one by one."""
    V, N = 3000, 40000
    tok, mask = _corpus(V, N + 8, 6)
    t_dev, m_dev = tok.to(DEV), mask.to(DEV)
    n = N - 5
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok[tok_off:tok_off + n].numpy(),
                                                    mask[mask_off:mask_off + n].numpy(), V)
    ws, nbytes = _ws(V, n)
    counts = torch.zeros(V, dtype=torch.int64, device=DEV)
    tally = torch.zeros(2, dtype=torch.int64, device=DEV)
    r = dels.dels_prior_count(t_dev[tok_off:], m_dev[mask_off:], n, V, counts, tally, ws, nbytes)
    assert r == 0
    torch.cuda.synchronize()
    np.testing.assert_array_equal(counts.cpu().numpy(), c_ref)
    assert tally.cpu().tolist() == [n_in, n_out]


def test_pieces_accumulate_then_log_equals_one_call():
    V, N = 151936, 300000
    tok, mask = _corpus(V, N, 7)
    t_dev, m_dev = tok.to(DEV), mask.to(DEV)
    ws, nbytes = _ws(V, N)
    counts = torch.zeros(V, dtype=torch.int64, device=DEV)
    tally = torch.zeros(2, dtype=torch.int64, device=DEV)
    cuts = [0, 12345, 12346, 200000, N]
    for a, b in zip(cuts[:-1], cuts[1:]):
        assert dels.dels_prior_count(t_dev[a:], m_dev[a:], b - a, V, counts, tally, ws, nbytes) == 0
    out = torch.empty(V, dtype=torch.float32, device=DEV)
    assert dels.dels_prior_log(counts, V, 1.0, out, ws, nbytes) == 0
    c_ref, n_in, _ = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    np.testing.assert_array_equal(counts.cpu().numpy(), c_ref)
    assert tally.cpu().tolist() == [n_in, 0]
    _check_log_prior(out, c_ref, 1.0)
    # the ticket of the two-level sum is re-armed: a second call gives the same result
    out2 = torch.empty_like(out)
    assert dels.dels_prior_log(counts, V, 1.0, out2, ws, nbytes) == 0
    assert torch.equal(out, out2)
    one, c1, _ = _estimate(t_dev, m_dev, V)
    assert torch.equal(one, out)


def test_empty_corpus_and_all_unmasked_give_the_uniform_prior():
    V = 1000
    ref = np.full(V, -np.log(V))
    for tok, mask in ((torch.zeros(0, dtype=torch.int32), torch.zeros(0, dtype=torch.uint8)),
                      (torch.arange(5000, dtype=torch.int32) % V, torch.zeros(5000, dtype=torch.uint8))):
        out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V)
        assert not c.any() and tally.tolist() == [0, 0]
        _check_log_prior(out, np.zeros(V, np.int64), 1.0)
        np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=1e-7)


def test_single_hot_id_and_nonunit_mask_bytes():
    """Every position the same id (all atomics on one address) and mask bytes other than 1."""
    V, N = 151936, (1 << 22) + 3
    tok = torch.full((N,), 4242, dtype=torch.int32)
    mask = torch.full((N,), 255, dtype=torch.uint8)
    mask[::3] = 0
    out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V)
    expect = int((mask != 0).sum())
    assert c[4242] == expect and c.sum() == expect and tally.tolist() == [expect, 0]
    c_ref = np.zeros(V, np.int64)
    c_ref[4242] = expect
    _check_log_prior(out, c_ref, 1.0)


def test_full_corpus_counts_match_oracle():
    """The benchmark corpus: 2^28 positions over V = 151936, generated on the device."""
    w = synth.WORKLOADS["qwen3_8b_batched"]
    tok, mask = synth.make_corpus(w.V, synth.CORPUS_TOKENS, w.seed, device=DEV)
    out, c, tally = _estimate(tok, mask, w.V)
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.cpu().numpy(), mask.cpu().numpy(), w.V)
    np.testing.assert_array_equal(c, c_ref)
    assert tally.tolist() == [n_in, n_out]
    _check_log_prior(out, c_ref, 1.0)


# ------------------------------------------------------------- long ranges of large vocabularies
# Vocabularies above 230400 ids: the hot/cold scheme (a prefix counted exactly,
# the most frequent ids so far on chip, the others added to the global counts
# directly). Up to that, the half-word slices; each test runs on both.

HOT_N = (1 << 24) + 1234
HALVES_V, HOT_V = 151936, 250000


@pytest.mark.parametrize("V", [HALVES_V, HOT_V])
def test_hot_cold_path_matches_oracle_with_bad_ids(V):
    tok, mask = _corpus(V, HOT_N, 8, bad=101)
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    ws, nbytes = _ws(V, HOT_N)
    out = torch.empty(V, dtype=torch.float32, device=DEV)
    counts = torch.empty(V, dtype=torch.int64, device=DEV)
    tally = torch.empty(2, dtype=torch.int64, device=DEV)
    assert dels.dels_prior_estimate(tok.to(DEV), mask.to(DEV), HOT_N, V, 1.0, out, counts, tally, ws, nbytes) == 0
    assert dels.dels_read_status(ws) == dels.DELS_STATUS_BAD_TOKEN
    np.testing.assert_array_equal(counts.cpu().numpy(), c_ref)
    assert tally.cpu().tolist() == [n_in, n_out] and n_out == 101
    _check_log_prior(out, c_ref, 1.0)


@pytest.mark.parametrize("V", [HALVES_V, HOT_V])
def test_hot_cold_path_when_the_prefix_misleads(V):
    """The prefix holds one id only, the rest is uniform over V: almost every
    later position is cold and is added to the global counts."""
    g = torch.Generator().manual_seed(9)
    tok = torch.randint(0, V, (HOT_N,), generator=g, dtype=torch.int32)
    tok[: 1 << 23] = 77
    mask = (torch.rand(HOT_N, generator=g) < 0.9).to(torch.uint8)
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V)
    np.testing.assert_array_equal(c, c_ref)
    assert tally.tolist() == [n_in, n_out]


@pytest.mark.parametrize("V", [HALVES_V, HOT_V])
def test_hot_cold_pieces_on_top_of_earlier_counts(V):
    """A second long piece chooses its hot set from counts that already hold the first."""
    tok, mask = _corpus(V, 2 * HOT_N, 10)
    t_dev, m_dev = tok.to(DEV), mask.to(DEV)
    ws, nbytes = _ws(V, HOT_N)
    counts = torch.zeros(V, dtype=torch.int64, device=DEV)
    tally = torch.zeros(2, dtype=torch.int64, device=DEV)
    for a in (0, HOT_N):
        assert dels.dels_prior_count(t_dev[a:], m_dev[a:], HOT_N, V, counts, tally, ws, nbytes) == 0
    torch.cuda.synchronize()
    c_ref, n_in, _ = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    np.testing.assert_array_equal(counts.cpu().numpy(), c_ref)
    assert tally.cpu().tolist() == [n_in, 0]


@pytest.mark.parametrize("V", [HALVES_V, HOT_V])
def test_hot_path_hand_off_of_a_single_id(V):
    """One id at every loss-masked position of a long range: every CTA's 16-bit
    bin for it passes 2^15 twice and hands it to the global count."""
    N = HOT_N if V == HALVES_V else 2 * HOT_N     # the hot scheme's bins start after its prefix
    tok = torch.full((N,), 4242, dtype=torch.int32)
    mask = torch.full((N,), 3, dtype=torch.uint8)
    mask[::3] = 0
    out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V)
    expect = int((mask != 0).sum())
    counted = expect - ((1 << 22) if V == HOT_V else 0)
    assert counted // torch.cuda.get_device_properties(0).multi_processor_count > 2 * 2 ** 15
    assert c[4242] == expect and c.sum() == expect and tally.tolist() == [expect, 0]


@pytest.mark.parametrize("V", [15 * 10129, 15 * 16666])
def test_hot_path_vocabulary_a_multiple_of_15_with_bad_ids(V):
    """An id clamped to V falls on the remap table's zero sentinel word, past the
    last word that holds vocabulary ids."""
    tok, mask = _corpus(V, HOT_N, 11, bad=57)
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V)
    np.testing.assert_array_equal(c, c_ref)
    assert tally.tolist() == [n_in, n_out] and n_out == 57


# ----------------------------------------------------------- half-word slices


@pytest.mark.parametrize("V,N", [
    (57601, 1 << 23),              # past one slice of 32-bit bins: one slice of halves
    (115200, (1 << 23) + 77),      # the largest vocabulary of one slice
    (115201, (1 << 23) + 5),       # two slices, an odd vocabulary
    (115208, (1 << 23) - 1),       # one position short of the rule: 32-bit slices
    (230400, (1 << 24) + 3),       # the largest vocabulary of two slices, a range the hot scheme would take
    (230401, (1 << 24) + 3),       # one id more: a prefix of 32-bit slices, then the hot scheme
    (230401, 100003),              # ... and a short range
])
def test_half_word_slices_match_oracle(V, N):
    """Uniform ids (every bin used), a share of bad ids and of one hot id, at the edges of the plan."""
    g = torch.Generator().manual_seed(V + N)
    tok = torch.randint(-2, V + 2, (N,), generator=g, dtype=torch.int32)
    tok[torch.rand(N, generator=g) < 0.2] = V - 1
    tok[::4999] = -(2 ** 31)
    mask = (torch.rand(N, generator=g) < 0.75).to(torch.uint8) * 2
    c_ref, n_in, n_out = oracle.count_masked_tokens(tok.numpy(), mask.numpy(), V)
    out, c, tally = _estimate(tok.to(DEV), mask.to(DEV), V)
    np.testing.assert_array_equal(c, c_ref)
    assert tally.tolist() == [n_in, n_out] and n_out > 0
    _check_log_prior(out, c_ref, 1.0)


@pytest.mark.parametrize("V", [100000, 151936, 250000])   # one and two half-word slices, the hot scheme
@pytest.mark.parametrize("ids", [[77776], [77777], [77776, 77777], [77776, 77777, 77776, 3]])
def test_bins_under_one_or_two_ids(V, ids):
    """A range of one or two ids, the two halves of one word of bins: every
    add of a CTA meets the same word, and every bin hands over many times."""
    N = (1 << 25) + 19
    tok = torch.tensor(ids, dtype=torch.int32, device=DEV).repeat((N + len(ids) - 1) // len(ids))[:N].contiguous()
    mask = torch.ones(N, dtype=torch.uint8, device=DEV)
    ref = np.bincount(tok.cpu().numpy(), minlength=V)
    for _ in range(3):
        out, c, tally = _estimate(tok, mask, V)
        np.testing.assert_array_equal(c, ref)
        assert tally.tolist() == [N, 0]


@pytest.mark.parametrize("V", [100000, 151936, 250000])
def test_pieces_counted_on_several_streams(V):
    """Pieces with workspaces of their own, counted at the same time into one
    set of counts."""
    N, S = (1 << 24) + 512, 3
    g = torch.Generator(device=DEV).manual_seed(V)
    tok = torch.randint(0, V, (N,), generator=g, device=DEV, dtype=torch.int32)
    mask = torch.ones(N, dtype=torch.uint8, device=DEV)
    one = torch.bincount(tok, minlength=V)
    streams = [torch.cuda.Stream() for _ in range(S)]
    ws = [_ws(V, N) for _ in range(S)]
    for _ in range(5):
        counts = torch.zeros(V, dtype=torch.int64, device=DEV)
        tally = torch.zeros(2, dtype=torch.int64, device=DEV)
        torch.cuda.synchronize()
        for s, (w, nbytes) in zip(streams, ws):
            assert dels.dels_prior_count(tok, mask, N, V, counts, tally, w, nbytes, stream=s) == 0
        torch.cuda.synchronize()
        assert torch.equal(counts, S * one) and tally.tolist() == [S * N, 0]


@pytest.mark.parametrize("lam", [5e-324, 1e-310, 1e-5, 0.3, 3e7, 1e301])
def test_log_prior_over_smoothing_weights(lam):
    """The table-driven logarithm and, where c + lambda is denormal, the general one."""
    V = 3000
    c_ref = np.concatenate([np.arange(2000), 2 ** np.linspace(0, 50, 1000)]).astype(np.int64)
    counts = torch.from_numpy(c_ref).to(DEV)
    ws, nbytes = _ws(V, 0)
    out = torch.empty(V, dtype=torch.float32, device=DEV)
    assert dels.dels_prior_log(counts, V, lam, out, ws, nbytes) == 0
    c = c_ref.astype(np.float64)
    ref = np.log(c + lam) - np.log(c.sum() + V * lam)
    got = out.cpu().numpy().astype(np.float64)
    # one float32 rounding of the result, and the float64 error of the two logarithms
    assert np.all(np.abs(got - ref) <= np.abs(ref) * 2.0 ** -24 + 1e-12), np.abs(got - ref).max()


@pytest.mark.parametrize("lam", [1e-310, 1e-9, 0.3, 1.0, 77.0])
@pytest.mark.parametrize("top", [1, 63, 2 ** 20 - 1, 2 ** 20, 2 ** 27 - 2, 2 ** 27, 2 ** 31 + 1])
def test_log_prior_of_a_dominating_id(top, lam):
    """One or two ids, one of them with nearly all of the mass and a count next to
    a power of two (the two logarithms' arguments on either side of a table
    interval): within one float32 rounding, relative to l_P itself."""
    for counts in ([top, 0], [3, top], [top, top], [top, top // 1000], [top // 1024, top], [top]):
        c = np.array(counts, np.int64)
        V = len(counts)
        ws, nbytes = _ws(V, 0)
        out = torch.empty(V, dtype=torch.float32, device=DEV)
        assert dels.dels_prior_log(torch.from_numpy(c).to(DEV), V, lam, out, ws, nbytes) == 0
        s = float(c.sum()) + V * lam
        with np.errstate(divide="ignore"):
            ref = np.where(c + lam > s / 2, np.log1p(-((c.sum() - c) + (V - 1) * lam) / s),
                           np.log((c + lam) / s))
        got = out.cpu().numpy().astype(np.float64)
        # half a unit of float32 (denormals too), and the float64 errors of either side
        assert np.all(np.abs(got - ref) <= np.abs(ref) * (2.0 ** -24 + 1e-12) + 2.0 ** -150), (got, ref)
