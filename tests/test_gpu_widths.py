"""Calls of every token-row padding on a decoder whose projections end in odd
and partial tiles (hidden 384: 3 tiles of 128; gate/up 7; vocabulary 8 and a
fraction; 10 heads): the first request of each call against the oracle, and
every request's rows against the same request verified alone, bit for bit."""
import numpy as np
import pytest

from synth import workloads as W
from tests.helpers import LOGIT_TOL, Pair, run_gpu_block

pytestmark = pytest.mark.gpu

ODD = W.ModelConfig("odd", 2, 384, 6, 2, 64, 448, 1032)
CAP = 256


@pytest.fixture(scope="module")
def pair():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return Pair(ODD, seed=0, gains="random")


# requests x rows: 1, 15, 16, 17 (a finishing CTA's rows), then one call past
# each padding's lower edge and at 256, 257, 272 and 320 rows (two halves), 323 (256
# and the rest), 353 (two), 391 (256 and the rest), 513, 529 and 544 (three)
@pytest.mark.parametrize("rows", [[1], [15], [16], [17], [17, 16], [17, 17, 15], [16] * 4, [17] * 4, [17] * 6,
                                  [17] * 8, [17] * 10, [17] * 12, [16] * 16, [17] * 15 + [2], [17] * 16,
                                  [17] * 18 + [14], [17] * 19, [17] * 20 + [13], [17] * 23, [17] * 30 + [3],
                                  [17] * 31 + [2], [17] * 32],
                         ids=lambda r: f"{sum(r)}rows")
def test_rows(pair, rows):
    check_rows(pair, rows)


# Few SMs give each CTA enough units for pairs of CTAs: with 2, whole tiles of
# odd counts (gate/up 23, down 3, vocabulary 9), with 4 also tiles of the
# residual projections cut between CTAs.  NB = 64, 96, 192, 256 and 16.  (A
# budget of 1 runs as 2, one of 3 on the groups of 2.)
@pytest.mark.parametrize("sms", [1, 2, 3, 4])
@pytest.mark.parametrize("rows", [[16] * 4, [17] * 4, [17] * 10, [17] * 16], ids=lambda r: f"{sum(r)}rows")
def test_rows_few_sms(rows, sms):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    few = Pair(W.ModelConfig("odd-few", 2, 384, 6, 2, 64, 1472, 1032), seed=0, gains="random")
    few.model.set_sm_budget(sms)
    check_rows(few, rows)


def check_wait_limits(pair, lens, cap, ks):
    """Calls whose kernels' waits run out, at once or somewhere on the way (the
    limits, ns), report it, and leave a state that gives the same bits again."""
    import paper_2609_37617_gb300 as lib
    rng = np.random.default_rng(len(lens))
    roots = [int(x) for x in rng.integers(0, pair.cfg.vocab, size=len(lens))]
    cands = [[int(t) for t in rng.integers(0, pair.cfg.vocab, size=k)] for k in ks]
    st = pair.state(lens, cap, roots)
    want = run_gpu_block(st, pair.cfg, cands)
    st.check()
    st.rollback(lens, roots)
    for limit in (0, 500, 1000, 2000, 4000, 8000, 16000, 32000):
        st.set_wait_limit(limit)
        for _ in range(4):
            run_gpu_block(st, pair.cfg, cands, want_logits=False)
            st.rollback(lens, roots)
        try:
            st.check()
            assert limit > 0, "a limit of 0 runs out"
        except lib.AS2DError as e:
            assert e.status == lib.AS2D_ERR_DEVICE and "timed out" in str(e)
        st.set_wait_limit(2_000_000_000)
        st.rollback(lens, roots)
        for a, b in zip(run_gpu_block(st, pair.cfg, cands), want):
            assert np.array_equal(a, b)
        st.check()
        st.rollback(lens, roots)
    st.close()


# pairs of CTAs with one accumulator and with two, whole and split tiles
@pytest.mark.parametrize("sms", [2, 4, 32])
@pytest.mark.parametrize("rows", [[16] * 4, [17] * 6, [17] * 10, [17] * 16], ids=lambda r: f"{sum(r)}rows")
def test_wait_limits_pairs(rows, sms):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    few = Pair(W.ModelConfig("odd-few", 2, 384, 6, 2, 64, 1472, 1032), seed=0, gains="random")
    few.model.set_sm_budget(sms)
    check_wait_limits(few, [int(x) for x in np.random.default_rng(0).integers(1, CAP - 20, size=len(rows))], CAP,
                      [r - 1 for r in rows])


# The embedding's 14 columns a thread in one batch (1792) and one more (1920).
@pytest.mark.parametrize("hidden", [1792, 1920])
def test_rows_embed_batches(hidden):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    check_rows(Pair(W.ModelConfig("odd-embed", 1, hidden, hidden // 64, 2, 64, 448, 1032), seed=0, gains="random"),
               [4, 1, 3])


def check_rows(pair, rows):
    cfg, n = pair.cfg, len(rows)
    rng = np.random.default_rng(sum(rows))
    lens = [int(x) for x in rng.integers(1, CAP - 20, size=n)]
    roots = [int(x) for x in rng.integers(0, cfg.vocab, size=n)]
    cands = [[int(t) for t in rng.integers(0, cfg.vocab, size=r - 1)] for r in rows]
    st = pair.state(lens, CAP, roots)
    acc, corr, greedy, logits = run_gpu_block(st, cfg, cands)
    st.check()
    kc, vc = st.kc.clone(), st.vc.clone()
    st.close()
    oc = pair.oracle_cache(lens[0], CAP)
    want = pair.oracle.verify_block(oc, lens[0], roots[0], cands[0])
    assert np.max(np.abs(want["logits"] - logits[:rows[0]])) <= LOGIT_TOL
    at = 0
    for b in range(n):
        one = pair.state([lens[b]], CAP, [roots[b]])
        # the request's own prefix (positions below its length)
        one.kc[:, 0, :, :lens[b]] = kc[:, b, :, :lens[b]]
        one.vc[:, 0, :, :lens[b]] = vc[:, b, :, :lens[b]]
        a1, c1, g1, l1 = run_gpu_block(one, cfg, [cands[b]])
        assert np.array_equal(l1, logits[at:at + rows[b]]), f"request {b}"
        assert a1[0] == acc[b] and c1[0] == corr[b] and np.array_equal(g1, greedy[at:at + rows[b]])
        one.close()
        at += rows[b]


# one chunk, two chunks in a cluster of 16 (or through memory), more chunks,
# lengths around the 128-key tiles and 1024-key chunks, one and two query
# tiles; together a launch of four CTAs per SM
LAYOUT_LENS = [1, 126, 127, 128, 129, 1015, 1023, 1024, 1025, 2030, 2047, 2049, 3000]
LAYOUT_KS = [0, 1, 16, 0, 3, 9, 0, 16, 2, 16, 0, 8, 12]
# with requests of more than four chunks: their partials folded by a kernel of
# their own (17 chunks: two rounds of its loads)
LONG_LENS = [4080, 4097, 127, 5000, 1024, 6143, 6145, 16500]
LONG_KS = [16, 0, 9, 16, 3, 1, 16, 12]


@pytest.mark.parametrize("d,lens,ks", [(64, LAYOUT_LENS, LAYOUT_KS), (128, LAYOUT_LENS, LAYOUT_KS),
                                       (64, LONG_LENS, LONG_KS), (128, LONG_LENS, LONG_KS)],
                         ids=["d64", "d128", "d64-long", "d128-long"])
def test_attention_layouts(d, lens, ks):
    """Every request of a large launch equals the same request alone (another
    layout of the attention) bit for bit, and the oracle."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cfg = W.ModelConfig(f"d{d}", 1, 256, 8, 2, d, 448, 1032)
    pair = Pair(cfg, seed=0)
    distinct, lens, ks = len(lens), lens * 2, ks * 2
    cap, n = max(lens) + 32, len(lens)
    rng = np.random.default_rng(d)
    roots = [int(x) for x in rng.integers(0, cfg.vocab, size=n)]
    cands = [[int(t) for t in rng.integers(0, cfg.vocab, size=k)] for k in ks]
    st = pair.state(lens, cap, roots)
    logits = run_gpu_block(st, cfg, cands)[3]
    st.check()
    kc, vc = st.kc.clone(), st.vc.clone()
    st.close()
    at = 0
    for b in range(distinct):
        one = pair.state([lens[b]], cap, [roots[b]])
        one.kc[:, 0, :, :lens[b]] = kc[:, b, :, :lens[b]]
        one.vc[:, 0, :, :lens[b]] = vc[:, b, :, :lens[b]]
        rows = logits[at:at + ks[b] + 1]
        assert np.array_equal(run_gpu_block(one, cfg, [cands[b]])[3], rows), f"length {lens[b]}"
        one.close()
        want = pair.oracle.verify_block(pair.oracle_cache(lens[b], cap, req=b), lens[b], roots[b], cands[b])
        assert np.max(np.abs(want["logits"] - rows)) <= LOGIT_TOL, f"length {lens[b]}"
        at += ks[b] + 1


# three CTAs per SM (17 requests of a chunk: 34 clusters), four, four with the fold kernel
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens", [[1015] * 17, LAYOUT_LENS * 2, LONG_LENS], ids=["three", "four", "fold"])
def test_wait_limits_attention(d, lens):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    check_wait_limits(Pair(W.ModelConfig(f"d{d}", 1, 256, 8, 2, d, 448, 1032), seed=0), lens, max(lens) + 32,
                      [3 + i % 5 for i in range(len(lens))])
