"""hyp_step_kernel where its work does not fit one round of its warps, or one early fetch: rows of more than 1024 values, more rows
or dot products than warps, one hypothesis, slot rings longer and shorter than the 32 slots that are looked at ahead, a pass cap and
a token capacity that are hit."""
import numpy as np
import pytest

import tw_synth
from helpers import nbest_from_arrays, oracle_model
from oracle import token_wise_search as tws
from oracle.exact_forward import forward_log_prob

pytestmark = pytest.mark.gpu

LENS = np.array([17, 9, 1, 0, 16], dtype=np.int32)

SHAPES = [                             # (the ring of an utterance has N (max_iters + 1) slots)
    (1088, 1, 1096, 4, 3, 0, 0),       # the parents' h and the carried operand rows past the early 1024 columns
    (64, 3, 64, 16, 7, 0, 0),          # 48 rows of h, 112 operand rows and dot products for 32 warps
    (64, 2, 72, 1, 1, 0, 0),
    (72, 1, 64, 16, 2, 1, 0),          # one pass a segment: nothing is ever kept
    (72, 1, 64, 16, 2, 2, 0),          # a ring of 48, of which up to 16 slots are carried and 16 taken in every segment
    (64, 1, 64, 5, 3, 2, 0),           # a ring of 15, and the pass cap drops what is left of a segment
    (64, 1, 64, 4, 1, 2, 0),           # a ring of 12, started over 17 times
    (64, 1, 64, 5, 3, 0, 1),           # sequences that may not grow any more
]


def _decode(H, layers, J, N, S, max_iters, max_tokens, sharp):
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    cfg = tw_synth.WorkloadConfig("shapes", 5, 17, (1, 17), 64, "lstm", H, layers, H, J, 512, -2.0 if max_tokens else 0.5, N, (S,), "bf16", 5)
    m = tw_synth.make_model(cfg)
    if sharp:
        m.W_out *= 4.0                 # a power of two: still bf16 values
        m.b_out[0] = 8.0
    rng = np.random.default_rng(N * S)
    enc = tw_synth.round_to_bf16(rng.standard_normal((5, 17, cfg.D_enc)).astype(np.float32))
    dec = TwDecoder(weights_from_synth(m), N=N, S=S, mode=MODE_BF16, max_batch=5, max_T=17, max_iters_per_segment=max_iters, max_tokens=max_tokens)
    got = []
    for inline in (True, False):
        dec.set_inline_gather(inline)
        got.append([t.cpu().numpy() for t in dec.decode(enc, LENS)[:4]])
    return m, enc, got


@pytest.mark.parametrize("H,layers,J,N,S,max_iters,max_tokens", SHAPES)
def test_decode_does_not_depend_on_the_route(H, layers, J, N, S, max_iters, max_tokens):
    """The default step against the one whose rows are gathered and numbered by other kernels: the same products in the same
    order, so the same N best, bit by bit.  (Both rank and take slots in the same way: for that see the next test.)"""
    _, _, got = _decode(H, layers, J, N, S, max_iters, max_tokens, False)
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
    tokens, n, scores, status = got[0]
    assert (n.max(axis=1) >= 0).all() and np.isfinite(scores[n >= 0]).all()
    if max_tokens:
        assert n.max() <= max_tokens and (status == 4).any()        # TW_ERR_LIMIT
    if max_iters:
        assert (status == 4).any()


@pytest.mark.parametrize("sharp", [False, True])
@pytest.mark.parametrize("H,layers,J,N,S,max_iters,max_tokens", [s for s in SHAPES if s[6] == 0])
def test_decode_against_the_oracle(H, layers, J, N, S, max_iters, max_tokens, sharp):
    """Ranks, threshold, slots: the oracle's best sequence and its score to 0.05, as in the other bf16 tests, for all utterances but
    at most one (near-ties); N sequences like the oracle's, distinct, in the order of their scores, none above its exact probability."""
    m, enc, got = _decode(H, layers, J, N, S, max_iters, max_tokens, sharp)
    tokens, n, scores, status = got[0]
    om = oracle_model(m)
    agree, longest = [], 0
    for b in np.flatnonzero(LENS):
        frames = enc[b, :LENS[b]].astype(np.float64)
        ref, _ = tws.token_wise_beam_search(om, frames, N, S, max_iters=max_iters or 4 * S + 16)
        nbest = nbest_from_arrays(tokens, n, scores, b)
        assert len(set(t for t, _ in nbest)) == len(nbest) == len(ref)
        assert all(1 <= k < 512 for t, _ in nbest for k in t)
        assert (np.diff([s for _, s in nbest]) <= 0).all()
        for t, s in nbest:
            assert s <= forward_log_prob(om, frames, t) + 0.05
        agree.append(nbest[0][0] == ref[0][0] and abs(nbest[0][1] - ref[0][1]) < 0.05)
        longest = max(longest, max(len(t) for t, _ in nbest))
    assert sum(agree) >= len(agree) - 1
    assert longest == 0 if max_iters == 1 or N == 1 else longest > 0
