"""Tokens whose probabilities are a few ulps of float32 apart: the in-kernel selection takes logarithms that may be equal or in the
other order, within a row and between rows.  Which of such tokens is kept is a matter of rounding; how many there are, how long the
sequences are and what the best one scores is not."""
import numpy as np
import pytest

import tw_synth
from helpers import nbest_from_arrays, oracle_model
from oracle import token_wise_search as tws
from oracle.exact_forward import forward_log_prob

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tied", [12, 255])          # within the survivors that are ranked directly, and past them
@pytest.mark.parametrize("N,S", [(4, 3), (10, 2), (5, 1), (16, 4)])
def test_near_ties_within_and_between_rows(N, S, tied):
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    cfg = tw_synth.WorkloadConfig("ties", 4, 9, (1, 9), 64, "lstm", 64, 1, 64, 64, 256, 3.0, N, (S,), "bf16", 3)
    m = tw_synth.make_model(cfg)
    rng = np.random.default_rng(N + tied)
    m.W_out[:] = 0.0
    m.b_out[:] = 1.0 + rng.integers(0, 4, 256) * 2.0 ** -23
    m.b_out[1 + tied:] = -5.0
    m.b_out[0] = 3.0
    enc, _ = tw_synth.make_encoder_batch(cfg)
    lens = np.array([9, 4, 1, 7], dtype=np.int32)
    dec = TwDecoder(weights_from_synth(m), N=N, S=S, mode=MODE_BF16, max_batch=4, max_T=9, max_iters_per_segment=6)
    assert dec.set_fused(True)
    tokens, olens, scores, status = [x.cpu().numpy() for x in dec.decode(enc, lens)[:4]]
    om = oracle_model(m)
    for b in range(4):
        ref, st = tws.token_wise_beam_search(om, enc[b, :lens[b]].astype(np.float64), N, S, max_iters=6)
        got = nbest_from_arrays(tokens, olens, scores, b)
        assert len(set(t for t, _ in got)) == len(ref) == len(got)
        assert all(1 <= k <= tied for t, _ in got for k in t)
        assert [len(t) for t, _ in got] == [len(t) for t, _ in ref]
        # One segment of one frame: the scores too.  Over more, which of the near ties survive decides what later passes add to them
        # (the oracle's own scores behind the first one differ by up to 1.1 where its log-probabilities are disturbed by 2e-7): no
        # sequence scores more than its exact probability.  2e-3: the approximate exponentials and logarithms of up to nine
        # frames, as in the test of exact ties.
        s = np.array([x for _, x in got])
        assert (np.diff(s) <= 0).all()
        np.testing.assert_allclose(s[0], ref[0][1], atol=2e-3)
        if lens[b] == 1:
            np.testing.assert_allclose(s, [x for _, x in ref], atol=2e-3)
        for t, x in got:
            assert x <= forward_log_prob(om, enc[b, :lens[b]].astype(np.float64), t) + 2e-3
        assert status[b] == (4 if st.limit_hit else 0)
    dec.close()
