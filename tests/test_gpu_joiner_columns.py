"""The fused joiner's column count per CTA follows the batch size; an utterance's result does not.

W_out = 0 makes every logit its bias: 0.5 for blank, 0 for token 1, and -39.875 for the others, too little to change a float32 sum.
Every sum over the vocabulary is then one addition, whatever the columns are split into, and 39.875 is the bound that is taken off the
logits: its product with log2(e) is 1.8e-6 from its rounding, about as far as it can be.  A normaliser that adds another product than
was taken off drifts by that difference with every token.
"""
import numpy as np
import pytest

import tw_synth
from helpers import nbest_from_arrays, oracle_model
from oracle import token_wise_search as tws

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norm", ["softmax", "hat"])
@pytest.mark.parametrize("S", [2, 3, 5, 10])
def test_scores_do_not_depend_on_the_columns_per_cta(S, norm):
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    N, T, V = 8, 40, 1024
    cfg = tw_synth.WorkloadConfig("columns", 1, T, (T, T), 64, "lstm", 64, 1, 64, 64, V, 3.0, N, (S,), "bf16", 11, joiner_norm=norm)
    m = tw_synth.make_model(cfg)
    m.W_out[:] = 0.0
    m.b_out[:] = -39.875
    m.b_out[:2] = 0.5, 0.0
    enc, _ = tw_synth.make_encoder_batch(cfg)
    per_tile = 4 * (32 // S)                               # hypotheses in a tile of 128 rows
    results = []
    for tiles in (1, 12, 24):                              # rows for 64, 128 and 256 columns per CTA at V = 1024
        B = (tiles * per_tile + N - 1) // N
        dec = TwDecoder(weights_from_synth(m), N=N, S=S, mode=MODE_BF16, max_batch=B, max_T=T)
        assert dec.set_fused(True)
        out = [x.cpu().numpy() for x in dec.decode(np.repeat(enc[:1], B, axis=0), np.full(B, T, dtype=np.int32))[:4]]
        dec.close()
        assert (out[3] == 0).all()
        for x in out[:3]:
            assert (x == x[:1]).all()                      # every utterance is the same one
        results.append(nbest_from_arrays(out[0], out[1], out[2], 0))
    assert results[0] == results[1] == results[2]          # tokens and scores, to the last bit
    ref, st = tws.token_wise_beam_search(oracle_model(m), enc[0].astype(np.float64), N, S, max_iters=4 * S + 16)
    assert not st.limit_hit
    assert [t for t, _ in results[0]] == [t for t, _ in ref]
    # the approximate exponentials and logarithms of up to some 80 passes, 2e-6 each
    np.testing.assert_allclose([s for _, s in results[0]], [s for _, s in ref], rtol=0, atol=2e-4)
