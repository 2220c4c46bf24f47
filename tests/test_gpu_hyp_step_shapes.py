"""hyp_step_kernel where its work does not fit one round of its warps, or one early fetch: rows of more than 1024 values, more rows
or dot products than warps, one hypothesis, a slot ring of its smallest length, a pass cap and a token capacity that are hit."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,layers,J,N,S,max_iters,max_tokens", [
    (1088, 1, 1096, 4, 3, 0, 0),       # the parents' h and the carried operand rows past the early 1024 columns
    (64, 3, 64, 16, 7, 0, 0),          # 48 rows of h, 112 operand rows and dot products for 32 warps
    (64, 2, 72, 1, 1, 0, 0),
    (72, 1, 64, 16, 2, 1, 0),          # a ring of 2 N slots, all but N of them wanted in every segment
    (64, 1, 64, 5, 3, 2, 0),           # the pass cap drops what is left of a segment
    (64, 1, 64, 5, 3, 0, 1),           # sequences that may not grow any more
])
def test_decode_does_not_depend_on_the_route(H, layers, J, N, S, max_iters, max_tokens):
    """The default step against the one whose rows are gathered and numbered by other kernels: the same products in the same
    order, so the same N best, bit by bit."""
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    cfg = tw_synth.WorkloadConfig("shapes", 5, 17, (1, 17), 64, "lstm", H, layers, H, J, 512, -2.0 if max_tokens else 0.5, N, (S,), "bf16", 5)
    m = tw_synth.make_model(cfg)
    rng = np.random.default_rng(N * S)
    lens = np.array([17, 9, 1, 0, 16], dtype=np.int32)
    enc = tw_synth.round_to_bf16(rng.standard_normal((5, 17, cfg.D_enc)).astype(np.float32))
    dec = TwDecoder(weights_from_synth(m), N=N, S=S, mode=MODE_BF16, max_batch=5, max_T=17, max_iters_per_segment=max_iters, max_tokens=max_tokens)
    got = []
    for inline in (True, False):
        dec.set_inline_gather(inline)
        got.append([t.cpu().numpy() for t in dec.decode(enc, lens)[:4]])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
    tokens, n, scores, status = got[0]
    assert (n.max(axis=1) >= 0).all() and np.isfinite(scores[n >= 0]).all()
    if max_tokens:
        assert n.max() <= max_tokens and (status == 4).any()        # TW_ERR_LIMIT
    if max_iters:
        assert (status == 4).any()
