"""The gate GEMM's small instance (one or two row tiles, lane quarters without rows not fetched, one or two 32-column chunks
per CTA) at the edges of its quarters and tiles, and whole decodes of batches whose steps use it, with finished utterances
(steps without rows) and more than one layer."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu
# operands rounded to bf16 (2^-9 of each product, random signs: 2^-9 of the gate), approximate tanh 2^-11: the stage tolerance
TOL = 2e-2


def _cfg(H, layers, J=640, V=256):
    return tw_synth.WorkloadConfig("small", 4, 30, (7, 30), 64, "lstm", H, layers, H, J, V, 3.0, 4, (3,), "bf16", 11)


@pytest.mark.parametrize("H,layers", [(640, 1), (512, 3), (72, 2), (1024, 2)])
@pytest.mark.parametrize("R", [1, 32, 33, 128, 129, 256])
def test_predictor_step_matches_float64(R, H, layers):
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    cfg = _cfg(H, layers)
    m = tw_synth.make_model(cfg)
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, mode=MODE_BF16, max_batch=(R + 3) // 4, max_T=3)
    rng = np.random.default_rng(R)
    tok = rng.integers(0, cfg.V, R).astype(np.int32)
    state = np.tanh(rng.standard_normal((R, layers, 2, H))).astype(np.float32)
    out, Pp = (t.cpu().numpy().astype(np.float64) for t in dec.predictor_step(tok, state))
    sig = lambda x: 1.0 / (1.0 + np.exp(-x))                                        # noqa: E731
    x = m.emb[tok].astype(np.float64)
    for l in range(layers):
        g = x @ m.lstm_W_ih[l].astype(np.float64).T + state[:, l, 0].astype(np.float64) @ m.lstm_W_hh[l].astype(np.float64).T
        i, f, c, o = (g[:, k * H:(k + 1) * H] for k in range(4))
        cn = sig(f) * state[:, l, 1] + sig(i) * np.tanh(c)
        x = sig(o) * np.tanh(cn)
        assert np.abs(out[:, l, 1] - cn).max() < TOL and np.abs(out[:, l, 0] - x).max() < TOL
    assert np.abs(Pp - x @ m.W_p.astype(np.float64).T).max() < TOL


@pytest.mark.parametrize("H,layers,S,B", [(640, 1, 3, 1), (512, 3, 5, 33), (72, 2, 1, 9), (640, 2, 7, 20)])
def test_decode_does_not_depend_on_how_the_rows_are_made(H, layers, S, B):
    """The default step (rows claimed by hyp_step_kernel, operand from the projection) against the one with the gather kernel,
    the numbering on a side branch and an operand kernel: the same products in the same order, so the same N best."""
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    cfg = _cfg(H, layers)
    m = tw_synth.make_model(cfg)
    rng = np.random.default_rng(S)
    lens = rng.integers(0, 25, B).astype(np.int32)
    lens[0] = 24
    enc = tw_synth.round_to_bf16(rng.standard_normal((B, 24, cfg.D_enc)).astype(np.float32))
    dec = TwDecoder(weights_from_synth(m), N=5, S=S, mode=MODE_BF16, max_batch=B, max_T=24)
    got = []
    for inline in (True, False, True):
        dec.set_inline_gather(inline)
        got.append([t.cpu().numpy() for t in dec.decode(enc, lens)[:4]])
    for other in got[1:]:
        for a, b in zip(got[0], other):
            np.testing.assert_array_equal(a, b)
