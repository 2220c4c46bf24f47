"""The fp32 GEMM at the edges of its tiles (16 rows, 256 or 64 columns, K blocks of 32), with K whole, split between two
and between four CTAs, one and two operand pairs, and with rows that allow no 16-byte copies, against float64.

Bound: a product of length K summed in fp32 in any order is off by at most K 2^-24 sum |a b|; with operands of size 1
and 1/sqrt(K) the sums of |a b| are below sqrt(K), and rounding errors of random sign stay below sqrt(K) 2^-24 times that,
K 2^-24: 7e-5 at K = 1200.  The tanh joiner adds its own 2 ulp, the cell its sigmoids: well inside the same figure."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu


def _cfg(D, H, J, V, layers):
    return tw_synth.WorkloadConfig("gemm", 4, 30, (30, 30), D, "lstm", H, layers, H, J, V, 2.0, 4, (3,), "f32", 5)


@pytest.mark.parametrize("R", [1, 16, 17, 160])
@pytest.mark.parametrize("H,J,V", [(600, 640, 1030), (36, 48, 64), (130, 250, 65), (33, 31, 300)])
def test_predictor_and_joiner_match_float64(R, H, J, V):
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    cfg = _cfg(40, H, J, V, 2)
    m = tw_synth.make_model(cfg)
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, mode=0, max_batch=(R + 3) // 4, max_T=3)
    rng = np.random.default_rng(R)
    tok = rng.integers(0, V, R).astype(np.int32)
    state = rng.standard_normal((R, 2, 2, H)).astype(np.float32)
    out, Pp = (t.cpu().numpy().astype(np.float64) for t in dec.predictor_step(tok, state))
    sig = lambda x: 1.0 / (1.0 + np.exp(-x))                                        # noqa: E731
    x, tol = m.emb[tok].astype(np.float64), 2 * H * 2.0 ** -24 + 2e-6
    for l in range(2):
        g = x @ m.lstm_W_ih[l].astype(np.float64).T + state[:, l, 0].astype(np.float64) @ m.lstm_W_hh[l].astype(np.float64).T
        i, f, c, o = (g[:, k * H:(k + 1) * H] for k in range(4))
        cn = sig(f) * state[:, l, 1] + sig(i) * np.tanh(c)
        x = sig(o) * np.tanh(cn)
        assert np.abs(out[:, l, 1] - cn).max() < tol and np.abs(out[:, l, 0] - x).max() < tol
    assert np.abs(Pp - x @ m.W_p.astype(np.float64).T).max() < 2 * tol
    E = rng.standard_normal((1, 3, J)).astype(np.float32)
    P32 = Pp.astype(np.float32)
    got = dec.joiner_segment(E, P32, np.zeros(R, np.int32), [2]).cpu().numpy().astype(np.float64)
    z = np.tanh(E[0, None, :2].astype(np.float64) + P32[:, None].astype(np.float64)) @ m.W_out.astype(np.float64).T + m.b_out
    ref = z - np.log(np.exp(z).sum(-1, keepdims=True))
    assert np.abs(got[:, :2] - ref).max() < 2 * J * 2.0 ** -24 + 1e-5
    assert np.all(got[:, 2, 0] == 0.0) and np.all(np.isneginf(got[:, 2, 1:]))
