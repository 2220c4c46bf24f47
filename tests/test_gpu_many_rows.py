"""TW_MODE_F32 above 65535 row tiles of the fp32 GEMM (1,048,560 rows): the encoder projection, a whole batch and the joiner."""
import numpy as np
import pytest

import tw_synth
from oracle import rnnt_model as rm
from oracle import segment_math as sm
from helpers import oracle_model

pytestmark = pytest.mark.gpu
TOL = 1e-5                                       # sums of four fp32 products and Eq. 3-7 over 64 frames, relative to the value


def _model(S):
    return tw_synth.make_model(tw_synth.WorkloadConfig("rows", 4, 30, (7, 30), 4, "stateless", 4, 0, 0, 4, 17, 2.0, 4, (S,), "f32", 3))


@pytest.mark.parametrize("rows", [1048560, 1048561, 1048609])
def test_projection(rows):
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = _model(3)
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, max_batch=1, max_T=3)
    x = np.random.default_rng(1).standard_normal((rows, 4)).astype(np.float32)
    got = dec.project_encoder(x).cpu().numpy()
    np.testing.assert_allclose(got, x.astype(np.float64) @ m.W_e.T.astype(np.float64), rtol=0, atol=TOL)


def test_decode_of_a_batch_with_many_frames():
    """1,050 utterances of room for 1,000 frames, three frames long: as the same batch without the room."""
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = _model(3)
    B, T, t = 1050, 1000, 3
    dec = TwDecoder(weights_from_synth(m), N=2, S=3, max_batch=B, max_T=T, max_tokens=16)
    dec.set_lanes(False)
    enc = np.zeros((B, T, 4), np.float32)
    enc[:, :t] = np.random.default_rng(2).standard_normal((B, t, 4))
    lens = np.full(B, t, np.int32)
    want = [x.cpu().numpy() for x in dec.decode(enc[:, :t], lens)[:4]]
    for got, ref in zip(dec.decode(enc, lens)[:4], want):
        np.testing.assert_array_equal(got.cpu().numpy(), ref)


def test_joiner_expand():
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    S, N, G = 64, 16, 1025
    m, R = _model(S), N * G
    dec = TwDecoder(weights_from_synth(m), N=N, S=S, max_batch=G, max_T=S, max_tokens=4)
    rng = np.random.default_rng(3)
    enc = rng.standard_normal((G, S, 4)).astype(np.float32)
    pred = rng.standard_normal((R, 4)).astype(np.float32)
    ld = (rng.standard_normal((R, S)) - 2).astype(np.float32)
    group = (np.arange(R) // N).astype(np.int32)
    om = oracle_model(m)
    E = dec.project_encoder(enc.reshape(-1, 4)).reshape(G, S, 4)
    Pp = (pred.astype(np.float64) @ om.W_p.T).astype(np.float32)
    phi, nb, la = (x.cpu().numpy().astype(np.float64) for x in dec.joiner_expand(E, Pp, group, np.full(G, S, np.int32), ld))
    for r in (0, 1, 8192, 16382, 16383, 16384, R - 1):          # row 16383's frames end at GEMM row 1,048,575
        lj = rm.joiner_log_probs(om, enc[group[r]], pred[r:r + 1])
        d0 = ld[r:r + 1].astype(np.float64)
        lBl = sm.blank_product(lj)
        ldt = sm.nonblank_expansion_t(lj, lBl, d0)
        scale = np.abs(la[r]).max()
        np.testing.assert_allclose(phi[r], sm.blank_expansion(lBl, d0)[0], rtol=0, atol=TOL * scale)
        np.testing.assert_allclose(nb[r, 1:], sm.nonblank_expansion(ldt)[0, 1:], rtol=0, atol=TOL * scale)
