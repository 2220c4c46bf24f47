"""Frames that hold NaN or infinity: they belong to their own utterance only.  An utterance's N best does not change because
another utterance of its batch, or of an earlier call on the same handle, had such frames."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu


def _model(act="tanh", J=64, H=72):
    return tw_synth.make_model(tw_synth.WorkloadConfig("nonfinite", 4, 30, (7, 30), 64, "lstm", H, 1, H, J, 256, 3.0, 4, (3,), "bf16", 11, act))


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("S,short", [(1, 1), (2, 1), (3, 2), (4, 1), (5, 3), (7, 2), (8, 3), (9, 4), (10, 1), (13, 5), (20, 6), (32, 31)])
def test_nan_frames_stay_with_their_utterance(mode, S, short):
    """The short last segment's padding frames have operand rows too, which the joiner's sums meet with a factor of 0."""
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = _model()
    N, B, T = 4, 8, 2 * S + short
    dec, fresh = (TwDecoder(weights_from_synth(m), N=N, S=S, mode=mode, max_batch=B, max_T=T) for _ in range(2))
    rng = np.random.default_rng(S)
    good = tw_synth.round_to_bf16(rng.standard_normal((B, T, 64)).astype(np.float32))
    bad = np.full((B, T, 64), np.nan, np.float32)
    lens = np.full(B, short, np.int32)
    lens[::2] += S                                       # half of them with a whole segment ahead of the short one
    want = [x.cpu().numpy() for x in fresh.decode(good, lens)[:4]]
    assert np.all(want[1][:, 0] >= 0) and np.all(np.isfinite(want[2]))
    dec.decode(bad, np.full(B, T, np.int32))             # leaves NaN in every operand row that it used
    for got, ref in zip(dec.decode(good, lens)[:4], want):
        np.testing.assert_array_equal(got.cpu().numpy(), ref)
    mixed, mixed_lens = good.copy(), lens.copy()
    mixed[::3], mixed_lens[::3] = np.nan, T
    for _ in range(2):
        for got, ref in zip(dec.decode(mixed, mixed_lens)[:4], want):
            for b in set(range(B)) - set(range(0, B, 3)):
                np.testing.assert_array_equal(got.cpu().numpy()[b], ref[b])


@pytest.mark.parametrize("D,rows", [(36, 40), (200, 3000), (204, 3000), (484, 3000), (256, 3000), (202, 300)])
def test_an_infinite_element_stays_infinite_in_the_fp32_projection(D, rows):
    """Row r of the frames has one infinite element, at column r mod D: every product with it is +-infinity and so is the sum,
    whatever the length of the last block of K (D a multiple of 32, of 4, of 2)."""
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    cfg = tw_synth.WorkloadConfig("inf", 4, 30, (7, 30), D, "stateless", 24, 0, 0, 48, 64, 3.0, 4, (3,), "f32", 11)
    m = tw_synth.make_model(cfg)
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, mode=0, max_batch=1, max_T=3)
    x = np.random.default_rng(D).standard_normal((rows, D)).astype(np.float32)
    r = np.arange(rows)
    x[r, r % D] = np.where(r % 2, np.inf, -np.inf)
    got = dec.project_encoder(x).cpu().numpy()
    np.testing.assert_array_equal(got, np.where(r % 2, 1.0, -1.0)[:, None] * np.sign(m.W_e[:, r % D].T) * np.inf)
