"""What a bounded wait that gave up leaves behind (its error word, put there by the tests' hooks; no wait runs out here): the
call that reports it, and the calls after it, which must not suffer from it."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu
TIMEOUT = 6


def _decoder(mode, B=3, T=14):
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = tw_synth.make_model(tw_synth.WorkloadConfig("words", 4, 30, (7, 30), 64, "lstm", 72, 2, 72, 64, 256, 3.0, 4, (3,), "f32", 11))
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, mode=mode, max_batch=B, max_T=T)
    enc = np.random.default_rng(1).standard_normal((B, T, 64)).astype(np.float32)
    return m, dec, enc, np.array([T, 5, T - 1][:B], np.int32)


def _timeout(call, *args):
    from paper_2302_14357_b200.binding import TwError
    with pytest.raises(TwError) as e:
        call(*args)
    assert e.value.status == TIMEOUT


@pytest.mark.parametrize("mode", [0, 1])
def test_stage_calls_report_it_once(mode):
    m, dec, enc, lens = _decoder(mode)
    R = 12
    rng = np.random.default_rng(2)
    state = np.tanh(rng.standard_normal((R, 2, 2, 72))).astype(np.float32)
    tok = rng.integers(0, 256, R).astype(np.int32)
    E = dec.project_encoder(enc[:, :3])
    Pp = dec.predictor_step(tok, state)[1]
    group, sl, ld = np.arange(R, dtype=np.int32) // 4, np.array([3, 2, 3], np.int32), rng.standard_normal((R, 3)).astype(np.float32)
    Es = E.reshape(3, 3, 64)
    decoded = [x.cpu().numpy() for x in dec.decode(enc, lens)[:4]]
    for call, args in ((dec.project_encoder, (enc[:, :3],)), (dec.predictor_step, (tok, state)), (dec.joiner_segment, (Es, Pp, group, sl)),
                       (dec.joiner_expand, (Es, Pp, group, sl, ld))):
        want = call(*args)
        assert dec.lib.tw_test_error_word(dec.h, 1, 1) == 0
        for got, ref in zip(dec.decode(enc, lens)[:4], decoded):          # a decode neither reports nor clears it
            np.testing.assert_array_equal(got.cpu().numpy(), ref)
        _timeout(call, *args)
        got = call(*args)
        for x, y in zip(got, want) if isinstance(got, tuple) else ((got, want),):
            np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("mode", [0, 1])
def test_a_session_reports_it_to_its_end(mode, graph):
    m, dec, enc, lens = _decoder(mode)
    dec.set_graph(graph)
    want = [x.cpu().numpy() for x in dec.decode(enc, lens)[:4]]
    seven = np.array([7, 5, 7], np.int32)
    dec.stream_open(3)
    dec.stream_push(enc[:, :7].copy(), seven)
    assert dec.lib.tw_test_error_word(dec.h, 0, 1) == 0
    _timeout(dec.stream_push, enc[:, 7:].copy(), lens - seven)
    _timeout(dec.stream_nbest)
    _timeout(dec.stream_close)
    dec.stream_open(3)                                                     # the next one starts afresh
    dec.stream_push(enc[:, :7].copy(), seven)
    dec.stream_push(enc[:, 7:].copy(), lens - seven)
    dec.stream_nbest()
    for got, ref in zip(dec.stream_close()[:4], want):
        np.testing.assert_array_equal(got.cpu().numpy(), ref)
    assert dec.lib.tw_test_error_word(dec.h, 0, 1) == 0                    # and so does a decode
    for got, ref in zip(dec.decode(enc, lens)[:4], want):
        np.testing.assert_array_equal(got.cpu().numpy(), ref)


def test_noalloc_call_starts_with_a_clear_word():
    import torch
    from paper_2302_14357_b200 import binding
    m, dec, enc, lens = _decoder(0)
    W_out, b_out = torch.from_numpy(m.W_out).cuda(), torch.from_numpy(m.b_out).cuda()
    rng = np.random.default_rng(3)
    E, Pp = torch.from_numpy(rng.standard_normal((2, 3, 64)).astype(np.float32)).cuda(), torch.from_numpy(rng.standard_normal((9, 64)).astype(np.float32)).cuda()
    group, ld = torch.arange(9, dtype=torch.int32, device="cuda") // 5, torch.zeros((9, 3), device="cuda")
    call = lambda: binding.joiner_expand_noalloc(W_out, b_out, 3, 0, E, Pp, group, None, ld)      # noqa: E731
    want = call()
    assert want[0] == 0 and dec.lib.tw_test_noalloc_word(1) == 0
    got = call()
    assert got[0] == 0 and dec.lib.tw_test_noalloc_word(0) == 0
    for x, y in zip(got[1:], want[1:]):
        assert torch.equal(x, y)
