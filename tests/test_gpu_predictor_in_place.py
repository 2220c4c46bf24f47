"""tw_predictor_step with state_out == state_in: the step of separate buffers, and nothing in it that a stream capture forbids
(a stage call allocates nothing, so its first call on a handle may be a captured one)."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,R", [(0, 3), (0, 40), (1, 3), (1, 40)])
def test_in_place_step_in_a_capture(mode, R):
    import torch
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = tw_synth.make_model(tw_synth.WorkloadConfig("inplace", 4, 30, (7, 30), 64, "lstm", 72, 2, 72, 64, 256, 3.0, 4, (3,), "f32", 11))
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, mode=mode, max_batch=(R + 3) // 4, max_T=3)
    rng = np.random.default_rng(R)
    tok = torch.from_numpy(rng.integers(0, 256, R).astype(np.int32)).cuda()
    state = torch.from_numpy(np.tanh(rng.standard_normal((R, 2, 2, 72))).astype(np.float32)).cuda()
    want, want_Pp = dec.predictor_step(tok, state)
    buf, Pp = state.clone(), torch.empty_like(want_Pp)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rc = dec.lib.tw_predictor_step(dec.h, tok.data_ptr(), buf.data_ptr(), R, buf.data_ptr(), Pp.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    for _ in range(2):
        buf.copy_(state)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, want) and torch.equal(Pp, want_Pp)
