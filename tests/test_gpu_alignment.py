"""Stage calls on buffers that start on a 4-byte boundary only (rows of a larger array, say): what they return for aligned ones."""
import numpy as np
import pytest

import tw_synth

pytestmark = pytest.mark.gpu
BF16_STAGE_TOL = 2e-2


@pytest.mark.parametrize("V", [256, 300])
@pytest.mark.parametrize("mode,S", [(0, 3), (1, 1), (1, 3), (1, 6), (1, 10), (1, 20), (1, 40)])
def test_joiner_expand(mode, S, V):
    import torch
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = tw_synth.make_model(tw_synth.WorkloadConfig("align", 4, 30, (7, 30), 64, "stateless", 24, 0, 0, 64, V, 3.0, 4, (3,), "bf16", 11))
    R, G = 24, 6
    dec = TwDecoder(weights_from_synth(m), N=4, S=S, mode=mode, max_batch=G, max_T=S)
    gen = torch.Generator(device="cuda").manual_seed(S)

    def off(n, *shape):                                    # a tensor n floats past a 256-byte boundary
        return torch.randn(int(np.prod(shape)) + 4, device="cuda", generator=gen)[n:n + int(np.prod(shape))].view(shape)
    group = torch.arange(R, device="cuda", dtype=torch.int32) // 4
    sl = torch.randint(1, S + 1, (G,), device="cuda", generator=gen, dtype=torch.int32)
    for shift in ((1, 0, 0), (0, 3, 0), (0, 0, 1), (2, 2, 2)):
        E, Pp, ld = off(shift[0], G, S, 64), off(shift[1], R, 64), off(1, R, S)
        want = dec.joiner_expand(E.clone(), Pp.clone(), group, sl, ld.clone())
        phi, nb, la = off(1, R), off(shift[2], R, V), off(3, R, S)
        rc = dec.lib.tw_joiner_expand(dec.h, E.data_ptr(), Pp.data_ptr(), group.data_ptr(), sl.data_ptr(), ld.data_ptr(), G, R,
                                      phi.data_ptr(), nb.data_ptr(), la.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0
        for got, ref in zip((phi, nb, la), want):
            inf = torch.isinf(ref)
            assert torch.equal(torch.isinf(got), inf)
            assert (got[~inf] - ref[~inf]).abs().max() < (BF16_STAGE_TOL if mode else 1e-5)


@pytest.mark.parametrize("mode", [0, 1])
def test_predictor_step(mode):
    import torch
    from paper_2302_14357_b200.binding import TwDecoder, weights_from_synth
    m = tw_synth.make_model(tw_synth.WorkloadConfig("align", 4, 30, (7, 30), 64, "lstm", 72, 2, 72, 64, 256, 3.0, 4, (3,), "bf16", 11))
    R = 24
    dec = TwDecoder(weights_from_synth(m), N=4, S=3, mode=mode, max_batch=6, max_T=3)
    state = torch.tanh(torch.randn(R * 2 * 2 * 72 + 4, device="cuda"))[1:-3].view(R, 2, 2, 72)
    tok = torch.arange(R, device="cuda", dtype=torch.int32)
    want, want_Pp = dec.predictor_step(tok, state.clone())
    tol = BF16_STAGE_TOL if mode else 2e-5  # other kernels, sums in another order
    for shift in (0, 1):
        out = torch.zeros(state.numel() + 4, device="cuda")[shift:shift + state.numel()].view_as(state)
        Pp = torch.zeros(R * 64 + 4, device="cuda")[1:-3].view(R, 64)
        rc = dec.lib.tw_predictor_step(dec.h, tok.data_ptr(), state.data_ptr(), R, out.data_ptr(), Pp.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        assert rc == 0 and (out - want).abs().max() <= tol and (Pp - want_Pp).abs().max() <= tol
