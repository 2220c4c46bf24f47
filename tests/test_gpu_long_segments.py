"""Whole bf16 decodes with long segments through the fused joiner: the selection from the chunk maxima that its instances for
S > 10 write (16 or 32 columns a chunk), the operand rows at two hypotheses or one to a warp, the side branch that completes
the new hypotheses, and the gate GEMM's instance that runs beside that branch."""
import numpy as np
import pytest

import tw_synth
from oracle import token_wise_search as tws
from helpers import nbest_from_arrays, oracle_model

pytestmark = pytest.mark.gpu
TOP1_GAP = 0.05     # nats: the stage tolerance of 2e-2 a pass, errors of random sign (as for the short segments)


def _cfg(H, layers, V, J=128, N=5):
    return tw_synth.WorkloadConfig("long", 4, 30, (7, 30), 64, "lstm", H, layers, H, J, V, 3.0, N, (3,), "bf16", 13)


def _decoder(cfg, S, B, T):
    from paper_2302_14357_b200.binding import MODE_BF16, TwDecoder, weights_from_synth
    m = tw_synth.make_model(cfg)
    rng = np.random.default_rng(100 * S + B)
    enc = tw_synth.round_to_bf16(rng.standard_normal((B, T, cfg.D_enc)).astype(np.float32))
    dec = TwDecoder(weights_from_synth(m), N=cfg.N, S=S, mode=MODE_BF16, max_batch=B, max_T=T)
    assert dec.stats()["fused_on"] == 1
    return m, dec, enc, rng


def _against_oracle(m, cfg, S, enc, lens, out, sample):
    om = oracle_model(m)
    agree = 0
    for b in sample:
        ref, _ = tws.token_wise_beam_search(om, enc[b, :lens[b]].astype(np.float64), cfg.N, S, max_iters=4 * S + 16)
        got = nbest_from_arrays(*out[:3], b)
        refd = dict(ref)
        assert got and all(abs(s - refd[t]) < TOP1_GAP for t, s in got[:1] if t in refd)
        agree += got[0][0] == ref[0][0]
    assert agree >= len(sample) - 1, (agree, len(sample))


@pytest.mark.parametrize("B,V", [(5, 256), (42, 256), (42, 501)])
@pytest.mark.parametrize("S", [6, 9, 11, 13, 16, 17, 20, 32])
def test_decode_matches_the_oracle_and_the_staged_kernels(S, B, V):
    cfg = _cfg(72, 1, V)
    T = 2 * S + S // 2
    m, dec, enc, rng = _decoder(cfg, S, B, T)
    lens = rng.integers(0, T + 1, B).astype(np.int32)
    lens[:3] = (T, S, 1)
    fused = [x.cpu().numpy() for x in dec.decode(enc, lens)[:4]]
    assert dec.set_fused(False)
    staged = [x.cpu().numpy() for x in dec.decode(enc, lens)[:4]]
    assert np.all(fused[3] == 0) and fused[0].max() < V
    same = sum(np.array_equal(fused[0][b, 0], staged[0][b, 0]) for b in range(B))
    assert same >= B - max(1, B // 20), (same, B)
    np.testing.assert_allclose(fused[2][:, 0], staged[2][:, 0], rtol=0, atol=TOP1_GAP)
    _against_oracle(m, cfg, S, enc, lens, fused, range(min(B, 6)))


@pytest.mark.parametrize("H,layers,B,S", [(640, 1, 32, 8), (640, 2, 64, 20), (1024, 2, 50, 8), (512, 3, 64, 13), (640, 1, 38, 10),
                                          (640, 1, 88, 8), (512, 1, 115, 10)])
def test_gate_gemm_beside_the_side_branch(H, layers, B, S):
    """Three to nine row tiles (320 to 1150 rows at N = 10), tiles of 64 to 128 gate columns, and lengths that empty whole row
    tiles on the way: with the work list from hyp_step_kernel and from the gather kernel, as a graph and kernel by kernel."""
    cfg = _cfg(H, layers, 256, N=10)
    T = 2 * S + 3
    m, dec, enc, rng = _decoder(cfg, S, B, T)
    lens = np.minimum(rng.integers(0, T + 1, B), rng.integers(0, 2 * T, B)).astype(np.int32)
    lens[:2] = (T, S + 1)
    out = []
    for graph, inline in ((True, True), (False, True), (True, False), (True, True)):
        dec.set_graph(graph)
        dec.set_inline_gather(inline)
        out.append([x.cpu().numpy() for x in dec.decode(enc, lens)[:4]])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)
    assert np.all(out[0][3] == 0)
    _against_oracle(m, cfg, S, enc, lens, out[0], (0, 1, 7, B - 1))
