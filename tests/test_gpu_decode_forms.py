"""Decode at the edges of its forms: the router's CTAs (8 experts each, one row or four), the selected-experts form (row
tiles of 16, 32 and 64) and the projections on pairs of SMs (above 128 slots), with one request and with all slots in use."""
import numpy as np
import pytest

from oracle import moe_oracle as mo
from paper_2608_14376_b200 import synth
from tests.helpers import have_gpu
from tests.test_gpu_moe import GAP, _device_op, _weights

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]
TOL = 3e-3          # logits of the tiny decoder (standard deviation 0.3) against the oracle; measured 5.6e-4 at most


@pytest.mark.parametrize("H,E,K,B", [(2176, 13, 3, 1), (12288, 9, 2, 3), (128, 8, 8, 96), (256, 13, 3, 97), (2176, 40, 4, 101), (256, 256, 16, 128)])
def test_router_shares(H, E, K, B):
    """Logits from several CTAs per row (remainders of experts, of rows and of the row's length), twice, since the CTAs
    of a launch leave their meeting point as they found it."""
    import torch

    from paper_2608_14376_b200 import corun

    w = _weights(H, E, 64, 0, seed=H + E)
    op = _device_op(corun, torch, w, H, E, K, 64, 0, B)
    rng = np.random.default_rng(B)
    for _ in range(2):
        X = rng.standard_normal((B, H)).astype(np.float32)
        _, ex, pr = op.forward(torch.tensor(X).cuda())
        op.sync()
        ex, pr = ex.cpu().numpy(), pr.cpu().numpy()
        for b in range(B):
            _, _, p_all = mo.router(X[b], w["router"], K)
            order = np.argsort(-p_all, kind="stable")
            near = np.diff(-p_all[order][:K + 1])
            if near.size == 0 or near.min() > GAP:
                assert list(ex[b]) == list(order[:K])
            # a logit of up to 12: its sum of H fp32 products is off by some 1e-6, and a probability by as much of itself
            np.testing.assert_allclose(pr[b], p_all[ex[b]], atol=2e-6, rtol=1e-5)


@pytest.mark.parametrize("arch,B", [("moe", 1), ("moe", 16), ("moe", 17), ("moe", 64), ("moe", 130), ("dense", 130), ("dense", 200)])
def test_one_request_and_all_slots(orc, arch, B):
    from paper_2608_14376_b200 import corun

    sh = synth.TINY
    w_np = synth.make_weights_numpy(sh, seed=11)
    m_np = synth.make_moe_numpy(sh, 8, 2, 128, 1, False, seed=11) if arch == "moe" else None
    kw = dict(moe=m_np) if m_np else {}
    model = orc.Model(orc.Shape(**sh.dict()), w_np, **kw)
    kw = dict(moe=synth.moe_numpy_to_torch(m_np, "cuda")) if m_np else {}
    eng = corun.Engine(sh, synth.weights_numpy_to_torch(w_np, "cuda"), B, 64, **kw)
    try:
        prompts = synth.make_prompts(sh.vocab, [5 + i % 9 for i in range(B)], seed=12)
        seeds = np.array([synth.request_seed(i) for i in range(B)], np.uint64)
        probe = sorted({0, B // 2, B - 1})
        first, alone = {}, {}
        for s in probe:                               # one request in the engine
            r = orc.Request(model, prompts[s], 1, max_T=64)
            r.prefill()
            first[s] = int(np.argmax(r.logits))
            active = np.zeros(B, np.uint8); active[s] = 1
            eng.prefill(s, prompts[s], len(prompts[s]) + 4)
            eng.force_token(s, first[s])
            eng.decode_step(active, seeds)
            r.decode(force_token=first[s])
            assert np.abs(eng.logits(s) - r.logits).max() <= TOL
            alone[s] = eng.logits(s).tobytes()
            eng.release(s)
        eng.prefill_batch(list(range(B)), prompts, [len(p) + 4 for p in prompts])
        for s in probe:
            eng.force_token(s, first[s])
        eng.decode_step(np.ones(B, np.uint8), seeds)
        for s in probe:
            assert eng.logits(s).tobytes() == alone[s]
    finally:
        eng.close()


@pytest.mark.parametrize("E,K,S,renorm", [(8, 3, 1, False), (16, 4, 0, True)])
def test_vanished_routing_weights_add_nothing(orc, E, K, S, renorm):
    """A saturated router (logits of some +-200: the weights of a row's second and later experts underflow to 0 in many
    layers): the row's values are the oracle's, and the same bytes whatever request used the row before."""
    from paper_2608_14376_b200 import corun

    sh, B = synth.TINY, 4
    w_np = synth.make_weights_numpy(sh, seed=13)
    m_np = synth.make_moe_numpy(sh, E, K, 128, S, renorm, seed=13, std=0.1, router_std=12.0)
    model = orc.Model(orc.Shape(**sh.dict()), w_np, moe=m_np)
    prompts = synth.make_prompts(sh.vocab, [11, 7, 9], seed=14)
    active, seeds = np.array([0, 1, 0, 0], np.uint8), np.zeros(B, np.uint64)
    w_t, m_t = synth.weights_numpy_to_torch(w_np, "cuda"), synth.moe_numpy_to_torch(m_np, "cuda")
    runs = []
    for before in ([], [prompts[1], prompts[2]]):
        eng = corun.Engine(sh, w_t, B, 64, moe=m_t)
        try:
            for p in before + [prompts[0]]:
                r = orc.Request(model, p, 1, max_T=64)
                r.prefill()
                eng.prefill(1, p, len(p) + 8)
                out = []
                for _ in range(4):
                    tok = int(np.argmax(r.logits))
                    eng.force_token(1, tok)
                    eng.decode_step(active, seeds)
                    r.decode(force_token=tok)
                    out.append(eng.logits(1))
                    # router logits, and what rounding moves them by, are 60 times those of the other tests (whose logits are
                    # off by some 3e-4): up to 60 * 3e-4; measured 9e-3, and 0.6 with what another layer left added
                    assert np.abs(out[-1] - r.logits).max() <= 10 * TOL
                eng.release(1)
            runs.append([o.tobytes() for o in out])
        finally:
            eng.close()
    assert runs[0] == runs[1]
