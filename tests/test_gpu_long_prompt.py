"""Prefill of prompts beyond the small chunk: the projections on pairs of SMs, chunks of up to 2048 rows, at the edges of
their tiles (256 rows, 128 per SM, 32 per store) and of the chunk."""
import numpy as np
import pytest

from paper_2608_14376_b200 import synth
from tests.helpers import Tiny, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]
TOL = 3e-2


@pytest.fixture(scope="module")
def tiny(orc):
    return Tiny(orc)


@pytest.mark.parametrize("lens", [[257], [513, 256, 287], [300, 640, 1, 1409], [2048, 257], [2049, 900]])
def test_long_prompts_alone_and_sharing_chunks(tiny, lens):
    """A long prompt's logits against the oracle, and byte for byte the same (with the cache and the decode step that
    follows) whether it is prefilled alone or with others, some of them short ones that take the small chunks."""
    from oracle import oracle
    from paper_2608_14376_b200 import corun

    B = 8
    sh = tiny.sh
    prompts = synth.make_prompts(sh.vocab, lens, seed=700 + lens[0])
    slots = [6, 1, 3, 0][:len(lens)]
    seeds = np.array([synth.request_seed(i) for i in range(len(lens))], np.uint64)
    res = [n + 4 for n in lens]
    e = corun.Engine(sh, tiny.w_t, B, max(res))

    def after():
        active = np.zeros(B, np.uint8); active[slots] = 1
        sd = np.zeros(B, np.uint64); sd[slots] = seeds
        out = [e.logits(s).tobytes() for s in slots]
        for layer in range(sh.n_layers):
            for s, n in zip(slots, lens):
                k, v = e.kv_read(s, layer, 0, n)
                out.append(k.tobytes() + v.tobytes())
        out.append(e.decode_step(active, sd).tobytes())
        out += [e.logits(s).tobytes() for s in slots]
        return out

    first = [e.prefill(s, p, r, 0.7, 0.95, seed=int(sd)) for s, p, r, sd in zip(slots, prompts, res, seeds)]
    for s, p in zip(slots, prompts):
        r = oracle.Request(tiny.oracle, p, 1, max_T=len(p) + 4)
        r.prefill()
        assert np.abs(e.logits(s) - r.logits).max() <= TOL
    alone = after()
    for s in slots:
        e.release(s)
    assert list(e.prefill_batch(slots, prompts, res, 0.7, 0.95, seeds)) == first
    assert after() == alone
    e.close()
