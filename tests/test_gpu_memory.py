"""Engines on a GPU that is nearly full: the prefill buffers give way to the caller's pool."""
import gc

import pytest

from paper_2608_14376_b200 import synth
from tests.helpers import have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def test_an_engine_fits_beside_what_is_left_and_gives_the_same_bytes():
    import torch

    from paper_2608_14376_b200 import corun

    sh = synth.ModelShape(2, 2048, 16, 4, 128, 8192, 4096, 1e-6, 10000.0)
    w = synth.make_weights_torch(sh, seed=3)
    prompts = synth.make_prompts(sh.vocab, [1900, 700, 60], seed=4)

    def run():
        eng = corun.Engine(sh, w, 8, 2048, kv_pool_blocks=3 * 128)
        try:
            eng.prefill_batch([1, 4, 6], prompts, [len(p) + 8 for p in prompts])
            return [eng.logits(s).tobytes() for s in (1, 4, 6)]
        finally:
            eng.close()

    want = run()                                      # (and every kernel it launches is loaded)
    gc.collect(); torch.cuda.empty_cache(); torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    eng = corun.Engine(sh, w, 8, 2048, kv_pool_blocks=3 * 128)
    used = free - torch.cuda.mem_get_info()[0]
    eng.close()
    # half of that: the pool and the decode step's buffers are a small part, chunks of 2048 rows need more
    hog = torch.empty(torch.cuda.mem_get_info()[0] - used // 2, dtype=torch.uint8, device="cuda")
    try:
        assert run() == want
    finally:
        del hog
        torch.cuda.empty_cache()
