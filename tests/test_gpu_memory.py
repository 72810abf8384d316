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


def test_an_engine_leaves_room_for_its_step():
    """The buffers of the largest chunks would fit and leave next to nothing: smaller ones are taken, 128 MiB stay free."""
    import torch

    from paper_2608_14376_b200 import corun

    sh = synth.ModelShape(2, 2048, 16, 4, 128, 8192, 4096, 1e-6, 10000.0)
    w = synth.make_weights_torch(sh, seed=3)
    prompts = synth.make_prompts(sh.vocab, [1900, 60], seed=4)

    def run():
        eng = corun.Engine(sh, w, 8, 2048, kv_pool_blocks=3 * 128)
        try:
            free = torch.cuda.mem_get_info()[0]
            eng.prefill_batch([1, 6], prompts, [len(p) + 8 for p in prompts])
            return free, [eng.logits(s).tobytes() for s in (1, 6)]
        finally:
            eng.close()

    run()                                             # (every kernel is loaded)
    gc.collect(); torch.cuda.empty_cache(); torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    free, want = run()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (before - free) - (32 << 20), dtype=torch.uint8, device="cuda")
    try:
        free, got = run()
        assert got == want and free >= 100 << 20      # (what was left, but for the step's graph)
    finally:
        del hog
        torch.cuda.empty_cache()


@pytest.mark.parametrize("experts", [False, True])
def test_chunks_of_more_rows_take_what_the_rows_need(experts):
    """A chunk may have 4096 rows where a prompt can have more than 2048 tokens.  What one half of a layer hands on and what the other
    does share memory, and so do an expert's gathered rows and its results."""
    import torch

    from paper_2608_14376_b200 import corun

    H, nq, nkv, hd, E, K, Fx = 4096, 32, 8, 128, 128, 16, 512
    F = 64 if experts else 12288
    sh = synth.ModelShape(1, H, nq, nkv, hd, F, 4096, 1e-6, 10000.0)
    w = synth.make_weights_torch(sh, seed=3, dense_ffn=not experts)
    kw = dict(moe=synth.make_moe_torch(sh, seed=3, n_experts=E, top_k=K, expert_ffn=Fx, n_shared=0, renormalize=True)) if experts else {}

    def used(max_context):
        gc.collect(); torch.cuda.empty_cache(); torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        eng = corun.Engine(sh, w, 8, max_context, kv_pool_blocks=64, **kw)
        try:
            return free - torch.cuda.mem_get_info()[0]
        finally:
            eng.close()

    used(2048)                                        # (kernels are loaded)
    # a row's normalised pair, residual, attention output and output of half a layer; beside them the larger of the projections and
    # queries, and of the feed-forward's hidden activations or K experts' rows (gathered, then results) with theirs
    row = 4 * H + 4 * H + 4 * nq * hd + 4 * H + max(4 * (2 * nq + 2 * nkv) * hd, K * 4 * (H + Fx) if experts else 4 * F)
    # (10 % for tables and partial tiles; apart, the buffers of a row take 1.5 and 1.9 times as much)
    more = used(4096) - used(2048)
    assert more <= 1.1 * 2048 * row + (32 << 20), (more, 2048 * row)
