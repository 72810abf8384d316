"""Prompts around the largest chunk (4096 rows), alone and behind others: the cut falls elsewhere, the bytes are the same."""
import numpy as np
import pytest

from paper_2608_14376_b200 import synth
from tests.helpers import have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]
TOL = 3e-3          # as in test_gpu_long_prompt


@pytest.mark.parametrize("arch,lens", [("dense", [300, 4096]), ("dense", [4097, 129]), ("moe", [300, 4097]), ("moe", [4500, 140]),
                                       ("mla", [140, 4097]), ("mla", [129] * 17 + [200]), ("mla", [4096 + 100] + [129] * 15 + [200])])
def test_where_a_chunk_ends_changes_no_byte(orc, arch, lens):
    """Expert layers: an expert's rows over a whole chunk, more than 64 words of row masks.  Latent attention: chunks
    full of requests (129 tokens take two tiles of 128 rows), 8 in one of 2048 rows; and as many as 4096 rows can hold, 17: the end of a
    longer prompt on one tile, 15 on two each, and the beginning of one on the last tile."""
    from paper_2608_14376_b200 import corun

    mla = dict(kv_lora_rank=256, qk_nope=128, qk_rope=32, v_head=128, first_dense=1)
    moe = dict(n_experts=16, top_k=3, expert_ffn=128, n_shared=1, renormalize=arch == "moe")
    kw, m, ex = {}, None, None
    if arch == "mla":
        sh = synth.ModelShape(2, 256, 4, 4, 128, 384, 1024, 1e-6, 10000.0)
        w, m = synth.make_mla_weights_numpy(sh, mla, seed=5)
        wt, kw["mla"] = synth.mla_numpy_to_torch(w, m, "cuda")
        kw["kv_block"] = 64
    else:
        sh = synth.ModelShape(2, 256, 4, 2, 64, 384 if arch == "dense" else 64, 1024, 1e-6, 10000.0)
        w = synth.make_weights_numpy(sh, seed=5)
        wt = synth.weights_numpy_to_torch(w, "cuda")
    if arch != "dense":
        ex = synth.make_moe_numpy(sh, seed=5, **moe)
        kw["moe"] = synth.moe_numpy_to_torch(ex, "cuda")
    model = orc.Model(orc.Shape(**sh.dict()), w, **{k: v for k, v in (("moe", ex), ("mla", m)) if v})
    B = max(len(lens), -(-4096 // (-(-(max(lens) + 2) // 128) * 128)))     # slots for a chunk of 4096 rows
    prompts = synth.make_prompts(sh.vocab, lens, seed=60 + len(lens))
    slots, res = list(range(len(lens))), [n + 2 for n in lens]
    e = corun.Engine(sh, wt, B, max(res), **kw)
    try:
        for s in slots:
            e.prefill(s, prompts[s], res[s])
        if arch == "mla" and lens[0] > 4096:          # the chunk has 4096 rows: its attention takes that many and no more
            q = np.zeros((4097, 4, 160), np.float32)
            e.prefill_attention(0, 0, 0, q[:4096])
            with pytest.raises(corun.CorunError):
                e.prefill_attention(0, 0, 0, q)
        for s in slots:
            if lens[s] <= 300 and s < 3:
                r = orc.Request(model, prompts[s], 1, max_T=lens[s] + 2)
                r.prefill()
                assert np.abs(e.logits(s) - r.logits).max() <= TOL

        def state():
            out = [e.logits(s).tobytes() for s in slots]
            for s in slots:
                k, v = e.kv_read(s, sh.n_layers - 1, 0, lens[s])
                out.append(k.tobytes() + (v.tobytes() if v is not None else b""))
            return out

        alone = state()
        for s in slots:
            e.release(s)
        e.prefill_batch(slots, prompts, res)
        assert state() == alone
    finally:
        e.close()
