"""The kernels of long prompts run by themselves against 64-bit arithmetic: the attention of a chunk's rows over the slot's
cached positions, and the GEMM on pairs of SMs."""
import numpy as np
import pytest

from paper_2608_14376_b200 import synth
from tests.helpers import have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]

HALF_ULP = 2.0 ** -11       # a weight in fp16 (11 significant bits) is off by at most this share of itself


def _dense(nq, nkv, hd, T):
    from paper_2608_14376_b200 import corun

    sh = synth.ModelShape(1, 256, nq, nkv, hd, 256, 512, 1e-6, 10000.0)
    return corun.Engine(sh, synth.weights_numpy_to_torch(synth.make_weights_numpy(sh, seed=1), "cuda"), 2, T)


def _fill(eng, slot, k, v):
    eng.adopt(slot, 0, k.shape[0], 0)
    eng.kv_write(slot, 0, 0, k, v)
    return eng.kv_read(slot, 0, 0, k.shape[0])


def _attend(q, k, v, pos0, scale):
    """q [n, nq, d], k [T, nkv, d], v [T, nkv, dv] -> (output, sqrt(sum p^2 v^2)) in fp64; row i sees positions 0 .. pos0 + i."""
    q, k, v = (np.asarray(x, np.float64) for x in (q, k, v))
    G = q.shape[1] // k.shape[1]
    out, spread = np.empty(q.shape[:2] + v.shape[2:]), np.empty(q.shape[:2] + v.shape[2:])
    for i in range(q.shape[0]):
        T = pos0 + i + 1
        for h in range(q.shape[1]):
            s = k[:T, h // G] @ q[i, h] * scale
            p = np.exp(s - s.max())
            p /= p.sum()
            out[i, h] = p @ v[:T, h // G]
            spread[i, h] = np.sqrt((p * p) @ (v[:T, h // G] ** 2))
    return out, spread


# group sizes 8, 4, 2, 1 and both head widths; one row, ragged tiles, several blocks of 128 keys, keys of an earlier chunk
@pytest.mark.parametrize("nq,nkv,hd,pos0,n", [(8, 1, 128, 0, 1), (8, 2, 128, 0, 77), (8, 2, 128, 500, 33), (4, 2, 64, 0, 130),
                                              (4, 4, 64, 700, 5), (16, 2, 64, 127, 18), (2, 2, 128, 255, 129)])
def test_prefill_attention_matches_fp64(nq, nkv, hd, pos0, n):
    rng = np.random.default_rng(nq + hd + n)
    T = pos0 + n
    eng = _dense(nq, nkv, hd, T)
    try:
        k, v = _fill(eng, 1, *(rng.standard_normal((T, nkv * hd)).astype(np.float32) for _ in range(2)))
        q = (8 * rng.standard_normal((n, nq, hd))).astype(np.float32)          # scores of +-8
        got = eng.prefill_attention(1, 0, pos0, q)
    finally:
        eng.close()
    k, v = k.reshape(T, nkv, hd), v.reshape(T, nkv, hd)
    want, spread = _attend(q, k, v, pos0, hd ** -0.5)
    rms = lambda x: np.sqrt(np.mean(np.square(x)))
    # rounding of the weights to fp16: an error uniform in +-half an ulp is 0.73 / sqrt(3) of HALF_ULP in the mean over the
    # binade; beside it 2^-17 of the result (stored as a bf16 pair) and scores of up to 40 in fp32
    bound = 1.25 * 0.73 / np.sqrt(3) * HALF_ULP * rms(spread) + 1e-5 * rms(want)
    assert rms(got - want) <= bound, (rms(got - want), bound)
    # queries in half the precision (their fp16 part alone) would not pass
    if T > 100:
        assert rms(_attend(q.astype(np.float16), k, v, pos0, hd ** -0.5)[0] - want) > bound


@pytest.mark.parametrize("hd", [64, 128])
def test_a_blocks_largest_weight_is_exact(hd):
    """One key per block of 128 carries the block's weight: fp16 weights are 1 for it, whatever the other blocks hold, so
    the result has the accuracy of its fp32 sums (a weight rounded to fp16 would be off by up to 5e-4 of itself)."""
    rng = np.random.default_rng(hd)
    T, A = 128 * 5 + 40, 32.0
    k = np.zeros((T, hd), np.float32)
    k[:, 0] = -40 * hd ** 0.5 / A
    top = [5, 130, 300, 511, 512, T - 3]
    k[top, 0] = np.array([-0.31, -1.27, 0.13, -0.74, -2.09, -0.55]) * hd ** 0.5 / A
    v = rng.standard_normal((T, hd)).astype(np.float32)
    q = np.zeros((1, 1, hd), np.float32)
    q[0, 0, 0] = A
    eng = _dense(1, 1, hd, T)
    try:
        k, v = _fill(eng, 1, k, v)
        got = eng.prefill_attention(1, 0, T - 1, q)
    finally:
        eng.close()
    want, _ = _attend(q, k.reshape(T, 1, hd), v.reshape(T, 1, hd), T - 1, hd ** -0.5)
    assert np.abs(got - want).max() <= 2e-5 * np.abs(want).max() + 2 ** -17 * np.abs(want).max()


def _product(form, N, K, R, seed):
    """The GEMM on pairs of SMs -> (result, 64-bit result, 64-bit result of the activations as bf16 pairs, that of their bf16 part
    alone).  Forms: 0 plain, 1 with SwiGLU, 2 keys and values; 3, 4: 0, 1 of a decode step."""
    import torch

    from paper_2608_14376_b200 import corun

    g = torch.Generator(device="cuda").manual_seed(seed)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.02).bfloat16()
    X = torch.randn((R, K), generator=g, device="cuda")
    hi = X.bfloat16()
    lo = (X - hi.float()).bfloat16()

    def f(x):
        y = x @ W.double().T
        return torch.nn.functional.silu(y[:, :N // 2]) * y[:, N // 2:] if form in (1, 4) else y

    return corun.debug_gemm_pair(form, W, X).double(), f(X.double()), f(hi.double() + lo.double()), f(hi.double())


# edges of the tiles (256 rows, 128 per SM, 32 per store; 256 columns, 96 or 128 outputs with SwiGLU), whole tiles and tiles dealt
# out slice by slice, one slice and eight
@pytest.mark.parametrize("form,N,K,R", [(0, 8, 64, 1), (0, 200, 192, 257), (0, 1536, 1024, 300), (0, 4096, 4096, 256), (0, 6144, 4096, 129),
                                        (0, 1024, 3072, 1000), (0, 4096, 12288, 515), (1, 128, 64, 31), (1, 1408, 1024, 255),
                                        (1, 2 * 12288, 4096, 256), (1, 2 * 3072, 1024, 777), (2, 256, 256, 65), (2, 1024, 512, 513),
                                        (3, 200, 192, 1), (3, 4096, 12288, 33), (3, 6144, 4096, 128), (3, 1536, 1024, 129), (3, 4096, 4096, 256),
                                        (4, 1408, 1024, 65), (4, 2 * 12288, 4096, 128), (4, 2 * 12288, 4096, 200), (4, 2 * 3072, 1024, 97)])
def test_pair_gemm_matches_fp64(form, N, K, R):
    got, want, pairs, bf16 = _product(form, N, K, R, seed=N + K + R)
    off = lambda a, b: float((a - b).norm() / b.norm())
    # 16 significand bits of the activations (2.5e-6), a slice's sum cut off at every MMA (1.7e-8 each, at most 24 k-blocks of 8:
    # 3.3e-6); a SwiGLU's result is a product of two such sums and stored as a bf16 pair (2e-6)
    bound = 8e-6 if form in (1, 4) else 4.5e-6
    assert off(got, want) <= bound, off(got, want)
    assert off(got, pairs) <= off(got, want) + 1e-6
    assert off(bf16, want) > 10 * bound                # without the lo part it would not pass


@pytest.mark.parametrize("form,N,K", [(3, 200, 192), (3, 6144, 4096), (3, 4096, 12288), (4, 1408, 1024), (4, 2 * 12288, 4096)])
def test_decode_pair_gemm_gives_a_row_the_same_bytes_in_both_forms(form, N, K):
    """Up to 128 rows the hi and lo parts are stacked in one operand, above they have an accumulator each."""
    import torch

    from paper_2608_14376_b200 import corun

    g = torch.Generator(device="cuda").manual_seed(N + K)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.02).bfloat16()
    X = torch.randn((256, K), generator=g, device="cuda")
    full = corun.debug_gemm_pair(form, W, X)
    for R in (1, 31, 64, 65, 97, 128, 129, 200):
        assert torch.equal(corun.debug_gemm_pair(form, W, X[:R].contiguous()), full[:R]), R
    assert torch.equal(corun.debug_gemm_pair(form, W, X[100:200].contiguous()), full[100:200])


# rows per expert at the edges of the padded counts (16, 32, 48, 64: two tiles in tensor memory; 80, 96, 128: one), experts of several
# groups, some without a row.  Weight rows of a tile: 256 in each SM, or 128 gate and their up rows: N and F that end in the first
# SM of a later tile, inside the second one, and in between
GROUPS = [[1, 16, 17, 0, 64, 65, 80], [81, 96, 97, 112, 128, 129, 200], [128, 1, 128, 31, 256, 5, 127], [0, 0, 48, 0, 0, 0, 300]]


@pytest.mark.parametrize("rows", GROUPS, ids=["few", "many", "mixed", "empty"])
@pytest.mark.parametrize("form,N,K", [(0, 128, 64), (0, 512, 384), (0, 768, 1408), (0, 896, 192), (0, 2048, 768), (1, 2 * 64, 64), (1, 2 * 200, 256),
                                      (1, 2 * 384, 768), (1, 2 * 456, 192), (1, 2 * 1408, 2048)])
def test_experts_of_a_prompt_match_fp64(form, N, K, rows):
    import torch

    from paper_2608_14376_b200 import corun

    g = torch.Generator(device="cuda").manual_seed(N + K + sum(rows))
    E, n = len(rows), sum(rows)
    W = (torch.randn((E, N, K), generator=g, device="cuda") * 0.02).bfloat16()
    X = torch.randn((n, K), generator=g, device="cuda")
    row_w = torch.rand((n,), generator=g, device="cuda") + 0.1
    flat = W if form else W.permute(1, 0, 2).reshape(N, E * K).contiguous()
    got = corun.debug_gemm_experts(form, flat, rows, X, row_w if form else None)
    # 16 significand bits of the activations (2.5e-6), sums cut off at each of 4 MMAs per k-block (1.7e-8); with SwiGLU a product of
    # two such sums, stored as a bf16 pair (2e-6)
    bound = (2.5e-6 + 4 * 1.7e-8 * K / 64) * (2 if form else 1) + (2e-6 if form else 0) + 5e-7
    at = 0
    for e, m in enumerate(rows):                      # expert by expert: a row's error is not hidden among the others'
        if m == 0:
            continue
        y = X[at:at + m].double() @ W[e].double().T
        if form:
            y = row_w[at:at + m, None].double() * torch.nn.functional.silu(y[:, :N // 2]) * y[:, N // 2:]
        off = ((got[at:at + m].double() - y).norm(dim=1) / y.norm(dim=1)).max()
        assert off <= 2.5 * bound, (e, float(off), bound)       # the worst row: of K = 64 products only, some 1.6 times the mean's error
        assert float((got[at:at + m].double() - y).norm() / y.norm()) <= bound, e
        at += m


MLA = dict(kv_lora_rank=256, qk_nope=128, qk_rope=32, v_head=128, first_dense=2)


def _latent(scale_k=None, scale_v=None, B=2, T=700, seed=2, kv_block=64, mla=MLA):
    """A dense decoder with latent attention; scale_k, scale_v: per head, powers of two that its keys (queries: their inverse)
    and its values (output projection: their inverse) are multiplied by, which changes nothing in exact arithmetic."""
    from paper_2608_14376_b200 import corun

    nh, nope, rope, vh = 4, mla["qk_nope"], mla["qk_rope"], mla["v_head"]
    sh = synth.ModelShape(2, 256, nh, nh, 128, 384, 1024, 1e-6, 10000.0)
    w, m = synth.make_mla_weights_numpy(sh, mla, seed=seed, std=0.05)

    def times(bits, where, f):
        x = synth.bf16_bits_to_f32(bits)
        x[where] *= np.float32(f)
        bits[:] = synth.f32_to_bf16_bits(x)

    for l in range(sh.n_layers):
        for h in range(nh) if scale_k is not None else ():
            times(m["wkv_b"][l], slice(h * (nope + vh), h * (nope + vh) + nope), scale_k[h])
            times(w["wqkv"][l], slice(h * (nope + rope), h * (nope + rope) + nope), 1 / scale_k[h])
            times(m["wkv_b"][l], slice(h * (nope + vh) + nope, (h + 1) * (nope + vh)), scale_v[h])
            times(w["wo"][l], (slice(None), slice(h * vh, (h + 1) * vh)), 1 / scale_v[h])
    wt, mt = synth.mla_numpy_to_torch(w, m, "cuda")
    return sh, m, corun.Engine(sh, wt, B, T, mla=mt, kv_block=kv_block)


@pytest.mark.parametrize("pos0,n", [(0, 1), (0, 129), (63, 2), (500, 77), (64, 300)])
def test_latent_prefill_attention_matches_fp64(pos0, n):
    rng = np.random.default_rng(n)
    T = pos0 + n
    sh, m, eng = _latent(T=T)
    nh, rank, nope, rope = 4, MLA["kv_lora_rank"], MLA["qk_nope"], MLA["qk_rope"]
    try:
        eng.adopt(1, 0, T, 0)
        eng.kv_write(1, 0, 0, rng.standard_normal((T, rank + rope)).astype(np.float32), None)
        c = eng.kv_read(1, 0, 0, T)[0].astype(np.float64)
        pair = lambda x: (lambda hi: hi + synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(x - hi)))(synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(x)))
        q = pair(2 * rng.standard_normal((n, nh, nope + rope)).astype(np.float32))   # what a bf16 pair holds exactly
        got = eng.prefill_attention(1, 0, pos0, q)
    finally:
        eng.close()
    W = synth.bf16_bits_to_f32(m["wkv_b"][0]).astype(np.float64).reshape(nh, nope + 128, rank)
    k = np.concatenate([np.einsum("tc,hdc->thd", c[:, :rank], W[:, :nope]), np.repeat(c[:, None, rank:], nh, 1)], -1)
    v = np.einsum("tc,hdc->thd", c[:, :rank], W[:, nope:])
    scale = (nope + rope) ** -0.5
    want, _ = _attend(q, k, v, pos0, scale)
    rms = lambda x: np.sqrt(np.mean(np.square(x)))
    # the result is stored as a bf16 pair (3e-6 in the mean); sums cut off by the tensor core (1.7e-8 for each of 64 MMAs over a
    # latent, 44 over a block) move scores of up to 20 by some 1e-6 and values by as much of themselves
    bound = 1e-5 * rms(want)
    assert rms(got - want) <= bound, rms(got - want) / rms(want)
    if T > 100:                                       # keys or values without their lo part would not pass
        assert rms(_attend(q, k.astype(np.float16), v, pos0, scale)[0] - want) > 3 * bound
        assert rms(_attend(q, k, v.astype(np.float16), pos0, scale)[0] - want) > 3 * bound


def test_latent_prefill_does_not_depend_on_the_scale_of_keys_and_values():
    """Keys, values and queries a million times larger or smaller, per head, are the same bytes in the end (as fp16 pairs they
    would overflow above 65504 and lose their low bits below 1e-4)."""
    prompt = synth.make_prompts(1024, [300], seed=5)[0]
    out = []
    for ks, vs in ((None, None), ([2.0 ** -20, 2.0 ** 20, 2.0 ** 9, 2.0 ** -20], [2.0 ** -20, 2.0 ** 20, 2.0 ** -9, 2.0 ** 22])):
        _, _, eng = _latent(ks, vs, T=310)
        try:
            eng.prefill(1, prompt, 310)
            out.append(eng.logits(1))
            eng.force_token(1, 7)
            eng.decode_step(np.array([0, 1], np.uint8), np.zeros(2, np.uint64))
            out.append(eng.logits(1))
        finally:
            eng.close()
    assert np.isfinite(out[2]).all()
    assert out[0].tobytes() == out[2].tobytes() and out[1].tobytes() == out[3].tobytes()
