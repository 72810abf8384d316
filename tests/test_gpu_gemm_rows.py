"""The GEMM with the weights as its M operand at the edges of its padded row counts (16, 32, 48, 64, 80, 96, 128)."""
import numpy as np
import pytest

from paper_2608_14376_b200 import synth
from tests.helpers import have_gpu
from tests.test_gpu_kernels import _gemm_case

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


@pytest.mark.parametrize("R", [1, 16, 17, 32, 33, 48, 49, 65, 80, 81, 96, 97, 112, 113, 128])
@pytest.mark.parametrize("N,K", [(328, 1152), (4096, 640)])
def test_padded_row_counts(orc, R, N, K):
    """One tile and a ragged rest (N = 328: no multiple of 32 either), CTAs that cross tiles and such that share one."""
    import torch

    out, ref, _, _ = _gemm_case(orc, torch, R, N, K, seed=R + N)
    # activations carry 16 significand bits: 2^-17 of every product, 0.02 * sqrt(K) * 4 being a bound of the sums seen
    tol = 2e-5 * 0.02 * np.sqrt(K) * 4 + 1e-6
    assert np.abs(out - ref).max() <= tol


@pytest.mark.parametrize("N,K", [(4096, 12288), (6144, 4096), (4096, 4096), (5120, 2048), (328, 1152), (20000, 1024)])
def test_few_rows_are_no_further_off_than_many(N, K):
    """The tensor core's accumulator cuts every sum off, so an error grows with the k-blocks that one accumulator takes.  Up to 32
    rows a tile may be half as wide, but not where half as many CTAs would then share its K.  Positive products: nothing of what is
    cut off cancels."""
    import torch

    from paper_2608_14376_b200 import corun

    g = torch.Generator(device="cuda").manual_seed(N + K)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.02).abs().bfloat16()
    X = (torch.rand((48, K), generator=g, device="cuda") + 0.5).bfloat16().float()      # exact as it is: only the sums are off
    want = X.double() @ W.double().T

    def off(rows):
        return float((corun.debug_gemm(W, X[:rows].contiguous()).double() - want[:rows]).norm() / want[:rows].norm())

    wide = off(48)
    for rows in (1, 16, 17, 32):
        assert off(rows) <= 1.1 * wide + 3e-8, (rows, off(rows), wide)    # (3e-8: the result's own rounding to fp32)


@pytest.mark.parametrize("B", [16, 40, 100, 128])
def test_rows_of_a_step_are_counted(B):
    """A request's logits are the same bytes with any number of requests in the step: the padded rows follow the count."""
    import torch

    from paper_2608_14376_b200 import corun

    sh = synth.TINY
    eng = corun.Engine(sh, synth.weights_numpy_to_torch(synth.make_weights_numpy(sh, seed=3), "cuda"), B, 64)
    try:
        prompts = synth.make_prompts(sh.vocab, [5 + i % 7 for i in range(B)], seed=4)
        seeds = np.array([synth.request_seed(i) for i in range(B)], np.uint64)
        want = None
        for n in [1, 15, 16, 17, 32, 33, 48, 49, 64, 65, 80, 81, 96, 97, 128]:
            if n > B:
                continue
            slots = list(range(B - n, B))             # the probe is slot B - 1: the last row of the step
            for s in slots:
                eng.prefill(s, prompts[s], 40, seed=int(seeds[s]))
            active = np.zeros(B, np.uint8)
            active[slots] = 1
            for s in slots:
                eng.force_token(s, 7)
            eng.decode_step(active, seeds)
            got = eng.logits(B - 1).copy()
            want = got if want is None else want
            np.testing.assert_array_equal(got, want)
            for s in slots:
                eng.release(s)
    finally:
        eng.close()
