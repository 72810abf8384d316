"""Debug readers: intermediate buffers of engines of every form, and the GEMM timelines (a library built with
CORUN_BUILD_DEBUG=1 only)."""
import numpy as np
import pytest

from paper_2608_14376_b200 import synth
from tests.helpers import have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def _engine(arch, B):
    from paper_2608_14376_b200 import corun

    sh = synth.TINY
    kw = dict(moe=synth.moe_numpy_to_torch(synth.make_moe_numpy(sh, 8, 2, 128, 1, False, seed=1), "cuda")) if arch == "moe" else {}
    eng = corun.Engine(sh, synth.weights_numpy_to_torch(synth.make_weights_numpy(sh, seed=1), "cuda"), B, 64, **kw)
    eng.prefill(B - 1, [3, 5, 7], 10)
    active = np.zeros(B, np.uint8); active[B - 1] = 1
    eng.decode_step(active, np.zeros(B, np.uint64))
    return eng


@pytest.mark.parametrize("arch,B", [("dense", 8), ("dense", 200), ("moe", 8), ("moe", 140)])
def test_every_buffer_is_read_or_refused(arch, B):
    from paper_2608_14376_b200 import corun

    eng = _engine(arch, B)
    try:
        for which in range(8):
            assert eng.debug_read(which, 64).shape == (64,)
        with pytest.raises(corun.CorunError) as err:
            eng.debug_read(8, 1)
        assert err.value.status == corun.EINVAL
    finally:
        eng.close()


def test_a_buffer_that_latent_attention_does_not_have_is_refused():
    from paper_2608_14376_b200 import corun
    from tests.test_gpu_prefill_kernels import _latent

    _, _, eng = _latent(T=64)
    try:
        for which in (0, 1, 2):                       # rotated queries and split partials of the other attention
            with pytest.raises(corun.CorunError) as err:
                eng.debug_read(which, 1)
            assert err.value.status == corun.EINVAL
    finally:
        eng.close()


@pytest.mark.parametrize("arch,B", [("dense", 8), ("dense", 200), ("moe", 8), ("moe", 140)])
def test_gemm_timelines_of_every_form(arch, B):
    from paper_2608_14376_b200 import corun

    if not hasattr(corun.lib(), "corun_debug_gemm_trace"):
        pytest.skip("needs a library built with CORUN_BUILD_DEBUG=1")
    eng = _engine(arch, B)
    try:
        for kind in range(5):
            if arch == "moe" and B > 64 and kind in (2, 3):   # grouped experts
                with pytest.raises(corun.CorunError):
                    eng.gemm_trace(kind, 1)
                continue
            t = eng.gemm_trace(kind, 1)
            ran = t[:, 0] >= 0
            assert ran.any() and (t[ran, 1] >= t[ran, 0]).all()
            assert t[:, 7].max() >= t[:, 2].max() > 0
    finally:
        eng.close()
