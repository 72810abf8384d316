"""ctypes binding of the C ABI in ``include/corun.h`` (argument marshalling only).

Every step of the hot path runs in the CUDA kernels of ``libcorun.so``; there
is no CPU or PyTorch fallback: if the library is missing or the call fails, an
exception is raised.
"""
from __future__ import annotations

import ctypes as C
import os

import numpy as np

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libcorun.so")

OK, EINVAL, ESLOT, ENOSPACE, ECTX, ECUDA, ETIMEOUT, ENOMEM, ELIMIT = 0, -1, -2, -3, -4, -5, -6, -7, -8

EXPORTS = [
    "corun_init", "corun_init_moe", "corun_init_mla", "corun_prefill", "corun_prefill_batch", "corun_decode_step", "corun_decode_enqueue", "corun_decode_wait",
    "corun_release", "corun_destroy", "corun_get_logits", "corun_force_token", "corun_context_len",
    "corun_free_blocks", "corun_debug_kv_read", "corun_debug_kv_write", "corun_debug_adopt",
    "corun_debug_set_eager", "corun_debug_read", "corun_debug_kv_fill", "corun_debug_time_kernel", "corun_decode_launches", "corun_debug_gemm", "corun_debug_gemm_pair", "corun_debug_gemm_experts", "corun_debug_prefill_attention", "corun_debug_variate",
    "corun_debug_sample", "corun_debug_wait_probe", "corun_debug_microbench", "corun_debug_check_index", "corun_gemm_static", "corun_strerror", "corun_last_cuda_error", "corun_engine_info",
    "corun_sched_create", "corun_sched_create_for_engine", "corun_sched_destroy", "corun_sched_submit",
    "corun_sched_step", "corun_sched_poll", "corun_sched_slot_of", "corun_sched_counts",
    "corun_sched_enable_batched_prefill", "corun_prefill_geometry", "corun_prefill_class",
    "corun_moe_create", "corun_moe_destroy", "corun_moe_forward", "corun_moe_sync", "corun_moe_weight_bytes",
    "corun_moe_launches", "corun_mla_attend", "corun_mla_workspace_floats", "corun_mla_sync",
]


# kernel timelines: present only in a library built with CORUN_BUILD_DEBUG=1 (include/corun_debug.h)
DEBUG_EXPORTS = ["corun_debug_gemm_trace", "corun_debug_attn_trace", "corun_debug_step_trace"]


def _need_debug_build():
    if not hasattr(lib(), "corun_debug_step_trace"):
        raise RuntimeError("kernel timelines need a library built with CORUN_BUILD_DEBUG=1 "
                           "(CORUN_BUILD_DEBUG=1 python -m paper_2608_14376_b200.build --force)")


class MoeShape(C.Structure):
    _fields_ = [("hidden", C.c_int32), ("n_experts", C.c_int32), ("top_k", C.c_int32), ("expert_ffn", C.c_int32),
                ("n_shared", C.c_int32), ("renormalize", C.c_int32)]


class MoeLayers(C.Structure):
    """``corun_moe_layers``."""
    _fields_ = [("n_experts", C.c_int32), ("top_k", C.c_int32), ("expert_ffn", C.c_int32), ("n_shared", C.c_int32),
                ("renormalize", C.c_int32), ("router", C.POINTER(C.c_void_p)), ("gate_up", C.POINTER(C.c_void_p)),
                ("down", C.POINTER(C.c_void_p))]


class MlaLayers(C.Structure):
    """``corun_mla_layers``."""
    _fields_ = [("kv_lora_rank", C.c_int32), ("qk_nope", C.c_int32), ("qk_rope", C.c_int32), ("v_head", C.c_int32),
                ("first_dense", C.c_int32), ("kv_norm", C.POINTER(C.c_void_p)), ("wkv_b", C.POINTER(C.c_void_p))]


class CorunError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        msg = lib().corun_strerror(status).decode()
        extra = f" (cuda error {lib().corun_last_cuda_error()})" if status == ECUDA else ""
        super().__init__(f"{where}: {msg}{extra} [{status}]")


class Shape(C.Structure):
    _fields_ = [(n, C.c_int32) for n in
                ("n_layers", "hidden", "n_q_heads", "n_kv_heads", "head_dim", "ffn", "vocab")] + [
        ("rms_eps", C.c_float), ("rope_theta", C.c_float), ("arch", C.c_int32)]


_PP = C.POINTER(C.c_void_p)


class Weights(C.Structure):
    _fields_ = [("embed", C.c_void_p), ("lm_head", C.c_void_p), ("final_norm", C.c_void_p),
                ("attn_norm", _PP), ("wqkv", _PP), ("wo", _PP), ("mlp_norm", _PP), ("wgate_up", _PP), ("wdown", _PP)]


class Sampling(C.Structure):
    _fields_ = [("temperature", C.c_float), ("top_p", C.c_float)]


PREFILL_FN = C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int32, C.POINTER(C.c_int32), C.c_int32, C.c_int32, C.POINTER(Sampling),
                         C.c_uint64, C.POINTER(C.c_int32))
DECODE_FN = C.CFUNCTYPE(C.c_int, C.c_void_p, C.POINTER(C.c_uint8), C.POINTER(C.c_uint64), C.POINTER(C.c_int32))
RELEASE_FN = C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int32)
FREE_BLOCKS_FN = C.CFUNCTYPE(C.c_int64, C.c_void_p)
PREFILL_BATCH_FN = C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int32, C.POINTER(C.c_int32), C.POINTER(C.c_int32),
                               C.POINTER(C.c_int32), C.POINTER(C.c_int32), C.POINTER(Sampling), C.POINTER(C.c_uint64),
                               C.POINTER(C.c_int32))


class SchedOps(C.Structure):
    """``corun_sched_ops``: the four engine calls the scheduler makes."""
    _fields_ = [("prefill", PREFILL_FN), ("decode_step", DECODE_FN), ("release", RELEASE_FN),
                ("free_blocks", FREE_BLOCKS_FN)]

SCHED_IDLE, SCHED_PREFILL, SCHED_DECODE = 0, 1, 2


_lib = None


def lib():
    """Loads libcorun.so (built in-tree by ``paper_2608_14376_b200.build``); fails loudly if absent."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(f"{LIB_PATH} is missing: run `python -m paper_2608_14376_b200.build` "
                               "(there is no fallback path)")
        L = C.CDLL(LIB_PATH)
        vp, i32, i64, u64 = C.c_void_p, C.c_int32, C.c_int64, C.c_uint64
        L.corun_init.argtypes = [C.POINTER(Shape), C.POINTER(Weights), i32, i32, i32, i64, vp, C.POINTER(vp)]
        L.corun_prefill.argtypes = [vp, i32, vp, i32, i32, C.POINTER(Sampling), u64, C.POINTER(i32)]
        L.corun_prefill_batch.argtypes = [vp, i32, vp, vp, vp, vp, vp, vp, vp]
        L.corun_decode_step.argtypes = [vp, vp, vp, vp]
        L.corun_decode_enqueue.argtypes = [vp, vp, vp]
        L.corun_decode_wait.argtypes = [vp, vp]
        L.corun_release.argtypes = [vp, i32]
        L.corun_destroy.argtypes = [vp]
        L.corun_destroy.restype = None
        L.corun_get_logits.argtypes = [vp, i32, vp]
        L.corun_force_token.argtypes = [vp, i32, i32]
        L.corun_context_len.argtypes = [vp, i32]
        L.corun_free_blocks.argtypes = [vp]
        L.corun_free_blocks.restype = i64
        L.corun_debug_kv_read.argtypes = [vp, i32, i32, i32, i32, vp, vp]
        L.corun_debug_kv_write.argtypes = [vp, i32, i32, i32, i32, vp, vp]
        L.corun_debug_adopt.argtypes = [vp, i32, i32, i32, i32, C.POINTER(Sampling), i32]
        L.corun_debug_set_eager.argtypes = [vp, i32]
        L.corun_debug_read.argtypes = [vp, i32, vp, i64]
        if hasattr(L, "corun_debug_step_trace"):              # a library built with CORUN_BUILD_DEBUG=1
            L.corun_debug_gemm_trace.argtypes = [vp, i32, i32, vp, C.POINTER(i32)]
            L.corun_debug_attn_trace.argtypes = [vp, i32, vp, C.POINTER(i32)]
            L.corun_debug_step_trace.argtypes = [vp, vp, i64]
        L.corun_debug_kv_fill.argtypes = [vp, i32, i32, C.c_float, u64]
        L.corun_debug_time_kernel.argtypes = [vp, i32, i32, C.POINTER(C.c_float)]
        L.corun_decode_launches.argtypes = [vp]
        L.corun_debug_gemm.argtypes = [vp, i32, i32, vp, i32, vp, vp]
        L.corun_prefill_class.argtypes = [vp, i32, C.POINTER(i32), C.POINTER(i32), C.POINTER(i32)]
        L.corun_debug_gemm_pair.argtypes = [i32, vp, i32, i32, vp, i32, vp, vp]
        L.corun_debug_gemm_experts.argtypes = [i32, vp, i32, i32, i32, vp, vp, vp, vp, vp]
        L.corun_debug_prefill_attention.argtypes = [vp, i32, i32, i32, i32, vp, vp]
        L.corun_debug_variate.argtypes = [u64, u64, C.POINTER(C.c_uint32)]
        L.corun_debug_sample.argtypes = [vp, i32, i32, C.POINTER(Sampling), vp, vp]
        L.corun_gemm_static.argtypes = [vp, i32, i32, vp, i32, vp, vp]
        L.corun_strerror.argtypes = [C.c_int]
        L.corun_strerror.restype = C.c_char_p
        L.corun_last_cuda_error.argtypes = []
        L.corun_engine_info.argtypes = [vp, C.POINTER(i32), C.POINTER(i32), C.POINTER(i32), C.POINTER(i64)]
        L.corun_sched_create.argtypes = [C.POINTER(SchedOps), vp, i32, i32, i32, C.POINTER(vp)]
        L.corun_sched_create_for_engine.argtypes = [vp, C.POINTER(vp)]
        L.corun_sched_destroy.argtypes = [vp]
        L.corun_sched_destroy.restype = None
        L.corun_sched_submit.argtypes = [vp, vp, i32, i32, C.POINTER(Sampling), u64, C.POINTER(i64)]
        L.corun_sched_step.argtypes = [vp, C.POINTER(i32), C.POINTER(i64), C.POINTER(i32)]
        L.corun_sched_poll.argtypes = [vp, i64, vp, i32, C.POINTER(i32), C.POINTER(i32)]
        L.corun_sched_slot_of.argtypes = [vp, i64, C.POINTER(i32)]
        L.corun_sched_counts.argtypes = [vp, C.POINTER(i32), C.POINTER(i32)]
        L.corun_moe_create.argtypes = [C.POINTER(MoeShape), vp, vp, vp, i32, vp, C.POINTER(vp)]
        L.corun_moe_destroy.argtypes = [vp]
        L.corun_moe_destroy.restype = None
        L.corun_moe_forward.argtypes = [vp, vp, vp, vp, vp]
        L.corun_moe_sync.argtypes = [vp]
        L.corun_moe_weight_bytes.argtypes = [vp]
        L.corun_moe_weight_bytes.restype = i64
        L.corun_moe_launches.argtypes = [vp]
        for n in EXPORTS:
            getattr(L, n)
        _lib = L
    return _lib


def _check(rc: int, where: str):
    if rc != OK:
        raise CorunError(rc, where)


class Engine:
    """One engine = one fixed decode shape (B, max_context) on the current CUDA device.

    ``weights``: dict of torch bf16 CUDA tensors laid out as ``corun_weights``
    describes (see ``synth.make_weights_*``); they are borrowed, keep them alive.
    """

    def __init__(self, shape, weights: dict, B: int, max_context: int, kv_pool_blocks: int = 0, stream=None, moe: dict = None,
                 mla: dict = None, kv_block: int = 16):
        """``moe``: Mixture-of-Experts feed-forward layers instead of the dense ones: a dict with n_experts, top_k,
        expert_ffn, n_shared, renormalize and lists of L CUDA bf16 tensors router [E, H], gate_up [(E+S)*2F, H],
        down [H, (E+S)*F] (``weights`` then needs no wgate_up / wdown).
        ``mla``: multi-head latent attention layers (``corun_init_mla``): a dict with kv_lora_rank, qk_nope, qk_rope,
        v_head, first_dense and lists of L CUDA bf16 tensors kv_norm [rank], wkv_b [nh*(nope+v), rank]; wqkv / wo of
        ``weights`` then have the MLA shapes, layers below first_dense are dense (wgate_up / wdown entries; None for
        the other layers), the others take ``moe`` (its entries below first_dense may be None).
        ``kv_block``: tokens per cache block: 16, or (``mla`` only) 64: the 16-token pages of a slot then come in aligned
        runs of four and the latent attention fetches a run with one TMA box; ``kv_pool_blocks`` counts these blocks."""
        import torch

        self._torch = torch
        self.shape, self.B, self.max_context = shape, B, max_context
        self._weights = weights
        d = shape.dict() if hasattr(shape, "dict") else dict(shape)
        self._cs = Shape(d["n_layers"], d["hidden"], d["n_q_heads"], d["n_kv_heads"], d["head_dim"], d["ffn"],
                         d["vocab"], d["rms_eps"], d["rope_theta"], 0)
        cw = Weights()
        self._arrs = {}
        for k in ("embed", "lm_head", "final_norm"):
            t = weights[k]
            assert t.is_cuda and t.dtype == torch.bfloat16 and t.is_contiguous()
            setattr(cw, k, t.data_ptr())
        def ptr_array(ts):
            assert len(ts) == d["n_layers"]
            for t in ts:
                assert t is None or (t.is_cuda and t.dtype == torch.bfloat16 and t.is_contiguous())
            return (C.c_void_p * len(ts))(*[(t.data_ptr() if t is not None else None) for t in ts])

        dense_needed = (not moe) or (mla is not None and mla["first_dense"] > 0)
        for k in ("attn_norm", "wqkv", "wo", "mlp_norm") + (("wgate_up", "wdown") if dense_needed else ()):
            arr = ptr_array(weights[k])
            self._arrs[k] = arr
            setattr(cw, k, C.cast(arr, _PP))
        self._cw = cw
        torch.cuda.synchronize()
        h = C.c_void_p()
        cm = None
        if moe:
            cm = MoeLayers(moe["n_experts"], moe["top_k"], moe["expert_ffn"], moe["n_shared"], 1 if moe.get("renormalize") else 0)
            self._moe = moe
            for k in ("router", "gate_up", "down"):
                arr = ptr_array(moe[k])
                self._arrs["moe_" + k] = arr
                setattr(cm, k, C.cast(arr, _PP))
        if mla is not None:
            cl = MlaLayers(mla["kv_lora_rank"], mla["qk_nope"], mla["qk_rope"], mla["v_head"], mla["first_dense"])
            self._mla = mla
            for k in ("kv_norm", "wkv_b"):
                arr = ptr_array(mla[k])
                self._arrs["mla_" + k] = arr
                setattr(cl, k, C.cast(arr, _PP))
            L = lib()
            L.corun_init_mla.argtypes = [C.POINTER(Shape), C.POINTER(Weights), C.POINTER(MlaLayers), C.POINTER(MoeLayers), C.c_int32,
                                         C.c_int32, C.c_int32, C.c_int64, C.c_void_p, C.POINTER(C.c_void_p)]
            _check(L.corun_init_mla(C.byref(self._cs), C.byref(cw), C.byref(cl), C.byref(cm) if cm is not None else None, B,
                                    max_context, kv_block, kv_pool_blocks, C.c_void_p(stream) if stream else None, C.byref(h)),
                   "corun_init_mla")
        elif moe:
            L = lib()
            L.corun_init_moe.argtypes = [C.POINTER(Shape), C.POINTER(Weights), C.POINTER(MoeLayers), C.c_int32, C.c_int32,
                                         C.c_int32, C.c_int64, C.c_void_p, C.POINTER(C.c_void_p)]
            _check(L.corun_init_moe(C.byref(self._cs), C.byref(cw), C.byref(cm), B, max_context, 16, kv_pool_blocks,
                                    C.c_void_p(stream) if stream else None, C.byref(h)), "corun_init_moe")
        else:
            _check(lib().corun_init(C.byref(self._cs), C.byref(cw), B, max_context, 16, kv_pool_blocks,
                                    C.c_void_p(stream) if stream else None, C.byref(h)), "corun_init")
        self._h = h
        self.vocab = d["vocab"]

    def close(self):
        if getattr(self, "_h", None):
            lib().corun_destroy(self._h)
            self._h = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    # -- the four calls of the boundary
    def prefill(self, slot: int, tokens, reserve_len: int, temperature: float = 0.0, top_p: float = 1.0,
                seed: int = 0) -> int:
        t = np.ascontiguousarray(tokens, dtype=np.int32)
        s = Sampling(temperature, top_p)
        first = C.c_int32(-1)
        _check(lib().corun_prefill(self._h, slot, t.ctypes.data, t.shape[0], reserve_len, C.byref(s),
                                   seed & (2**64 - 1), C.byref(first)), "corun_prefill")
        return int(first.value)

    def prefill_batch(self, slots, prompts, reserve_lens, temperature: float = 0.0, top_p: float = 1.0, seeds=None) -> np.ndarray:
        """Prefill of several requests in shared chunks; returns their first tokens."""
        n = len(slots)
        sl = np.ascontiguousarray(slots, dtype=np.int32)
        lens = np.ascontiguousarray([len(p) for p in prompts], dtype=np.int32)
        toks = np.ascontiguousarray(np.concatenate([np.asarray(p, dtype=np.int32) for p in prompts]), dtype=np.int32)
        res = np.ascontiguousarray(reserve_lens, dtype=np.int32)
        smp = (Sampling * n)(*[Sampling(temperature, top_p) for _ in range(n)])
        sd = np.ascontiguousarray(seeds if seeds is not None else np.zeros(n), dtype=np.uint64)
        out = np.full(n, -1, np.int32)
        assert sl.shape == lens.shape == res.shape == sd.shape == (n,)
        _check(lib().corun_prefill_batch(self._h, n, sl.ctypes.data, toks.ctypes.data, lens.ctypes.data, res.ctypes.data,
                                         C.cast(smp, C.c_void_p), sd.ctypes.data, out.ctypes.data), "corun_prefill_batch")
        return out

    def decode_step(self, active, seeds) -> np.ndarray:
        a = np.ascontiguousarray(active, dtype=np.uint8)
        s = np.ascontiguousarray(seeds, dtype=np.uint64)
        assert a.shape == (self.B,) and s.shape == (self.B,)
        out = np.empty(self.B, np.int32)
        _check(lib().corun_decode_step(self._h, a.ctypes.data, s.ctypes.data, out.ctypes.data), "corun_decode_step")
        return out

    def decode_enqueue(self, active, seeds):
        a = np.ascontiguousarray(active, dtype=np.uint8)
        s = np.ascontiguousarray(seeds, dtype=np.uint64)
        _check(lib().corun_decode_enqueue(self._h, a.ctypes.data, s.ctypes.data), "corun_decode_enqueue")

    def decode_wait(self) -> np.ndarray:
        out = np.empty(self.B, np.int32)
        _check(lib().corun_decode_wait(self._h, out.ctypes.data), "corun_decode_wait")
        return out

    def release(self, slot: int):
        _check(lib().corun_release(self._h, slot), "corun_release")

    # -- accessors
    def logits(self, slot: int) -> np.ndarray:
        out = np.empty(self.vocab, np.float32)
        _check(lib().corun_get_logits(self._h, slot, out.ctypes.data), "corun_get_logits")
        return out

    def force_token(self, slot: int, token: int):
        _check(lib().corun_force_token(self._h, slot, int(token)), "corun_force_token")

    def prefill_class(self, n_tokens: int):
        """(class, rows to count as a chunk, tile rows) of prompts of that length (``corun_prefill_class``)."""
        c, ch, t = C.c_int32(-1), C.c_int32(-1), C.c_int32(-1)
        _check(lib().corun_prefill_class(self._h, n_tokens, C.byref(c), C.byref(ch), C.byref(t)), "corun_prefill_class")
        return c.value, ch.value, t.value

    def context_len(self, slot: int) -> int:
        rc = lib().corun_context_len(self._h, slot)
        if rc < 0:
            raise CorunError(rc, "corun_context_len")
        return rc

    def free_blocks(self) -> int:
        return int(lib().corun_free_blocks(self._h))

    def kv_read(self, slot: int, layer: int, pos0: int, n: int):
        if getattr(self, "_mla", None):                   # latent cache: rows of rank + rope values, no second array
            k = np.empty((n, self._mla["kv_lora_rank"] + self._mla["qk_rope"]), np.float32)
            _check(lib().corun_debug_kv_read(self._h, slot, layer, pos0, n, k.ctypes.data, None), "kv_read")
            return k, None
        kd = self._cs.n_kv_heads * self._cs.head_dim
        k = np.empty((n, kd), np.float32)
        v = np.empty((n, kd), np.float32)
        _check(lib().corun_debug_kv_read(self._h, slot, layer, pos0, n, k.ctypes.data, v.ctypes.data), "kv_read")
        return k, v

    def kv_write(self, slot: int, layer: int, pos0: int, k, v):
        k = np.ascontiguousarray(k, dtype=np.float32)
        if v is None:                                     # latent cache
            _check(lib().corun_debug_kv_write(self._h, slot, layer, pos0, k.shape[0], k.ctypes.data, None), "kv_write")
            return
        v = np.ascontiguousarray(v, dtype=np.float32)
        _check(lib().corun_debug_kv_write(self._h, slot, layer, pos0, k.shape[0], k.ctypes.data, v.ctypes.data),
               "kv_write")

    def adopt(self, slot: int, n_ctx: int, reserve_len: int, pending: int, temperature=0.0, top_p=1.0, step=1):
        s = Sampling(temperature, top_p)
        _check(lib().corun_debug_adopt(self._h, slot, n_ctx, reserve_len, pending, C.byref(s), step), "adopt")

    def kv_fill(self, slot: int, n_ctx: int, std: float, seed: int):
        _check(lib().corun_debug_kv_fill(self._h, slot, n_ctx, std, seed & (2**64 - 1)), "kv_fill")

    KERNEL_KINDS = ("gemm_qkv", "gemm_o", "gemm_gate_up", "gemm_down", "gemm_lm_head", "attention",
                    "resid_norm", "rope_kv_append", "swiglu", "sampler")
    # further kinds of corun_debug_time_kernel: engines with multi-head latent attention / with expert layers
    MLA_KERNEL_KINDS = {"mla_up_k": 10, "mla_up_v": 11}
    MOE_KERNEL_KINDS = {"moe_router": 12}
    MOE_GROUPED_KERNEL_KINDS = {"moe_group_gather": 13}   # decode programs with more than 64 padded rows

    def time_kernel(self, kind: int, reps: int) -> float:
        ms = C.c_float(0.0)
        _check(lib().corun_debug_time_kernel(self._h, kind, reps, C.byref(ms)), "time_kernel")
        return float(ms.value)

    def gemm_trace(self, kind: int, layer: int = 0) -> np.ndarray:
        """Per-CTA timeline [n_ctas, 8] (ns, relative to the earliest kernel entry) of one GEMM launch."""
        st = np.zeros(8 * 256, np.uint64)
        n = C.c_int32(0)
        _need_debug_build()
        _check(lib().corun_debug_gemm_trace(self._h, kind, layer, st.ctypes.data, C.byref(n)), "gemm_trace")
        t = st[:8 * n.value].reshape(n.value, 8).astype(np.int64)
        return t - t[:, 0].min()

    def step_trace(self, n_sms: int = 148) -> np.ndarray:
        """GEMM timelines of the last decode step, [4 * n_layers, n_sms, 8] ns (engine made with CORUN_TRACE_STEP=1)."""
        n = 4 * self._cs.n_layers * n_sms * 8
        st = np.zeros(n, np.uint64)
        _need_debug_build()
        _check(lib().corun_debug_step_trace(self._h, st.ctypes.data, n), "step_trace")
        return st.reshape(4 * self._cs.n_layers, n_sms, 8).astype(np.int64)

    def attn_trace(self, layer: int = 0) -> np.ndarray:
        """Per-CTA, per-item attention timeline [n_ctas, 64, 8] in ns (0 where an item does not exist)."""
        st = np.zeros(256 * 64 * 8, np.uint64)
        n = C.c_int32(0)
        _need_debug_build()
        _check(lib().corun_debug_attn_trace(self._h, layer, st.ctypes.data, C.byref(n)), "attn_trace")
        return st[:n.value * 512].reshape(n.value, 64, 8).astype(np.int64)

    def debug_read(self, which: int, n: int) -> np.ndarray:
        out = np.empty(n, np.float32)
        _check(lib().corun_debug_read(self._h, which, out.ctypes.data, n), "corun_debug_read")
        return out

    def prefill_attention(self, slot: int, layer: int, pos0: int, q) -> np.ndarray:
        """The long prompts' attention kernel for query rows q [n, heads, dims] at positions pos0 .."""
        q = np.ascontiguousarray(q, dtype=np.float32)
        out = np.empty(q.shape[:2] + (self._mla["v_head"] if getattr(self, "_mla", None) else q.shape[2],), np.float32)
        _check(lib().corun_debug_prefill_attention(self._h, slot, layer, pos0, q.shape[0], q.ctypes.data, out.ctypes.data),
               "corun_debug_prefill_attention")
        return out

    def set_eager(self, eager: bool):
        _check(lib().corun_debug_set_eager(self._h, int(eager)), "set_eager")

    def decode_launches(self) -> int:
        return int(lib().corun_decode_launches(self._h))


class Scheduler:
    """Host scheduler (isolated prefill in front of the padded decode iteration) around an
    ``Engine``, or around a table of callbacks standing in for one (``ops``: a ``SchedOps`` whose
    callbacks the caller keeps alive, with ``B``, ``kv_block`` and ``max_context``)."""

    def __init__(self, engine: "Engine" = None, ops: SchedOps = None, B: int = 0, kv_block: int = 16,
                 max_context: int = 0):
        h = C.c_void_p()
        if engine is not None:
            _check(lib().corun_sched_create_for_engine(engine._h, C.byref(h)), "corun_sched_create_for_engine")
        else:
            _check(lib().corun_sched_create(C.byref(ops), None, B, kv_block, max_context, C.byref(h)), "corun_sched_create")
        self._h, self._keep = h, (engine, ops)

    def close(self):
        if self._h:
            lib().corun_sched_destroy(self._h)
            self._h = None

    def enable_batched_prefill(self, fn=None, chunk_rows: int = 0, tile_rows: int = 0):
        """Prefill decisions take the requests behind the head that fit into the padding of the head's chunks
        (``fn``: a PREFILL_BATCH_FN for a stand-in engine; None = the engine's corun_prefill_batch)."""
        self._batch_fn = fn                                   # keep the callback alive
        L = lib()
        L.corun_sched_enable_batched_prefill.argtypes = [C.c_void_p, C.c_void_p, C.c_int32, C.c_int32]
        _check(L.corun_sched_enable_batched_prefill(self._h, C.cast(fn, C.c_void_p) if fn is not None else None,
                                                    chunk_rows, tile_rows), "corun_sched_enable_batched_prefill")

    def submit(self, prompt, max_new_tokens: int, temperature: float = 0.0, top_p: float = 1.0, seed: int = 0) -> int:
        t = np.ascontiguousarray(prompt, dtype=np.int32)
        s = Sampling(temperature, top_p)
        rid = C.c_int64(-1)
        _check(lib().corun_sched_submit(self._h, t.ctypes.data, t.shape[0], max_new_tokens, C.byref(s),
                                        seed & (2**64 - 1), C.byref(rid)), "corun_sched_submit")
        return int(rid.value)

    def step(self):
        """One scheduling decision -> (action, request id of a prefill or -1, requests that took part)."""
        a, rid, n = C.c_int32(0), C.c_int64(-1), C.c_int32(0)
        _check(lib().corun_sched_step(self._h, C.byref(a), C.byref(rid), C.byref(n)), "corun_sched_step")
        return int(a.value), int(rid.value), int(n.value)

    def poll(self, rid: int):
        """-> (tokens produced so far, finished?)"""
        n, fin = C.c_int32(0), C.c_int32(0)
        _check(lib().corun_sched_poll(self._h, rid, None, 0, C.byref(n), C.byref(fin)), "corun_sched_poll")
        out = np.empty(max(1, n.value), np.int32)
        _check(lib().corun_sched_poll(self._h, rid, out.ctypes.data, n.value, C.byref(n), C.byref(fin)), "corun_sched_poll")
        return out[:n.value].copy(), bool(fin.value)

    def slot_of(self, rid: int) -> int:
        s = C.c_int32(-1)
        _check(lib().corun_sched_slot_of(self._h, rid, C.byref(s)), "corun_sched_slot_of")
        return int(s.value)

    def counts(self):
        w, r = C.c_int32(0), C.c_int32(0)
        _check(lib().corun_sched_counts(self._h, C.byref(w), C.byref(r)), "corun_sched_counts")
        return int(w.value), int(r.value)


def debug_gemm(W, X):
    """out[r, n] = sum_k W[n, k] X[r, k]; W torch bf16 [N, K] cuda, X torch fp32 [R, K] cuda."""
    import torch

    N, K = W.shape
    R = X.shape[0]
    out = torch.empty((R, N), dtype=torch.float32, device=X.device)
    torch.cuda.synchronize()
    _check(lib().corun_debug_gemm(W.data_ptr(), N, K, X.data_ptr(), R, out.data_ptr(), None), "corun_debug_gemm")
    return out


def debug_gemm_pair(form, W, X):
    """The GEMM on pairs of SMs (``corun_debug_gemm_pair``): form 0 plain, 1 with SwiGLU (result [R, N / 2]), 2 keys and
    values; 3, 4: 0, 1 as a decode step runs them."""
    import torch

    N, K = W.shape
    R = X.shape[0]
    out = torch.empty((R, N // 2 if form in (1, 4) else N), dtype=torch.float32, device=X.device)
    torch.cuda.synchronize()
    _check(lib().corun_debug_gemm_pair(form, W.data_ptr(), N, K, X.data_ptr(), R, out.data_ptr(), None), "corun_debug_gemm_pair")
    return out


def debug_gemm_experts(form, W, rows, X, row_w=None):
    """The GEMMs of a prompt's experts (``corun_debug_gemm_experts``), rows[e] rows of X through expert e: form 0 W [N, E K], 1 gate / up
    with SwiGLU, W [E, 2F, K]."""
    import torch

    E, K = len(rows), X.shape[1]
    N = W.shape[1] if form else W.shape[0]
    out = torch.empty((X.shape[0], N // 2 if form else N), dtype=torch.float32, device=X.device)
    counts = np.asarray(rows, np.int32)
    torch.cuda.synchronize()
    _check(lib().corun_debug_gemm_experts(form, W.data_ptr(), E, N, K, counts.ctypes.data, X.data_ptr(),
                                          row_w.data_ptr() if row_w is not None else None, out.data_ptr(), None), "corun_debug_gemm_experts")
    return out


def gemm_static(W, X):
    """Same product as ``debug_gemm`` through ``corun_gemm_static``: the library's own fixed scratch
    array is used instead of fresh allocations (for callers that must not allocate device memory).
    The output tensor is the caller's; rows <= 16, K <= 4096, N <= 8192."""
    import torch

    N, K = W.shape
    R = X.shape[0]
    out = torch.empty((R, N), dtype=torch.float32, device=X.device)
    torch.cuda.synchronize()
    _check(lib().corun_gemm_static(W.data_ptr(), N, K, X.data_ptr(), R, out.data_ptr(), None), "corun_gemm_static")
    return out


def debug_variate(seed: int, t: int) -> int:
    o = C.c_uint32(0)
    _check(lib().corun_debug_variate(seed & (2**64 - 1), t, C.byref(o)), "corun_debug_variate")
    return int(o.value)


def debug_sample(logits, temperature: float, top_p: float, u24) -> np.ndarray:
    lg = np.ascontiguousarray(logits, dtype=np.float32)
    if lg.ndim == 1:
        lg = lg[None]
    u = np.ascontiguousarray(u24, dtype=np.uint32).reshape(-1)
    assert u.shape[0] == lg.shape[0]
    out = np.empty(lg.shape[0], np.int32)
    s = Sampling(temperature, top_p)
    _check(lib().corun_debug_sample(lg.ctypes.data, lg.shape[0], lg.shape[1], C.byref(s), u.ctypes.data,
                                    out.ctypes.data), "corun_debug_sample")
    return out


class MoeFfn:
    """Mixture-of-Experts feed-forward block (``include/corun_moe.h``).  Weights are CUDA bf16 tensors:
    router [E, H], gate_up [(E + S) * 2F, H], down [H, (E + S) * F]; B padded rows per call."""

    def __init__(self, hidden: int, n_experts: int, top_k: int, expert_ffn: int, n_shared: int, router, gate_up, down,
                 B: int, renormalize: bool = False):
        import torch

        self._torch = torch
        self.B, self.H, self.top_k = B, hidden, top_k
        self._w = (router, gate_up, down)                     # keep the borrowed tensors alive
        for t in self._w:
            assert t.is_cuda and t.dtype == torch.bfloat16 and t.is_contiguous()
        assert tuple(router.shape) == (n_experts, hidden)
        assert tuple(gate_up.shape) == ((n_experts + n_shared) * 2 * expert_ffn, hidden)
        assert tuple(down.shape) == (hidden, (n_experts + n_shared) * expert_ffn)
        sh = MoeShape(hidden, n_experts, top_k, expert_ffn, n_shared, 1 if renormalize else 0)
        h = C.c_void_p()
        self._stream = torch.cuda.current_stream()
        _check(lib().corun_moe_create(C.byref(sh), router.data_ptr(), gate_up.data_ptr(), down.data_ptr(), B,
                                      self._stream.cuda_stream, C.byref(h)), "corun_moe_create")
        self._h = h

    def forward(self, x, want_routing: bool = True):
        """x: CUDA fp32 [B, H] -> (y fp32 [B, H], experts int32 [B, top_k], probs fp32 [B, top_k]); asynchronous."""
        torch = self._torch
        assert x.is_cuda and x.dtype == torch.float32 and tuple(x.shape) == (self.B, self.H) and x.is_contiguous()
        y = torch.empty_like(x)
        ex = torch.empty((self.B, self.top_k), dtype=torch.int32, device=x.device) if want_routing else None
        pr = torch.empty((self.B, self.top_k), dtype=torch.float32, device=x.device) if want_routing else None
        _check(lib().corun_moe_forward(self._h, x.data_ptr(), y.data_ptr(), ex.data_ptr() if want_routing else None,
                                       pr.data_ptr() if want_routing else None), "corun_moe_forward")
        return y, ex, pr

    def sync(self):
        _check(lib().corun_moe_sync(self._h), "corun_moe_sync")

    def weight_bytes(self) -> int:
        return int(lib().corun_moe_weight_bytes(self._h))

    def launches(self) -> int:
        return int(lib().corun_moe_launches(self._h))

    def close(self):
        if self._h:
            lib().corun_moe_destroy(self._h)
            self._h = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


class MlaAttention:
    """Absorbed multi-head latent attention for one query token per row over a paged latent cache
    (``include/corun_mla.h``) with its workspace and output allocated once: ``run`` only enqueues."""

    def __init__(self, B: int, n_heads: int, d_latent: int, d_rope: int, max_blocks: int, device="cuda"):
        import torch

        L = lib()
        L.corun_mla_workspace_floats.restype = C.c_int64
        L.corun_mla_workspace_floats.argtypes = [C.c_int32] * 4
        L.corun_mla_attend.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int64, C.c_void_p, C.c_int32, C.c_void_p] + \
            [C.c_int32] * 4 + [C.c_float, C.c_void_p, C.c_void_p, C.c_void_p]
        L.corun_mla_sync.argtypes = [C.c_void_p, C.c_void_p]
        self.shape = (B, n_heads, d_latent, d_rope, max_blocks)
        self.ws = torch.empty(int(L.corun_mla_workspace_floats(B, n_heads, d_latent, max_blocks * 16)), dtype=torch.float32, device=device)
        self.out = torch.zeros((B, n_heads, d_latent), dtype=torch.float32, device=device)

    def run(self, q_lat, q_rope, pool, block_table, ctx, scale: float):
        """q_lat fp32 [B, n_heads, d_c], q_rope fp32 [B, n_heads, d_r], pool fp16 [pool_pages, 16, d_c + d_r],
        block_table int32 [B, max_blocks], ctx int32 [B] (contiguous CUDA tensors) -> o_lat fp32 [B, n_heads, d_c]
        (rows with ctx 0 keep what they held).  Asynchronous on torch's current stream."""
        import torch

        B, nh, dc, dr, mb = self.shape
        assert tuple(q_lat.shape) == (B, nh, dc) and q_lat.dtype == torch.float32 and q_lat.is_contiguous() and q_lat.is_cuda
        assert tuple(q_rope.shape) == (B, nh, dr) and q_rope.dtype == torch.float32 and q_rope.is_contiguous()
        assert pool.dtype == torch.float16 and pool.is_contiguous() and tuple(pool.shape[1:]) == (16, dc + dr)
        assert block_table.dtype == torch.int32 and block_table.is_contiguous() and tuple(block_table.shape) == (B, mb)
        assert ctx.dtype == torch.int32 and ctx.is_contiguous() and tuple(ctx.shape) == (B,)
        st = torch.cuda.current_stream().cuda_stream
        _check(lib().corun_mla_attend(q_lat.data_ptr(), q_rope.data_ptr(), pool.data_ptr(), pool.shape[0], block_table.data_ptr(),
                                      mb, ctx.data_ptr(), B, nh, dc, dr, float(scale), self.out.data_ptr(), self.ws.data_ptr(), st),
               "corun_mla_attend")
        return self.out

    def sync(self):
        """Waits for the stream; raises if a bounded device-side wait expired."""
        import torch

        _check(lib().corun_mla_sync(self.ws.data_ptr(), torch.cuda.current_stream().cuda_stream), "corun_mla_sync")


def mla_attend(q_lat, q_rope, pool, block_table, ctx, scale: float):
    """One call of ``MlaAttention`` with fresh buffers (rows with ctx 0 come back as zeros); waits for the result."""
    op = MlaAttention(q_lat.shape[0], q_lat.shape[1], q_lat.shape[2], q_rope.shape[2], block_table.shape[1], q_lat.device)
    out = op.run(q_lat, q_rope, pool, block_table, ctx, scale)
    op.sync()
    return out


MICROBENCH_KINDS = ("rmsnorm", "softmax", "column_sum")


def microbench(kind: int, variant: int, x, reps: int = 20):
    """``corun_debug_microbench`` on a CUDA fp32 matrix x [R, N]: (y, microseconds per launch, tiling used).
    kind: index into MICROBENCH_KINDS; variant 0 = tiling fixed for every R, 1 = adapted to R."""
    import torch

    assert x.is_cuda and x.dtype == torch.float32 and x.is_contiguous() and x.dim() == 2
    R, N = x.shape
    y = torch.empty((N,) if kind == 2 else (R, N), dtype=torch.float32, device=x.device)
    us, til = C.c_float(0.0), C.c_int32(0)
    L = lib()
    L.corun_debug_microbench.argtypes = [C.c_int32, C.c_int32, C.c_void_p, C.c_int32, C.c_int32, C.c_void_p, C.c_int32,
                                         C.POINTER(C.c_float), C.POINTER(C.c_int32), C.c_void_p]
    _check(L.corun_debug_microbench(kind, variant, x.data_ptr(), R, N, y.data_ptr(), reps, C.byref(us), C.byref(til),
                                    torch.cuda.current_stream().cuda_stream), "corun_debug_microbench")
    return y, float(us.value), int(til.value)
