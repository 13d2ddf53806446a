"""PagedAttention: pool + plan + workspace of one serving instance.

torch supplies device memory and the current stream; every computation is a
call through the C ABI.
"""
from __future__ import annotations

import subprocess
import threading

from . import binding as B
from . import build

_torch_calls = None  # False: this torch has none
_torch_calls_lock = threading.Lock()


def torch_calls():
    """The extension module of the calls of every iteration that takes torch tensors, or None where it can be neither loaded nor
    built: the calls through addresses do the same, some microseconds slower."""
    global _torch_calls
    with _torch_calls_lock:
        if _torch_calls is None:
            import ctypes
            import importlib.util
            import os
            import warnings

            lib = B.load()
            try:
                path = build.build_torch_calls(build=os.environ.get("PS_ATTN_NO_BUILD") != "1")
                spec = importlib.util.spec_from_file_location(__package__ + "._torch_calls", path)
                module = importlib.util.module_from_spec(spec)
                spec.loader.exec_module(module)
                module.bind(*(ctypes.cast(f, ctypes.c_void_p).value for f in (lib.ps_kv_write, lib.ps_kv_gather, lib.ps_attn_run)))
                _torch_calls = module
            except (ImportError, OSError, subprocess.SubprocessError) as e:
                warnings.warn("the calls with tensors go through addresses: %s" % e, RuntimeWarning)
                _torch_calls = False
    return _torch_calls or None


def take_tensors(pa):
    """The class whose instances `pa` hands to the extension: torch.Tensor itself, or none."""
    pa._tensor_calls = torch_calls()
    pa._tensor = pa.torch.Tensor if pa._tensor_calls else object()  # (the class of nothing)


class PagedAttention:
    """A paged K/V pool with the per-iteration plan / run cycle.

    >>> pa = PagedAttention(32, 8, 128, num_pages)
    >>> pa.write(k_new, v_new, block_table_dev, prior, q_len)   # cache the new tokens
    >>> pa.plan(prior, q_len, max_pages)                        # host partition
    >>> out, lse = pa.run(q, block_table_dev)                   # attention
    """

    def __init__(self, n_q_heads, n_kv_heads, head_dim, num_pages, page_size=16, device="cuda", poison=False, kv_dtype=0):
        """``kv_dtype``: 0 = bf16 cache, 1 = FP8 (E4M3) cache with a scale per (token, kv head); see ps_shape."""
        import torch

        self.torch = torch
        self._calls = B.calls()
        take_tensors(self)
        self.device = torch.device(device)
        self.shape = B.make_shape(n_q_heads, n_kv_heads, head_dim, page_size, kv_dtype)
        self.num_pages = int(num_pages)
        nbytes = B.ps_kv_bytes(self.shape, self.num_pages)
        # 0xFF bytes are bf16 NaN: any read of a slot nobody wrote shows in the output
        if poison:
            self.pool = torch.full((nbytes + 1024,), 0xFF, dtype=torch.uint8, device=self.device)
        else:
            self.pool = torch.empty((nbytes + 1024,), dtype=torch.uint8, device=self.device)
        base = (self.pool.data_ptr() + 1023) // 1024 * 1024  # the pool must start on a 1024-byte boundary
        self.kv = B.ps_kv_alloc(self.shape, self.num_pages, base, nbytes)
        self._plan = None
        self._ws = None
        self._ws_bytes = 0
        self._ws_ptr = 0
        self._total_q = 0
        self._n_q_heads = int(n_q_heads)
        index = self.pool.device.index
        raw = getattr(torch._C, "_cuda_getCurrentRawStream", None)  # (a tenth of the time that current_stream() takes)
        self._stream = (lambda: raw(index)) if raw else (lambda: torch.cuda.current_stream(index).cuda_stream)

    def close(self):
        if self._plan is not None:
            B.ps_plan_free(self._plan)
            self._plan = None
        if self.kv is not None:
            B.ps_kv_free(self.kv)
            self.kv = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    def write(self, k_new, v_new, block_table_dev, prior, q_len, max_pages=None):
        """Scatter new tokens' K, V (bf16 [T, Hkv, d]) into their pages."""
        t = self._tensor
        if type(k_new) is t and type(v_new) is t and type(block_table_dev) is t:
            B._check(self._tensor_calls.write(self.kv, k_new, v_new, block_table_dev, None if max_pages is None else int(max_pages), B.lengths(prior),
                                              B.lengths(q_len), self._stream()))
            return
        if max_pages is None:
            max_pages = block_table_dev.size(-1)
        assert k_new.is_contiguous() and v_new.is_contiguous() and block_table_dev.is_contiguous()
        B._check(self._calls.kv_write(self.kv, k_new.data_ptr(), v_new.data_ptr(), block_table_dev.data_ptr(), int(max_pages), B.lengths(prior),
                                     B.lengths(q_len), self._stream()))

    def gather_fp8(self, block_table_row_dev, length):
        """FP8 cache: logical tokens [0, length) of one sequence as (K codes, V codes) uint8 [length, Hkv, d] and
        (K scales, V scales) float32 [length, Hkv]."""
        t = self.torch
        kc = t.empty((length, self.shape.n_kv_heads, self.shape.head_dim), dtype=t.uint8, device=self.device)
        vc = t.empty_like(kc)
        ks = t.empty((length, self.shape.n_kv_heads), dtype=t.float32, device=self.device)
        vs = t.empty_like(ks)
        B.ps_kv_gather_fp8(self.kv, block_table_row_dev, int(length), kc, vc, ks, vs, self._stream())
        return kc, vc, ks, vs

    def gather(self, block_table_row_dev, length):
        """Logical tokens [0, length) of one sequence as contiguous (K, V) bf16 [length, Hkv, d] (bf16 cache)."""
        t = self.torch
        assert self.shape.dtype == 0, "use gather_fp8 on an FP8 cache"
        hkv, d = self.shape.n_kv_heads, self.shape.head_dim
        if type(block_table_row_dev) is self._tensor:
            status, k, v = self._tensor_calls.gather(self.kv, block_table_row_dev, length, hkv, d, self.pool, self._stream())
            B._check(status)
            return k, v
        k = t.empty_strided((length, hkv, d), (hkv * d, d, 1), dtype=t.bfloat16, device=self.device)
        v = t.empty_like(k)
        B.ps_kv_gather(self.kv, block_table_row_dev, int(length), k.data_ptr(), v.data_ptr(), self._stream())
        return k, v

    def check_pool(self):
        B.ps_kv_status(self.kv, self._stream())

    def plan(self, prior, q_len, max_pages, opts=None):
        """Partition the batch; grows the workspace if the plan needs more."""
        self._plan, need = B.ps_attn_plan(self.shape, prior, q_len, int(max_pages), opts, self._plan)
        if need > self._ws_bytes:
            self._ws = self.torch.empty(int(need * 1.25) + 256, dtype=self.torch.uint8, device=self.device)
            self._ws_bytes = self._ws.numel()
            self._ws_ptr = self._ws.data_ptr()
        info = B.ps_plan_get_info(self._plan)
        self._total_q = info.total_q_tokens
        return info

    def items(self):
        return B.ps_plan_get_items(self._plan)

    def run(self, q, block_table_dev, out=None, lse=None, want_lse=True):
        """Attention for the planned batch.  q: bf16 [T, Hq, d].  Returns (out, lse)."""
        t = self.torch
        assert self._plan is not None, "call plan() first"
        total_q, hq = self._total_q, self._n_q_heads
        exact = self._tensor
        if type(q) is exact and type(block_table_dev) is exact and (out is None or type(out) is exact) and (lse is None or type(lse) is exact):
            status, out, lse = self._tensor_calls.run(self._plan, self.kv, q, block_table_dev, out, lse, bool(want_lse), total_q, hq, self.pool, self._ws_ptr,
                                                      self._ws_bytes, self._stream())
            B._check(status)
            return out, lse
        assert q.is_contiguous() and q.size(0) == total_q and block_table_dev.is_contiguous()
        if out is None:
            out = t.empty_like(q)
        if lse is None and want_lse:
            lse = t.empty_strided((total_q, hq), (hq, 1), dtype=t.float32, device=self.device)  # (two thirds of empty()'s time)
        B._check(self._calls.attn_run(self._plan, self.kv, q.data_ptr(), block_table_dev.data_ptr(), out.data_ptr(), None if lse is None else lse.data_ptr(),
                                     self._ws_ptr, self._ws_bytes, self._stream()))
        return out, lse

    def check(self):
        """Synchronise and raise if the last run saw a device-side error."""
        B.ps_plan_status(self._plan, self._stream())
