"""The calls of csrc/binding.cpp through ctypes: same names, same positional arguments, same results.  binding.py uses them where
the native module has not been built for the running torch and Python; a call takes 6 to 20 us of host time instead of 1 to 5."""
from __future__ import annotations

import ctypes

import torch

from . import binding as B

_ref = ctypes.byref


def _bytes(t: torch.Tensor) -> int:
    return t.numel() * t.element_size()


def _require(ok: bool, what: str) -> None:
    if not ok:
        raise AssertionError(what)


def plan_init(geom, batch, plan, order, kept_count, query_start, score_accum, stream):
    return B.load_library().cf_plan_init_scores(_ref(geom), _ref(batch), B._ptr(order), B._ptr(kept_count), query_start,
                                                B._ptr(score_accum), plan.data_ptr(), _bytes(plan), B._stream(stream))


def prune_topk(geom, batch, plan, score_accum, keep, keep_per_request, strategy, stream):
    return B.load_library().cf_prune_topk(_ref(geom), _ref(batch), plan.data_ptr(), score_accum.data_ptr(), keep,
                                          B._ptr(keep_per_request), strategy, B._stream(stream))


def reposition_keys(geom, batch, plan, k_in, k_out, n_layers, layer_stride, stream):
    return B.load_library().cf_reposition_keys(_ref(geom), _ref(batch), plan.data_ptr(), n_layers, layer_stride, k_in.data_ptr(),
                                               k_out.data_ptr(), B._stream(stream))


def query_prefill_attn(geom, batch, plan, q, k, v, out, workspace, lse, doc_scores, score_accum, scale, stream):
    return B.load_library().cf_query_prefill_attn(_ref(geom), _ref(batch), plan.data_ptr(), q.data_ptr(), k.data_ptr(), v.data_ptr(),
                                                  scale, out.data_ptr(), B._ptr(lse), B._ptr(doc_scores), B._ptr(score_accum),
                                                  workspace.data_ptr(), _bytes(workspace), B._stream(stream))


def query_prefill_attn_slot(geom, batch, plan, slot, n_slots, q, k, v, out, workspace, lse, scale, stream):
    return B.load_library().cf_query_prefill_attn_slot(_ref(geom), _ref(batch), plan.data_ptr(), slot, n_slots, q.data_ptr(),
                                                       k.data_ptr(), v.data_ptr(), scale, out.data_ptr(), B._ptr(lse),
                                                       workspace.data_ptr(), _bytes(workspace), B._stream(stream))


def accumulate_scores(geom, batch, plan, n_filled, n_slots, workspace, doc_scores, score_accum, stream):
    return B.load_library().cf_accumulate_scores(_ref(geom), _ref(batch), plan.data_ptr(), n_filled, n_slots, B._ptr(doc_scores),
                                                 B._ptr(score_accum), workspace.data_ptr(), _bytes(workspace), B._stream(stream))


def assemble_final_cache(geom, batch, plan, k, v, k_self, v_self, k_out, v_out, final_rows, stream):
    _require(k_out.is_contiguous() and v_out.is_contiguous() and k_out.shape == v_out.shape, "k_out and v_out: contiguous, of one shape")
    _require(final_rows.dtype == torch.int32 and k.stride(0) == v.stride(0), "final_rows: int32; k_cache and v_cache: one layer stride")
    return B.load_library().cf_assemble_final_cache(_ref(geom), _ref(batch), plan.data_ptr(), k.shape[0], k.stride(0), k.data_ptr(),
                                                    v.data_ptr(), k_self.stride(0), k_self.data_ptr(), v_self.data_ptr(),
                                                    k_out.shape[2], k_out.data_ptr(), v_out.data_ptr(), final_rows.data_ptr(),
                                                    B._stream(stream))


def document_prefill_attn(geom, doc_offsets, max_doc_len, q, k, v, out, k_prefix, v_prefix, lse, scale, token_stride, status, stream):
    n = q.shape[0]
    _require(doc_offsets.dtype == torch.int32 and doc_offsets.is_contiguous(), "doc_offsets: contiguous int32")
    _require(k.shape[0] == n and v.shape[0] == n and out.shape[0] == n, "q, k, v and out: one number of layers")
    _require(k.stride(0) == v.stride(0) and (lse is None or lse.is_contiguous()), "k and v: one layer stride; lse: contiguous")
    prefix = 0 if k_prefix is None else k_prefix.shape[1]
    _require(prefix == 0 or (v_prefix is not None and k_prefix.stride(0) == v_prefix.stride(0)), "k_prefix and v_prefix: one layer stride")
    docs = B.cf_doc_batch(doc_offsets.numel() - 1, max_doc_len, prefix, 0, q.shape[1],
                          k.shape[2] * k.shape[3] if token_stride is None else token_stride, doc_offsets.data_ptr())
    return B.load_library().cf_document_prefill_attn(_ref(geom), _ref(docs), n, q.data_ptr(), q.stride(0), k.data_ptr(), v.data_ptr(),
                                                     k.stride(0), B._ptr(k_prefix) if prefix else None,
                                                     B._ptr(v_prefix) if prefix else None, k_prefix.stride(0) if prefix else 0, scale,
                                                     out.data_ptr(), out.stride(0), B._ptr(lse), B._ptr(status), B._stream(stream))


def decode_plan(geom, n_requests, cache_rows, rows, extra_rows, plan, stream):
    return B.load_library().cf_decode_plan(_ref(geom), n_requests, cache_rows, rows.data_ptr(), extra_rows, plan.data_ptr(),
                                           _bytes(plan), B._stream(stream))


def decode_attn(geom, n_requests, cache_rows, plan, q, k, v, out, workspace, lse, scale, stream):
    n = q.shape[0]
    _require(k.shape[0] == n and v.shape[0] == n and out.shape[0] == n, "q, k_final, v_final and out: one number of layers")
    _require(k.stride(0) == v.stride(0) and (lse is None or lse.is_contiguous()), "k_final and v_final: one layer stride; lse: contiguous")
    return B.load_library().cf_decode_attn(_ref(geom), n_requests, cache_rows, plan.data_ptr(), n, q.data_ptr(), q.stride(0),
                                           k.data_ptr(), v.data_ptr(), k.stride(0), scale, out.data_ptr(), out.stride(0), B._ptr(lse),
                                           workspace.data_ptr(), _bytes(workspace), B._stream(stream))


def decode_append(geom, n_requests, cache_rows, k, v, rows, step, k_new, v_new, status, stream):
    n = k.shape[0]
    _require(v.shape[0] == n and k_new.shape[0] == n and v_new.shape[0] == n, "k_final, v_final, k_new and v_new: one number of layers")
    _require(k.stride(0) == v.stride(0) and k_new.stride(0) == v_new.stride(0), "keys and values: one layer stride")
    return B.load_library().cf_decode_append(_ref(geom), n_requests, cache_rows, n, k.data_ptr(), v.data_ptr(), k.stride(0),
                                             rows.data_ptr(), step, k_new.data_ptr(), v_new.data_ptr(), k_new.stride(0),
                                             B._ptr(status), B._stream(stream))


def run_stack(geom, batch, plan, workspace, q, k, v, out, score_accum, schedule, strategy, batch_layers, lse, layer_scores, k_final,
              k_self, v_self, scale, doc_len, req_doc_begin, k_prefix, v_prefix, stream):
    stack, keepalive = B.make_stack(q, k, v, out, score_accum, schedule, strategy, batch_layers, lse, layer_scores, k_final, k_self,
                                    v_self, scale, doc_len, req_doc_begin, k_prefix, v_prefix)
    lib = B.load_library()
    need = lib.cf_run_stack_workspace_bytes(_ref(geom), _ref(batch), _ref(stack))
    if need > _bytes(workspace):
        return 0, need
    code = lib.cf_run_stack(_ref(geom), _ref(batch), _ref(stack), plan.data_ptr(), _bytes(plan), workspace.data_ptr(),
                            _bytes(workspace), B._stream(stream))
    del keepalive
    return code, 0
