"""Parity of paths the diffuse synthetic workloads leave cold: logits far above the ones the
single-pass softmax takes its reference from (peaked attention), a caller-chosen softmax scale, a store with padded rows, the
"sort" allocation with several parallel windows on the tensor-core path, both stack drivers, and the
bounded device-side wait.  Everything is compared with the fp64 oracle through the C ABI."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_11101_b200 import workloads as W
from tests import harness

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    assert torch.cuda.is_available()
    from paper_2502_11101_b200 import build
    build.build()
    import paper_2502_11101_b200 as cf
    cf.load_library()


def _peaked_inputs(meta, seed, self_level=0.0):
    """Inputs whose logits sit on a few well separated levels: a running reference of the softmax would have
    to move several times, in the middle of a key tile and from tile to tile, a fixed one (the maximum over a
    unit's first keys) is left behind by 10 to 30 log2 units, well inside its range, while the lower levels still
    carry a visible part of the result.  (Rows that leave the range: tests/test_gpu_attn_line.py.)

    Per (layer, request, kv head) a unit direction u; query rows a*u + noise with a in [6, 10]; a key
    that should score `level` (log2 units for a = 8) is level/(8*scale*log2 e) * u + noise, counter-
    rotated by the document's delta so that the library's re-positioning brings it back onto u.
    Most keys are on level 0, about one in 20 on the second level (8.5 higher), one per request and layer on the third.
    Values carry a level-dependent constant, so every level is visible in the output.
    With `self_level` the query tokens' own keys get one spike on that level (the largest logit then
    sits in the causal query-self block)."""
    cfg = meta.cfg
    rng = np.random.default_rng(seed)
    n_layers, n_req, hq, hkv, d, lq = cfg.n_layers, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.q_len
    g = hq // hkv
    total = meta.total_tokens
    unit = 1.0 / (8.0 * (1.0 / np.sqrt(d)) * np.log2(np.e))          # key length along u per log2 unit at a = 8
    u = rng.standard_normal((n_layers, n_req, hkv, d))
    u /= np.linalg.norm(u, axis=-1, keepdims=True)
    a = rng.uniform(6.0, 10.0, size=(n_layers, n_req, lq, hq))
    q = a[..., None] * np.repeat(u, g, axis=2)[:, :, None] + 0.05 * rng.standard_normal((n_layers, n_req, lq, hq, d))
    k = np.zeros((n_layers, total, hkv, d))
    v = np.zeros((n_layers, total, hkv, d))
    pattern = rng.standard_normal((3, d))
    for b in range(n_req):
        lo, hi = int(meta.req_doc_begin[b]), int(meta.req_doc_begin[b + 1])
        dst, _, _, _ = oracle.allocate_positions(meta.doc_len[lo:hi], range(hi - lo), cfg.pos_range, 0, lq)
        r0, r1 = int(meta.doc_offsets[lo]), int(meta.doc_offsets[hi])
        delta = np.repeat(dst - meta.doc_src_start[lo:hi], meta.doc_len[lo:hi]).astype(np.float64)
        for l in range(n_layers):
            level = np.zeros(r1 - r0)
            level[rng.random(r1 - r0) < 1.0 / 20.0] = 8.5
            level[rng.integers(0, r1 - r0)] = 17.0
            k_rot = (level * unit)[:, None, None] * u[l, b][None] + 0.3 * rng.standard_normal((r1 - r0, hkv, d))
            k[l, r0:r1] = oracle.rope_rotate(k_rot, -np.broadcast_to(delta[:, None], (r1 - r0, hkv)), cfg.rope_theta)
            which = (level / 8.5).astype(int)
            v[l, r0:r1] = (np.array([20.0, -3.0, 0.5])[which])[:, None, None] * pattern[which][:, None, :] \
                + 0.5 * rng.standard_normal((r1 - r0, hkv, d))
    k_self = 0.3 * rng.standard_normal((n_layers, n_req, lq, hkv, d))
    v_self = rng.standard_normal((n_layers, n_req, lq, hkv, d))
    if self_level:
        for l in range(n_layers):
            for b in range(n_req):
                j = int(rng.integers(0, lq))
                k_self[l, b, j] += self_level * unit * u[l, b]
    to = lambda x: torch.from_numpy(x).to(cfg.torch_dtype)
    return to(q), to(k), to(v), to(k_self), to(v_self)


@pytest.mark.parametrize("heads,q_len", [((4, 2), 32), ((16, 2), 32), ((12, 2), 48)])
@pytest.mark.parametrize("self_level", [None, 0.0, 26.0])
def test_peaked_attention_moves_the_softmax_reference(heads, q_len, self_level):
    """64 rows (both warpgroups on the same rows, alternate key tiles), 256 rows (two row tiles side by
    side) and 288 rows (three one-tile CTAs) per kv head; without the query-self block, with it, and
    with the largest logit of every row inside it; one call per layer and one call for all layers."""
    lens = [160, 131, 192, 128, 97, 33, 170, 200, 144, 129, 64, 181]
    cfg = W.WorkloadConfig("peaked", 3, heads[0], heads[1], 128, "bf16", 1e6, 32768, len(lens), 1, 300, q_len, 2, 1, ())
    meta = W.make_meta(cfg, 0, doc_len_override=lens * 2)
    q, k, v, k_self, v_self = _peaked_inputs(meta, 11, self_level or 0.0)
    # With a few keys carrying a row's whole mass, the rounding of a re-positioned key to the cache's
    # 16-bit type shifts that row's logits by more than the averaged-out amount of a diffuse softmax;
    # the oracle therefore attends its own re-positioned keys in that storage type as well.
    ref = harness.oracle_stack(meta, q, k, v, oracle.ALLOC_ALIGN, key_round=oracle.round_to_bf16)
    # the construction does what it is for: in most rows the largest logit is far above the first chunk's
    top = ref[0]["layers"][0]["lse"].max()
    assert top > 8.0
    if self_level is not None:
        harness.add_self_block(meta, ref, q, k_self, v_self)
    for batch_layers in (False, True):
        got = harness.gpu_stack(meta, q, k, v, oracle.ALLOC_ALIGN, batch_layers=batch_layers,
                                k_self=None if self_level is None else k_self,
                                v_self=None if self_level is None else v_self)
        harness.compare(meta, ref, got, k)


@pytest.mark.parametrize("scale", [0.05, 0.2])
@pytest.mark.parametrize("self_block", [False, True])
def test_caller_chosen_softmax_scale(scale, self_block):
    """cf_query_prefill_attn and cf_query_prefill_attn_full with softmax_scale != 1/sqrt(head_dim), on the
    tensor-core path and on the CUDA-core path (fp32, head_dim 64), both stack drivers.  A scale above
    1/sqrt(head_dim) amplifies the storage rounding of the re-positioned keys in the logits, so for the
    16-bit store the oracle attends its re-positioned keys in that type too."""
    cfg = W.scaled_config(W.CONFIGS[3], n_layers=3, n_docs=14, n_planted=3, schedule=((2, 7),))
    for driver in ("library", "calls"):
        harness.run_and_compare(cfg, 1, oracle.ALLOC_ALIGN, min_margin=1e-3, self_block=self_block, driver=driver,
                                softmax_scale=scale, batch_layers=driver == "library", key_round=oracle.round_to_bf16)
    lens = [1, 63, 64, 65, 127, 128, 129, 200, 300, 17, 256, 31]
    small = W.WorkloadConfig("ragged", 2, 8, 2, 64, "f32", 1e4, 4096, len(lens), 1, 300, 5, 1, 2, ((1, 7),))
    harness.run_and_compare(small, 1, oracle.ALLOC_ALIGN, doc_len_override=lens, min_margin=1e-3,
                            self_block=self_block, softmax_scale=scale)


@pytest.mark.parametrize("dtype,head_dim", [("bf16", 128), ("f32", 64)])
def test_store_with_padded_rows(dtype, head_dim):
    """token_stride = n_kv_heads * head_dim + 64: attention (tensor maps and plain loads) and the final
    re-positioning read and write rows at the caller's stride and leave the padding alone."""
    lens = [129, 64, 192, 1, 128, 150, 97]
    cfg = W.WorkloadConfig("padded", 3, 8, 2, head_dim, dtype, 1e4, 4096, len(lens), 1, 300, 9, 2, 2, ((1, 4),))
    stride = 2 * head_dim + 64
    for batch_layers in (False, True):
        harness.run_and_compare(cfg, 2, oracle.ALLOC_ALIGN, doc_len_override=lens * 2, min_margin=1e-3,
                                batch_layers=batch_layers, token_stride=stride, self_block=batch_layers)


@pytest.mark.parametrize("dtype,head_dim", [("bf16", 128), ("f32", 64)])
def test_assembled_final_cache_from_a_padded_store(dtype, head_dim):
    from paper_2502_11101_b200.session import Session
    lens = [129, 64, 192, 1, 128]
    cfg = W.WorkloadConfig("padded-assemble", 2, 4, 2, head_dim, dtype, 1e4, 4096, len(lens), 1, 300, 6, 1, 1, ())
    meta = W.make_meta(cfg, 4, doc_len_override=lens)
    k, v = W.make_kv(meta)
    k_self, v_self = W.make_kv_self(meta)
    stride = 2 * head_dim + 64
    sess = Session(cfg.n_q_heads, cfg.n_kv_heads, head_dim, cfg.torch_dtype, cfg.pos_range, cfg.rope_theta, cfg.q_len,
                   meta.doc_len, meta.req_doc_begin, meta.doc_src_start, tail_reserve=cfg.q_len, token_stride=stride)
    kg, vg = harness.padded_store(k, stride, "cuda"), harness.padded_store(v, stride, "cuda")
    sess.init()
    out_rows = sum(lens) + cfg.q_len
    k_out = torch.zeros((cfg.n_layers, 1, out_rows, cfg.n_kv_heads, head_dim), dtype=cfg.torch_dtype, device="cuda")
    v_out = torch.zeros_like(k_out)
    final_rows = torch.zeros(1, dtype=torch.int32, device="cuda")
    sess.assemble(kg, vg, k_self.cuda(), v_self.cuda(), k_out, v_out, final_rows)
    torch.cuda.synchronize()
    assert sess.status() == 0 and int(final_rows[0]) == out_rows
    plan = sess.read_plan()
    for l in range(cfg.n_layers):
        kr = oracle.reposition_keys(k[l].double().numpy(), meta.doc_offsets, meta.doc_src_start, plan["dst_start"],
                                    plan["order"][0], cfg.rope_theta)
        kf, vf = oracle.assemble_final_cache(kr, v[l].double().numpy(), meta.doc_offsets, plan["order"][0],
                                             k_self[l, 0].double().numpy(), v_self[l, 0].double().numpy())
        n_docs_rows = out_rows - cfg.q_len
        err = np.abs(k_out[l, 0, :n_docs_rows].float().cpu().numpy() - kf[:n_docs_rows]) / \
            harness.rotated_key_tolerance(kf[:n_docs_rows], dtype)
        assert err.max() <= 1.0
        assert np.array_equal(k_out[l, 0, n_docs_rows:].float().cpu().numpy(), kf[n_docs_rows:])
        assert np.array_equal(v_out[l, 0].float().cpu().numpy(), vf)
    assert bool(torch.all(harness.padding_of(kg, stride) == harness.PAD_SENTINEL))


def test_sort_allocation_with_parallel_windows_on_the_tensor_core_path():
    """Attention-Guided Allocation ("sort") while Eq. 6 asks for several parallel windows, bf16 and
    head_dim 128: a 1088-position range holds five 160-200-token documents per window, so 24 documents
    need 5 windows, 10 survivors 2, 5 survivors 1."""
    cfg = W.scaled_config(W.CONFIGS[5], n_layers=3, n_docs=24, n_planted=3, batch=2, pos_range=1088,
                          n_q_heads=8, n_kv_heads=8, schedule=((1, 10), (2, 5)))
    seed = None
    for s in range(12):
        meta = W.make_meta(cfg, s)
        ref = harness.oracle_stack(meta, W.make_q(meta), *W.make_kv(meta), oracle.ALLOC_SORT, final_reposition=False)
        if harness.cut_margins(meta, ref, oracle.ALLOC_SORT) >= 1e-3:
            seed = s
            break
    assert seed is not None, "no seed with a safe margin between neighbouring survivors"
    assert [rec["n_reuse"] for rec in ref[0]["layers"]] == [5, 2, 1]
    for batch_layers in (False, True):
        harness.run_and_compare(cfg, seed, oracle.ALLOC_SORT, min_margin=1e-3, batch_layers=batch_layers)


@pytest.mark.parametrize("batch_layers", [False, True])
def test_both_stack_drivers_agree_bit_for_bit(batch_layers):
    """cf_run_stack issues the same launches as the per-step calls: identical results."""
    cfg = W.scaled_config(W.CONFIGS[3], n_layers=5, n_docs=18, n_planted=3, schedule=((1, 12), (3, 6), (5, 3)))
    meta = W.make_meta(cfg, 2)
    q, (k, v) = W.make_q(meta), W.make_kv(meta)
    a = harness.gpu_stack(meta, q, k, v, oracle.ALLOC_SORT, batch_layers=batch_layers, driver="library")
    b = harness.gpu_stack(meta, q, k, v, oracle.ALLOC_SORT, batch_layers=batch_layers, driver="calls")
    assert a["status"] == 0 and b["status"] == 0 and a["plan"]["order"] == b["plan"]["order"]
    for key in ("out", "lse", "scores", "accum", "k_final"):
        assert np.array_equal(a[key], b[key]), key


def test_bounded_wait_gives_up_and_reports_a_timeout():
    """A wait that nothing satisfies ends after its limit, CF_ERR_TIMEOUT arrives in the plan's status
    word, and the device carries on: the next attention call over the same plan buffer is correct."""
    import paper_2502_11101_b200 as cf
    cfg = W.scaled_config(W.CONFIGS[3], n_layers=1, n_docs=6, n_planted=1, schedule=())
    meta = W.make_meta(cfg, 0)
    q, (k, v) = W.make_q(meta), W.make_kv(meta)
    ref = harness.oracle_stack(meta, q, k, v, oracle.ALLOC_ALIGN)
    got = harness.gpu_stack(meta, q, k, v, oracle.ALLOC_ALIGN)
    sess = got["session"]
    assert got["status"] == 0
    cf.cf_debug_wait_timeout(sess.geom, sess.batch, sess.plan, 2_000_000)         # about a millisecond
    assert sess.status() == cf.CF_ERR_TIMEOUT
    assert cf.cf_error_string(cf.CF_ERR_TIMEOUT) == "device-side wait timed out"
    again = harness.gpu_stack(meta, q, k, v, oracle.ALLOC_ALIGN)                     # a fresh plan: status 0, results right
    harness.compare(meta, ref, again, k)
    sess.init()                                                                     # the old plan is usable again too
    assert sess.status() == 0
