"""Decoding over the final caches (cf_decode_append / cf_decode_plan / cf_decode_attn) against the oracle's
decode_steps: the caches come out of cf_assemble_final_cache, every step appends one token per request and
its query row attends the grown cache."""
import numpy as np
import pytest
import torch

import oracle
import paper_2502_11101_b200 as cf
from paper_2502_11101_b200 import workloads as W
from paper_2502_11101_b200.session import Session
from tests import harness

pytestmark = pytest.mark.gpu


def _final_caches(cfg, seed, slack):
    """Runs the stack and Phase 2 on the GPU; returns the packed final caches, the rows in use, and the
    oracle's final caches per (layer, request)."""
    meta = W.make_meta(cfg, seed)
    q, (k, v), (k_self, v_self) = W.make_q(meta), W.make_kv(meta), W.make_kv_self(meta)
    ref = harness.oracle_stack(meta, q, k, v, oracle.ALLOC_ALIGN)
    assert harness.cut_margins(meta, ref, oracle.ALLOC_ALIGN) >= 1e-3
    sess = Session(cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.torch_dtype, cfg.pos_range, cfg.rope_theta, cfg.q_len,
                   meta.doc_len, meta.req_doc_begin, meta.doc_src_start, tail_reserve=cfg.q_len)
    qg, kg, vg, ksg, vsg = [t.cuda() for t in (q, k, v, k_self, v_self)]
    sess.run_stack(qg, kg, vg, cfg.schedule, oracle.ALLOC_ALIGN, torch.empty_like(qg))
    keep = cfg.schedule[-1][1] if cfg.schedule else cfg.n_docs
    cache_rows = keep * cfg.doc_len_hi + cfg.q_len + slack
    k_fin = torch.zeros((cfg.n_layers, cfg.batch, cache_rows, cfg.n_kv_heads, cfg.head_dim), dtype=cfg.torch_dtype, device="cuda")
    v_fin = torch.zeros_like(k_fin)
    rows = torch.zeros(cfg.batch, dtype=torch.int32, device="cuda")
    sess.assemble(kg, vg, ksg, vsg, k_fin, v_fin, rows)
    torch.cuda.synchronize()
    assert sess.status() == 0
    want = {}
    for b in range(cfg.batch):
        lo = int(meta.req_doc_begin[b])
        for l in range(cfg.n_layers):
            want[l, b] = oracle.assemble_final_cache(ref[b]["k_final"][l], v[l].double().numpy(), meta.doc_offsets,
                                                     ref[b]["order"], k_self[l, b].double().numpy(),
                                                     v_self[l, b].double().numpy(), doc_base=lo)
    return sess.geom, k_fin, v_fin, rows, cache_rows, want


@pytest.mark.parametrize("which", ["gqa-bf16-tensor-core", "mha-f32-cuda-core"])
def test_four_decoding_steps_over_the_assembled_caches(which):
    if which == "gqa-bf16-tensor-core":
        cfg = W.WorkloadConfig("decode", 2, 8, 2, 128, "bf16", 1e4, 4096, 7, 20, 150, 5, 2, 2, ((1, 3),))
        steps, layers_per_call = 4, 2                      # both layers of a step in one call
    else:
        cfg = W.WorkloadConfig("decode", 2, 4, 4, 64, "f32", 1e4, 2048, 6, 10, 70, 3, 2, 2, ((1, 3),))
        steps, layers_per_call = 4, 1                      # one call per layer, as a running model issues them
    seed = next(s for s in range(20) if _margin_ok(cfg, s))
    geom, k_fin, v_fin, rows, cache_rows, want = _final_caches(cfg, seed, slack=steps + 3)
    rows_h = rows.cpu().numpy()
    L, B, hq, hkv, d = cfg.n_layers, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim
    gen = torch.Generator().manual_seed(7)
    q_new = torch.randn((steps, L, B, hq, d), generator=gen).to(cfg.torch_dtype)
    k_new = torch.randn((steps, L, B, hkv, d), generator=gen).to(cfg.torch_dtype)
    v_new = torch.randn((steps, L, B, hkv, d), generator=gen).to(cfg.torch_dtype)
    plan = torch.zeros(cf.cf_decode_plan_bytes(geom, B, cache_rows), dtype=torch.uint8, device="cuda")
    work = torch.empty(cf.cf_decode_workspace_bytes(geom, B, cache_rows, layers_per_call), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got_out = torch.full((steps, L, B, hq, d), float("nan"), dtype=cfg.torch_dtype, device="cuda")
    got_lse = torch.full((steps, L, B, hq), float("nan"), device="cuda")
    untouched_k = k_fin.clone()
    for t in range(steps):
        cf.cf_decode_append(geom, B, cache_rows, k_fin, v_fin, rows, t, k_new[t].cuda(), v_new[t].cuda(), status)
        cf.cf_decode_plan(geom, B, cache_rows, rows, t + 1, plan)
        qt = q_new[t].cuda()
        for l0 in range(0, L, layers_per_call):
            l1 = l0 + layers_per_call
            cf.cf_decode_attn(geom, B, cache_rows, plan, qt[l0:l1], k_fin[l0:l1], v_fin[l0:l1], got_out[t, l0:l1], work,
                              got_lse[t, l0:l1])
    torch.cuda.synchronize()
    assert cf.cf_decode_status(geom, B, cache_rows, plan) == 0 and int(status.item()) == 0
    for b in range(B):
        n = int(rows_h[b])
        # the appended rows sit right behind the rows in use, bit for bit; nothing else moved
        assert torch.equal(k_fin[:, b, n:n + steps].cpu(), k_new[:, :, b].transpose(0, 1))
        assert torch.equal(v_fin[:, b, n:n + steps].cpu(), v_new[:, :, b].transpose(0, 1))
        assert torch.equal(k_fin[:, b, :n], untouched_k[:, b, :n]) and torch.equal(k_fin[:, b, n + steps:], untouched_k[:, b, n + steps:])
        for l in range(L):
            kf, vf = want[l, b]
            assert kf.shape[0] == n
            o_ref, lse_ref = oracle.decode_steps(kf, vf, q_new[:, l, b].double().numpy(), k_new[:, l, b].double().numpy(),
                                                 v_new[:, l, b].double().numpy())
            got = got_out[:, l, b].float().cpu().numpy()
            assert np.all(np.abs(got - o_ref) <= 1e-2 + 2e-2 * np.abs(o_ref)), (l, b)
            assert np.all(np.abs(got_lse[:, l, b].cpu().numpy() - lse_ref) <= 1e-2), (l, b)


def _margin_ok(cfg, seed):
    meta = W.make_meta(cfg, seed)
    q, (k, v) = W.make_q(meta), W.make_kv(meta)
    ref = harness.oracle_stack(meta, q, k, v, oracle.ALLOC_ALIGN, final_reposition=False)
    return harness.cut_margins(meta, ref, oracle.ALLOC_ALIGN) >= 1e-3


def test_decode_calls_report_a_full_slot():
    geom = cf.make_geom(4, 4, 64, cf.CF_F32, 2048, 1e4)
    B, cache_rows = 2, 40
    plan = torch.zeros(cf.cf_decode_plan_bytes(geom, B, cache_rows), dtype=torch.uint8, device="cuda")
    rows = torch.tensor([10, 40], dtype=torch.int32, device="cuda")          # the second slot is full
    cf.cf_decode_plan(geom, B, cache_rows, rows, 1, plan)
    assert cf.cf_decode_status(geom, B, cache_rows, plan) == cf.CF_ERR_RANGE
    k_fin = torch.zeros((1, B, cache_rows, 4, 64), device="cuda")
    v_fin = torch.zeros_like(k_fin)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    new = torch.ones((1, B, 4, 64), device="cuda")
    cf.cf_decode_append(geom, B, cache_rows, k_fin, v_fin, rows, 0, new, new, status)
    torch.cuda.synchronize()
    assert int(status.item()) == cf.CF_ERR_RANGE
    assert bool(torch.all(k_fin[0, 0, 10] == 1)) and float(k_fin[0, 1].abs().sum()) == 0.0   # the full slot was skipped
    with pytest.raises(cf.CacheFocusError):
        cf.cf_decode_plan(geom, B, cache_rows, rows, 1, plan[: plan.numel() // 2])


@pytest.mark.parametrize("layers_per_call", [1, 2])
def test_bench_sized_caches_one_step(layers_per_call):
    """Caches of the size bench.py times for decoding (28 query / 4 kv heads, four requests with up to 16 000 rows in
    use: every CTA walks tens of full key tiles), ragged fill levels, one appended token; every (layer, request) against
    the oracle."""
    L, B, hq, hkv, d, cache_rows = 2, 4, 28, 4, 128, 16064
    geom = cf.make_geom(hq, hkv, d, cf.CF_BF16, 32768, 1e6)
    used = np.array([16000, 15001, 9000, 127], dtype=np.int32)
    gen = torch.Generator().manual_seed(11)
    k_fin = torch.randn((L, B, cache_rows, hkv, d), generator=gen).bfloat16()
    v_fin = torch.randn((L, B, cache_rows, hkv, d), generator=gen).bfloat16()
    q_new = torch.randn((L, B, hq, d), generator=gen).bfloat16()
    k_new = torch.randn((L, B, hkv, d), generator=gen).bfloat16()
    v_new = torch.randn((L, B, hkv, d), generator=gen).bfloat16()
    kg, vg, rows = k_fin.cuda(), v_fin.cuda(), torch.from_numpy(used).cuda()
    plan = torch.zeros(cf.cf_decode_plan_bytes(geom, B, cache_rows), dtype=torch.uint8, device="cuda")
    work = torch.empty(cf.cf_decode_workspace_bytes(geom, B, cache_rows, layers_per_call), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full((L, B, hq, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((L, B, hq), float("nan"), device="cuda")
    cf.cf_decode_append(geom, B, cache_rows, kg, vg, rows, 0, k_new.cuda(), v_new.cuda(), status)
    cf.cf_decode_plan(geom, B, cache_rows, rows, 1, plan)
    qg = q_new.cuda()
    for l0 in range(0, L, layers_per_call):
        l1 = l0 + layers_per_call
        cf.cf_decode_attn(geom, B, cache_rows, plan, qg[l0:l1], kg[l0:l1], vg[l0:l1], out[l0:l1], work, lse[l0:l1])
    torch.cuda.synchronize()
    assert cf.cf_decode_status(geom, B, cache_rows, plan) == 0 and int(status.item()) == 0
    for l in range(L):
        for b in range(B):
            n = int(used[b])
            o_ref, lse_ref = oracle.decode_steps(k_fin[l, b, :n].double().numpy(), v_fin[l, b, :n].double().numpy(),
                                                 q_new[l, b][None].double().numpy(), k_new[l, b][None].double().numpy(),
                                                 v_new[l, b][None].double().numpy())
            got = out[l, b].float().cpu().numpy()
            assert np.all(np.abs(got - o_ref[0]) <= 1e-2 + 2e-2 * np.abs(o_ref[0])), (l, b)
            assert np.all(np.abs(lse[l, b].cpu().numpy() - lse_ref[0]) <= 1e-2), (l, b)


@pytest.mark.parametrize("hq,hkv,cache_rows,used", [
    (12, 2, 90, [1, 15, 16, 17, 63, 64, 65, 90]),        # one cluster per kv head: step and warp edges
    (5, 5, 40, [40]),                                     # a single head per kv head
    (16, 2, 600, [600, 3]), (27, 3, 600, [599, 33]),      # eight and nine heads per kv head
    (40, 1, 200, [200, 1, 129]),                          # forty: tiles of sixteen heads, the last one half empty
    (8, 1, 6000, [6000, 1, 257]), (20, 2, 9000, [9000, 5]),   # equal shares of all rows, units cut several times
    (64, 64, 3000, [3000, 2999, 7]),                      # several whole units per share
])
def test_decode_kernel_at_the_edges_of_its_splits(hq, hkv, cache_rows, used):
    L, B, d = 2, len(used), 128
    geom = cf.make_geom(hq, hkv, d, cf.CF_BF16, 32768, 1e6)
    gen = torch.Generator().manual_seed(hq + cache_rows)
    k = torch.randn((L, B, cache_rows, hkv, d), generator=gen).bfloat16()
    v = torch.randn((L, B, cache_rows, hkv, d), generator=gen).bfloat16()
    q = (2 * torch.randn((L, B, hq, d), generator=gen)).bfloat16()
    rows = torch.tensor(used, dtype=torch.int32, device="cuda")
    plan = torch.full((cf.cf_decode_plan_bytes(geom, B, cache_rows),), 255, dtype=torch.uint8, device="cuda")
    cf.cf_decode_plan(geom, B, cache_rows, rows, 0, plan)
    kg, vg, qg = k.cuda(), v.cuda(), q.cuda()
    for per_call in (1, L):
        work = torch.full((cf.cf_decode_workspace_bytes(geom, B, cache_rows, per_call),), 255, dtype=torch.uint8, device="cuda")
        out = torch.full((L, B, hq, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((L, B, hq), float("nan"), device="cuda")
        for l in range(0, L, per_call):
            cf.cf_decode_attn(geom, B, cache_rows, plan, qg[l:l + per_call], kg[l:l + per_call], vg[l:l + per_call],
                              out[l:l + per_call], work, lse[l:l + per_call])
        assert cf.cf_decode_status(geom, B, cache_rows, plan) == 0
        for l in range(L):
            for b, n in enumerate(used):
                heads = np.arange(hq) // (hq // hkv)
                logits = np.einsum("hd,nhd->hn", q[l, b].double().numpy(), k[l, b, :n].double().numpy()[:, heads]) / np.sqrt(d)
                top = logits.max(axis=1, keepdims=True)
                w = np.exp(logits - top)
                ref = np.einsum("hn,nhd->hd", w / w.sum(axis=1, keepdims=True), v[l, b, :n].double().numpy()[:, heads])
                got = out[l, b].double().cpu().numpy()
                assert np.all(np.abs(got - ref) <= 1e-2 + 2e-2 * np.abs(ref)), (l, b, per_call)
                assert np.all(np.abs(lse[l, b].cpu().numpy() - (top[:, 0] + np.log(w.sum(axis=1)))) <= 1e-2), (l, b, per_call)


@pytest.mark.parametrize("graph", [False, True])
def test_steps_queued_behind_one_another(graph):
    """Plan, append, attention and merge of many steps in one queue, the requests' fill levels changing from step to step so
    that every step cuts its rows into other shares: bit for bit the results of the steps run one at a time."""
    hq, hkv, room, d = 8, 1, 6000, 128
    levels = [[5990, 1, 257], [33, 5900, 4000], [2000, 2001, 1], [1, 1, 5999]] * 3
    geom = cf.make_geom(hq, hkv, d, cf.CF_BF16, 32768, 1e6)
    gen = torch.Generator(device="cuda").manual_seed(5)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    k0, v0 = rand(1, 3, room, hkv, d), rand(1, 3, room, hkv, d)
    q, k_new, v_new = rand(len(levels), 1, 3, hq, d), rand(len(levels), 1, 3, hkv, d), rand(len(levels), 1, 3, hkv, d)
    rows = torch.tensor(levels, dtype=torch.int32, device="cuda")
    plan = torch.full((cf.cf_decode_plan_bytes(geom, 3, room),), 255, dtype=torch.uint8, device="cuda")
    work = torch.full((cf.cf_decode_workspace_bytes(geom, 3, room, 1),), 255, dtype=torch.uint8, device="cuda")

    def steps(k, v, out, lse, one_at_a_time):
        for i in range(len(levels)):
            cf.cf_decode_plan(geom, 3, room, rows[i], 1, plan)
            cf.cf_decode_append(geom, 3, room, k, v, rows[i], 0, k_new[i], v_new[i])
            cf.cf_decode_attn(geom, 3, room, plan, q[i], k, v, out[i], work, lse[i])
            if one_at_a_time:
                torch.cuda.synchronize()

    results = []
    for queued in (False, True):
        k, v = k0.clone(), v0.clone()
        out = torch.full((len(levels), 1, 3, hq, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((len(levels), 1, 3, hq), float("nan"), device="cuda")
        torch.cuda.synchronize()
        if queued and graph:
            recorded = torch.cuda.CUDAGraph()
            with torch.cuda.graph(recorded):
                steps(k, v, out, lse, False)
            recorded.replay()
        else:
            steps(k, v, out, lse, not queued)
        torch.cuda.synchronize()
        results.append((out, lse))
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])
    assert not bool(torch.isnan(results[0][1]).any())


def test_both_marshallers_give_the_same_results(monkeypatch):
    """A stack, its final caches, a decoding step and cache construction with the calls marshalled natively and by ctypes."""
    from paper_2502_11101_b200 import binding, build, marshal_ctypes
    from paper_2502_11101_b200.session import Session
    native = binding._load_native(build.NATIVE_PATH)
    assert native is not None
    L, B, q_len, hq, hkv = 3, 2, 5, 4, 2
    lens, begin = np.asarray([40, 97, 20, 130, 64], np.int32), np.asarray([0, 3, 5], np.int32)
    gen = torch.Generator(device="cuda").manual_seed(9)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rand(L, B, q_len, hq, 128), rand(L, int(lens.sum()), hkv, 128), rand(L, int(lens.sum()), hkv, 128)
    ks, vs, qd = rand(L, B, q_len, hkv, 128), rand(L, B, q_len, hkv, 128), rand(L, B, hq, 128)
    kn, vn, qt = rand(L, B, hkv, 128), rand(L, B, hkv, 128), rand(L, int(lens.sum()), hq, 128)
    results = []
    for module in (native, marshal_ctypes):
        monkeypatch.setattr(binding, "_NATIVE", module)
        room = int(lens.sum()) + q_len + 1
        sess = Session(hq, hkv, 128, torch.bfloat16, 32768, 1e6, q_len, lens, begin, np.zeros(5, np.int32), tail_reserve=q_len)
        out, outs, lse = torch.zeros_like(q), torch.zeros_like(q), torch.zeros(L, B, hq, q_len, device="cuda")
        scores = torch.zeros(L, 5, device="cuda")
        sess.run_stack(q, k, v, [(1, 2)], 1, out, lse, layer_scores=scores)
        sess.run_stack(q, k, v, [(1, 2)], 1, outs, driver="calls")
        k_cache, v_cache = (torch.zeros(L, B, room, hkv, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        rows = torch.zeros(B, dtype=torch.int32, device="cuda")
        sess.assemble(k, v, ks, vs, k_cache, v_cache, rows)
        moved = torch.zeros_like(k)
        sess.reposition(k, moved, L, k.stride(0))
        plan = torch.zeros(cf.cf_decode_plan_bytes(sess.geom, B, room), dtype=torch.uint8, device="cuda")
        work = torch.zeros(cf.cf_decode_workspace_bytes(sess.geom, B, room, L), dtype=torch.uint8, device="cuda")
        token, token_lse = torch.zeros_like(qd), torch.zeros(L, B, hq, device="cuda")
        cf.cf_decode_plan(sess.geom, B, room, rows, 1, plan)
        cf.cf_decode_append(sess.geom, B, room, k_cache, v_cache, rows, 0, kn, vn)
        cf.cf_decode_attn(sess.geom, B, room, plan, qd, k_cache, v_cache, token, work, token_lse)
        built, off = torch.zeros_like(qt), torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda()
        cf.cf_document_prefill_attn(sess.geom, off, int(lens.max()), qt, k, v, built)
        torch.cuda.synchronize()
        assert sess.status() == 0
        results.append((out, outs, lse, scores, sess.score_accum.clone(), k_cache, v_cache, rows, moved, token, token_lse, built))
    for a, b in zip(*results):
        assert torch.equal(a, b) and float(a.float().abs().max()) > 0


@pytest.mark.parametrize("heads,room", [((12, 2), 1075), ((20, 2), 513), ((4, 4), 40)])
def test_rows_not_in_use_hold_anything(heads, room):
    """Keys and values of a slot behind the rows in use may be read before their number is known, but count for nothing, whatever
    they hold: around the steps of 16 keys, the 64 of a CTA's warps and the 512 of a cluster."""
    import paper_2502_11101_b200 as cf
    hq, hkv = heads
    rows = [r for r in (1, 15, 16, 17, 63, 64, 65, 511, 512, 513, 1000) if r <= room]
    b = len(rows)
    gen = torch.Generator(device="cuda").manual_seed(room)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rand(1, b, hq, 128), rand(1, b, room, hkv, 128), rand(1, b, room, hkv, 128)
    for i, r in enumerate(rows):
        k[:, i, r:], v[:, i, r:] = float("nan"), float("inf")
    geom = cf.make_geom(hq, hkv, 128, torch.bfloat16, 1 << 20, 1.0e4)
    used = torch.tensor(rows, dtype=torch.int32, device="cuda")
    plan = torch.zeros(cf.cf_decode_plan_bytes(geom, b, room), dtype=torch.uint8, device="cuda")
    work = torch.empty(cf.cf_decode_workspace_bytes(geom, b, room, 1), dtype=torch.uint8, device="cuda")
    out, lse = torch.empty_like(q), torch.empty(1, b, hq, device="cuda")
    cf.cf_decode_plan(geom, b, room, used, 0, plan)
    cf.cf_decode_attn(geom, b, room, plan, q, k, v, out, work, lse)
    torch.cuda.synchronize()
    for i, r in enumerate(rows):
        kk, vv = (x[0, i, :r].double().repeat_interleave(hq // hkv, dim=1) for x in (k, v))
        s = torch.einsum("hd,thd->ht", q[0, i].double(), kk) / np.sqrt(128.0)
        # one bf16 rounding of the probabilities and of the output; fp32 sums for the log-sum-exp
        assert torch.allclose(out[0, i].double(), torch.einsum("ht,thd->hd", s.softmax(-1), vv), rtol=1e-2, atol=1e-2), r
        assert torch.allclose(lse[0, i].double(), s.logsumexp(-1), rtol=0, atol=1e-4), r
