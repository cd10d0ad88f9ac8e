"""Rows whose unit was cut between shares, against 64 bits: what a share leaves of them and how the parts are joined."""
import numpy as np
import pytest
import torch

from tests.test_gpu_attn_line import _library  # noqa: F401

pytestmark = pytest.mark.gpu

TILE = 96


def _session(heads, q_len, lens, docs, prefix=0):
    """Documents that keep their positions: keys enter the logits as they lie in the store."""
    from paper_2502_11101_b200.session import Session
    begin = np.concatenate([[0], np.cumsum(docs)]).astype(np.int32)
    make = lambda start: Session(heads[0], heads[1], 128, torch.bfloat16, 1 << 20, 1e6, q_len, np.asarray(lens, np.int32), begin, start,
                                 tail_reserve=q_len, prefix_len=prefix)
    sess = make(np.zeros(len(lens), np.int32))
    sess.init()
    torch.cuda.synchronize()
    sess = make(sess.read_plan()["dst_start"].astype(np.int32))
    sess.init()
    return sess


def _logits(q, k, hkv):
    """[heads, q_len, keys] in 64 bits."""
    return torch.einsum("jhd,thd->hjt", q.double(), k.double().repeat_interleave(q.shape[1] // hkv, dim=1)) / np.sqrt(128.0)


@pytest.mark.parametrize("heads,q_len,docs,layers", [
    ((2, 1), 16, [4], 1),                                            # one unit in many parts: merged in runs
    ((16, 16), 16, [4], 1),                                          # sixteen units of four parts
    ((4, 1), 40, [84, 84, 84, 84, 84, 84, 84], 1),                   # pairs, shares that hold documents or prefix or both
])
@pytest.mark.parametrize("above", [100.0, 130.0])
def test_scores_of_documents_far_below_the_prefix(heads, q_len, docs, layers, above):
    """The prefix weighs 2^above times as much as the documents.  Beyond 2^126 the documents' share of the sum is a number below
    the normal ones, and their scores are measured against it.  Such numbers are 2^-149 apart, 2^-13 of the smallest weights here
    (row and part differ by 6 from the mean), of which a score takes the mean over parts and rows."""
    import paper_2502_11101_b200 as cf
    hq, hkv = heads
    lens, prefix = [TILE] * sum(docs), 84 * TILE if len(docs) > 1 else 4 * TILE
    sess = _session(heads, q_len, lens, docs, prefix)
    assert cf.cf_debug_attn_kernel(sess.geom, sess.batch, layers, prefix) == (2 if len(docs) > 1 else 1)
    gen = torch.Generator(device="cuda").manual_seed(7)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    b, total = len(docs), sum(lens)
    q, k, v = rand(layers, b, q_len, hq, 128), rand(layers, total, hkv, 128), rand(layers, total, hkv, 128)
    kp, vp = rand(layers, prefix, hkv, 128), rand(layers, prefix, hkv, 128)
    q[..., 0], k[..., 0], kp[..., 0] = 32.0, 0.0, above / np.log2(np.e) * np.sqrt(128.0) / 32.0
    out, lse = torch.empty_like(q), torch.empty(layers, b, hq, q_len, device="cuda")
    scores = torch.empty(layers, len(lens), device="cuda")
    work = torch.empty(cf.cf_attn_workspace_bytes_full(sess.geom, sess.batch, layers), dtype=torch.uint8, device="cuda")
    cf.cf_query_prefill_attn_prefix(sess.geom, sess.batch, sess.plan, q, k, v, kp, vp, out, work, None, None, lse, scores, sess.score_accum)
    torch.cuda.synchronize()
    assert sess.status() == 0
    for i in range(b):
        first, n = sum(docs[:i]), docs[i]
        x = _logits(q[0, i], k[0, first * TILE:(first + n) * TILE], hkv)
        want = x.softmax(-1).reshape(hq, q_len, n, TILE).sum(-1).mean((0, 1))
        got = scores[0, first:first + n].double()
        assert bool(torch.isfinite(got).all()) and bool(((got - want).abs() <= 2.0 ** -11 * want).all()), float(((got - want) / want).abs().max())
    torch.testing.assert_close(sess.score_accum, scores[0], rtol=0, atol=0)


@pytest.mark.parametrize("heads,q_len,docs", [
    ((2, 1), 13, [31]),                                              # one unit in many parts: merged in runs; a ragged group of rows
    ((16, 16), 16, [30]),                                            # sixteen units of about nine parts
    ((16, 2), 17, [340]),                                            # pairs
])
@pytest.mark.parametrize("every", [1, 3])
def test_rows_from_scratch_are_rounded_once(heads, q_len, docs, every):
    """Every share of a row holds keys 2^100 heavier than the first sixteen it meets, of like weight in all shares: the row is
    computed from scratch everywhere and its result is the sum of many parts.  Probabilities are off by 2^-17 (two bf16 values) and
    by the error of logits near 100 (3e-5), sums are fp32; the one rounding to bf16 is that of the result."""
    import paper_2502_11101_b200 as cf
    hq, hkv = heads
    lens, total = [TILE] * sum(docs), TILE * sum(docs)
    sess = _session(heads, q_len, lens, docs)
    assert cf.cf_debug_attn_kernel(sess.geom, sess.batch, 1) == (2 if docs[0] == 340 else 1)
    gen = torch.Generator(device="cuda").manual_seed(total)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    heavy = (torch.arange(total, device="cuda") % TILE >= 16) & (rand(total) > 0.7)
    q, k, v = 0.05 * rand(1, 1, q_len, hq, 128), 0.5 * rand(1, total, hkv, 128), rand(1, total, hkv, 128).bfloat16()
    rows = torch.arange(q_len, device="cuda") % every == 0           # the rows that find them heavy
    q[:, :, rows, :, 0] += 28.0
    q[:, :, ~rows, :, 1] += 4.0
    k[:, heavy, :, 0] += 28.0
    q, k = q.bfloat16(), k.bfloat16()
    out, lse = torch.empty_like(q), torch.empty(1, 1, hq, q_len, device="cuda")
    scores = torch.empty(1, len(lens), device="cuda")
    work = torch.empty(cf.cf_attn_workspace_bytes_layers(sess.geom, sess.batch, 1), dtype=torch.uint8, device="cuda")
    cf.cf_query_prefill_attn_layers(sess.geom, sess.batch, sess.plan, q, k, v, out, work, lse, scores, sess.score_accum)
    torch.cuda.synchronize()
    assert sess.status() == 0
    x = _logits(q[0, 0], k[0], hkv)
    spread = x[:, rows].log_softmax(-1).exp().reshape(hq, -1, len(lens), TILE).sum(-1)
    assert float(x[:, rows][..., ::TILE].amax()) + 80 * np.log(2.0) < float(x[:, rows][..., heavy].amin()) and float(spread.max()) < 0.5
    p, vv = x.softmax(-1), v[0].double().repeat_interleave(hq // hkv, dim=1)
    want, mass = (torch.einsum("hjt,thd->jhd", p, y) for y in (vv, vv.abs()))
    error = (out[0, 0].double() - want).abs()[rows]
    ulp = torch.exp2(torch.floor(torch.log2(want.abs().clamp_min(2.0 ** -100))) - 7)
    bound = (0.5 * ulp + 2.0 ** -13 * mass)[rows]
    print(heads, every, "error", float(error.square().mean().sqrt() / want[rows].square().mean().sqrt()), "of bound", float((error / bound).max()))
    assert bool((error <= bound).all()), float((error / bound).max())
    assert float((lse[0, 0].double() - x.logsumexp(-1)).abs().max()) <= 1e-4
    assert float((scores[0].double() - p.reshape(hq, q_len, len(lens), TILE).sum(-1).mean((0, 1))).abs().max()) <= 1e-4


def test_static_scratch_holds_what_it_held_without_low_halves():
    """The limit of the entry point without workspace stands on what a call needs without the low halves of its parts."""
    import paper_2502_11101_b200 as cf
    docs, q_len, hq, hkv = [740, 740], 64, 28, 4
    sess = _session((hq, hkv), q_len, [TILE] * sum(docs), docs)
    need = cf.cf_attn_workspace_bytes(sess.geom, sess.batch)
    assert 32 << 20 < need <= 42 << 20
    gen = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rand(2, q_len, hq, 128), rand(sum(docs) * TILE, hkv, 128), rand(sum(docs) * TILE, hkv, 128)
    k[21::TILE * 7, 0] = 40.0                                        # some rows from scratch
    outs, lses = [torch.empty_like(q) for _ in range(2)], [torch.empty(2, hq, q_len, device="cuda") for _ in range(2)]
    sums = [torch.zeros(sum(docs), device="cuda") for _ in range(2)]
    work = torch.empty(need, dtype=torch.uint8, device="cuda")
    cf.cf_query_prefill_attn(sess.geom, sess.batch, sess.plan, q, k, v, outs[0], work, lses[0], None, sums[0])
    cf.cf_query_prefill_attn_static(sess.geom, sess.batch, sess.plan, q, k, v, outs[1], lses[1], None, sums[1])
    torch.cuda.synchronize()
    assert sess.status() == 0
    for a, b in (outs, lses, sums):
        assert torch.equal(a, b)
