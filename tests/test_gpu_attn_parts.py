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
