"""The tensor-core attention kernel cuts the key tiles of all units into equal shares: parity with the CUDA-core kernel where
shares end inside units, hold several of them, or find nothing to do, and for rows that leave the range of their reference."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    assert torch.cuda.is_available()
    from paper_2502_11101_b200 import build
    build.build()
    import paper_2502_11101_b200 as cf
    cf.load_library()


def _both_paths(heads, q_len, lens, docs_per_request, layers=1, prefix=0, self_block=False, kept=None, peak=None,
                peak_every=1, rope_layout=0, kernel=None):
    """Outputs, log-sum-exps and scores of both kernel families on the same inputs; `kernel`: the tensor-core one that has to run
    (1: a CTA per tile of query rows, 2: pairs)."""
    import paper_2502_11101_b200 as cf
    from paper_2502_11101_b200.session import Session
    b = len(docs_per_request)
    begin = np.concatenate([[0], np.cumsum(docs_per_request)]).astype(np.int32)
    total, (hq, hkv) = int(sum(lens)), heads
    gen = torch.Generator(device="cuda").manual_seed(total + hq)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rand(layers, b, q_len, hq, 128), rand(layers, total, hkv, 128), rand(layers, total, hkv, 128)
    if peak is not None:                                     # one key per kv head far above all others for every row
        q[:, :, ::peak_every].abs_()
        k[:, peak] = 40.0
    ks, vs = rand(layers, b, q_len, hkv, 128), rand(layers, b, q_len, hkv, 128)
    kp, vp = rand(layers, max(prefix, 1), hkv, 128), rand(layers, max(prefix, 1), hkv, 128)
    results = []
    try:
        for path in (1, 0):
            cf.cf_set_attn_path(path)
            sess = Session(hq, hkv, 128, torch.bfloat16, 32768, 1e6, q_len, np.asarray(lens, np.int32), begin,
                           np.zeros(len(lens), np.int32), tail_reserve=q_len, prefix_len=prefix, rope_layout=rope_layout)
            assert path == 1 or kernel is None or cf.cf_debug_attn_kernel(sess.geom, sess.batch, layers, prefix, self_block) == kernel
            counts = None if kept is None else torch.tensor(kept, dtype=torch.int32, device="cuda")
            sess.init(kept_count=counts)
            out = torch.full_like(q, float("nan"))
            lse = torch.full((layers, b, hq, q_len), float("nan"), device="cuda")
            scores = torch.full((layers, len(lens)), float("nan"), device="cuda")
            work = torch.full((cf.cf_attn_workspace_bytes_full(sess.geom, sess.batch, layers),), 255, dtype=torch.uint8, device="cuda")
            if prefix:
                cf.cf_query_prefill_attn_prefix(sess.geom, sess.batch, sess.plan, q, k, v, kp, vp, out, work,
                                                ks if self_block else None, vs if self_block else None, lse, scores, sess.score_accum)
            elif self_block:
                cf.cf_query_prefill_attn_full(sess.geom, sess.batch, sess.plan, q, k, v, ks, vs, out, work, lse, scores, sess.score_accum)
            else:
                cf.cf_query_prefill_attn_layers(sess.geom, sess.batch, sess.plan, q, k, v, out, work, lse, scores, sess.score_accum)
            torch.cuda.synchronize()
            assert sess.status() == 0
            results.append((out.float().cpu(), lse.cpu(), scores.cpu()))
    finally:
        cf.cf_set_attn_path(0)
    (o_a, l_a, s_a), (o_b, l_b, s_b) = results
    assert torch.all((o_a - o_b).abs() <= 1e-2 + 2e-2 * o_a.abs()), float((o_a - o_b).abs().max())
    inf = torch.isinf(l_a)
    assert torch.equal(inf, torch.isinf(l_b))
    assert torch.all((l_a - l_b)[~inf].abs() <= 1e-3 + 1e-5 * l_a[~inf].abs())
    assert torch.all((s_a - s_b).abs() <= 1e-3 * s_a.abs() + 1e-5)
    return results[1]


@pytest.mark.parametrize("heads,q_len,lens,docs,layers,prefix,self_block", [
    ((1, 1), 1, [1], [1], 1, 0, False),                              # one row, one key
    ((2, 1), 65, [95, 96, 97, 15, 16, 17, 193], [7], 1, 0, False),   # tile edges; two row tiles of 96 and 34 rows
    ((8, 8), 33, [160] * 12, [5, 4, 3], 2, 0, False),                # several units per share
    ((6, 2), 128, [96, 31], [2], 1, 97, True),                       # the query's own keys are two tiles, the prefix too
    ((4, 2), 97, [40], [1], 3, 5, True),                             # rows that see nothing of a share's one tile
    ((2, 2), 9, [20] * 130, [2, 1] * 43 + [1], 1, 0, False),         # more requests than the line's table has entries
])
def test_shares_at_their_edges(heads, q_len, lens, docs, layers, prefix, self_block):
    _both_paths(heads, q_len, lens, docs, layers, prefix, self_block)


@pytest.mark.parametrize("self_block", [False, True])
def test_requests_that_keep_nothing(self_block):
    out, lse, _ = _both_paths((4, 2), 12, [50, 130, 64, 33], [1, 2, 1], 2, 0, self_block, kept=[1, 0, 1])
    if not self_block:
        assert float(out[:, 1].abs().max()) == 0.0 and bool(torch.all(torch.isinf(lse[:, 1])))


@pytest.mark.parametrize("heads,docs", [((4, 2), [9]), ((16, 16), [3, 3, 3])])
def test_rows_far_outside_the_range_of_their_reference(heads, docs):
    """A key more than 2^80 heavier than the first sixteen of its segment: the row is computed from scratch, whether its unit
    was cut between shares or finished by one."""
    out, lse, _ = _both_paths(heads, 20, [150] * 9, docs, peak=[149 + 150 * 1, 149 + 150 * 4, 149 + 150 * 7])
    assert float(lse.max()) > 60.0


@pytest.mark.parametrize("docs,q_len", [(37, 3), (14, 128)])
def test_few_units_in_many_shares(docs, q_len):
    """Two to six units whose rows have many parts each, merged in runs; the last slice of rows is not whole."""
    _both_paths((6, 2), q_len, [200 - 3 * i for i in range(docs)], [docs])


@pytest.mark.parametrize("heads,q_len", [((3, 1), 1), ((5, 5), 3), ((4, 2), 7), ((12, 2), 48)])
@pytest.mark.parametrize("layers", [1, 2, 3, 9, 17])
def test_scores_do_not_depend_on_the_layers_beside_them(heads, q_len, layers):
    """The same layer several times in one call (clusters of one to eight blocks, layers beyond them, rows that are no multiple
    of four): every layer's scores are those of a call with one, they sum to 1 per request, and S takes them in order."""
    import paper_2502_11101_b200 as cf
    from paper_2502_11101_b200.session import Session
    hq, hkv = heads
    lens, begin = [97, 1, 40, 200, 13], np.asarray([0, 3, 5], np.int32)
    gen = torch.Generator(device="cuda").manual_seed(layers)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    q, k, v = rand(1, 2, q_len, hq, 128), rand(1, sum(lens), hkv, 128), rand(1, sum(lens), hkv, 128)
    got = []
    for n in (1, layers):
        sess = Session(hq, hkv, 128, torch.bfloat16, 32768, 1e6, q_len, np.asarray(lens, np.int32), begin,
                       np.zeros(len(lens), np.int32), tail_reserve=q_len)
        sess.init(kept_count=torch.tensor([2, 2], dtype=torch.int32, device="cuda"))
        scores = torch.full((n, len(lens)), float("nan"), device="cuda")
        qn, kn, vn = (x.expand(n, *x.shape[1:]).contiguous() for x in (q, k, v))
        sess.attend_layers(qn, kn, vn, torch.empty_like(qn), layer_scores=scores)
        torch.cuda.synchronize()
        assert sess.status() == 0
        got.append((scores.cpu(), sess.score_accum.cpu()))
    (one, _), (scores, accum) = got
    torch.testing.assert_close(scores, one.expand_as(scores), rtol=1e-3, atol=1e-6)
    torch.testing.assert_close(scores[:, :3].sum(1), torch.ones(layers), rtol=1e-3, atol=0)
    torch.testing.assert_close(scores[:, 3:].sum(1), torch.ones(layers), rtol=1e-3, atol=0)
    total = torch.zeros_like(accum)
    for s in scores:
        total += s
    assert torch.equal(accum[[0, 1, 3, 4]], total[[0, 1, 3, 4]]) and float(scores[:, 2].abs().max()) == 0.0


def test_log_sum_exp_of_a_single_key():
    """A row that sees one key has its logit as log-sum-exp.  Queries of one non-zero element make the product exact, so what is
    left are the roundings of the scale, the reference, the exponential (2^-22) and the logarithm: absolute 2^-22, relative
    8 x 2^-24, as far as the row's own magnitude goes and no further."""
    import paper_2502_11101_b200 as cf
    from paper_2502_11101_b200.session import Session
    q_len, heads = 128, 4
    sess = Session(heads, heads, 128, torch.bfloat16, 32768, 1e6, q_len, np.ones(1, np.int32), np.asarray([0, 1], np.int32),
                   np.zeros(1, np.int32), tail_reserve=q_len)
    sess.init()
    gen = torch.Generator(device="cuda").manual_seed(1)
    k = torch.randn(1, 1, heads, 128, generator=gen, device="cuda").bfloat16()
    rotated, q = torch.empty_like(k), torch.zeros(1, 1, q_len, heads, 128, device="cuda", dtype=torch.bfloat16)
    sess.reposition(k, rotated, 1, 0)
    for j in range(q_len):
        q[0, 0, j, :, j] = 8.0
    lse = torch.empty(1, 1, heads, q_len, device="cuda")
    sess.attend_layers(q, k, torch.ones_like(k), torch.empty_like(q), lse)
    torch.cuda.synchronize()
    want = rotated[0, 0].double() * 8.0 / np.sqrt(128.0)
    error = (lse[0, 0].double() - want).abs()
    assert bool((error <= 2.0 ** -22 + 8 * 2.0 ** -24 * want.abs()).all()), float(error.max())


@pytest.mark.parametrize("rope_layout", [0, 1])
@pytest.mark.parametrize("heads,q_len,lens,docs,prefix,self_block,every", [
    ((4, 2), 11, [97, 15, 1, 33, 130, 80], [6], 0, False, 1),        # odd tiles; the last group of rows is not whole
    ((6, 2), 35, [64, 100, 47], [2, 1], 77, True, 3),                # some rows of a slice; prefix and query tokens as well
    ((16, 16), 40, [50] * 24, [8, 8, 8], 0, True, 5),                # units finished by one share
    ((1, 1), 3, [96] * 60, [60], 0, False, 1),                       # one unit in many shares, merged in runs
])
def test_rows_computed_from_scratch(heads, q_len, lens, docs, prefix, self_block, every, rope_layout):
    """Rows that leave the range of their reference beside rows that do not, in every place they can lie."""
    starts = np.concatenate([[0], np.cumsum(lens)])
    peak = [int(starts[i + 1]) - 1 for i in range(len(lens)) if i % 2 == 1]
    _both_paths(heads, q_len, lens, docs, 2, prefix, self_block, peak=peak, peak_every=every, rope_layout=rope_layout)


def test_a_row_out_of_range_does_not_stop_the_call():
    """One kv head whose rows leave the range of their reference: such rows are an exception, not a reason to take two hundred
    times as long (they were computed by one warp each, a memory latency after the other).  The factor is about twenty."""
    import paper_2502_11101_b200 as cf
    from paper_2502_11101_b200.session import Session
    hq, hkv, q_len, docs, length, layers = 12, 2, 48, 50, 160, 4
    sess = Session(hq, hkv, 128, torch.bfloat16, 32768, 1e6, q_len, np.full(docs, length, np.int32), np.asarray([0, docs], np.int32),
                   np.zeros(docs, np.int32), tail_reserve=q_len)
    sess.init()
    gen = torch.Generator(device="cuda").manual_seed(0)
    q = torch.randn(layers, 1, q_len, hq, 128, generator=gen, device="cuda").bfloat16()
    k = torch.randn(layers, docs * length, hkv, 128, generator=gen, device="cuda").bfloat16()
    v = torch.randn(layers, docs * length, hkv, 128, generator=gen, device="cuda").bfloat16()
    out, work = torch.empty_like(q), torch.empty(cf.cf_attn_workspace_bytes_layers(sess.geom, sess.batch, layers), dtype=torch.uint8, device="cuda")
    times = []
    for peaked in (False, True):
        if peaked:
            q[..., :hq // hkv, :].abs_()
            k[:, 2 * length - 1, 0] = 40.0
        best = float("inf")
        for _ in range(6):
            begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            begin.record()
            cf.cf_query_prefill_attn_layers(sess.geom, sess.batch, sess.plan, q, k, v, out, work)
            end.record()
            torch.cuda.synchronize()
            best = min(best, begin.elapsed_time(end))
        times.append(best)
    assert sess.status() == 0 and times[1] <= 40 * times[0], times
