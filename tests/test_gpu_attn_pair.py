"""Attention by pairs of CTAs (more than one tile of query rows per kv head, shares long enough): parity with the CUDA-core kernel at
the edges of the halves a key tile is cut into, with a pair's second CTA short of rows or without any, and with rows that leave the
range of their reference."""
import numpy as np
import pytest
import torch

from tests.test_gpu_attn_line import _both_paths, _library  # noqa: F401

pytestmark = pytest.mark.gpu

EDGES = [1, 15, 16, 17, 31, 32, 33, 48, 49, 63, 64, 65, 80, 95, 96, 97, 193]


def _lens(n):
    return [EDGES[i % len(EDGES)] for i in range(n)]


@pytest.mark.parametrize("heads,q_len,docs,layers,prefix,self_block,rope_layout,kept", [
    ((16, 2), 17, [340], 1, 0, False, 0, None),                      # 136 rows: tiles of 96 and 40
    ((16, 2), 32, [340], 1, 0, False, 1, [3]),                       # few documents left of many: shares of two tiles, CTAs without one
    ((32, 8), 50, [60, 1, 79], 1, 77, True, 1, None),                # prefix and query tokens as further tiles, not whole
    ((24, 8), 107, [300], 1, 0, True, 0, None),                      # 321 rows: a pair's second CTA has none; two tiles of query tokens
    ((8, 1), 80, [60, 75], 9, 0, False, 0, None),                    # five tiles of rows, several layers per call
    ((12, 2), 64, [150, 150, 7], 2, 9, False, 0, [150, 0, 7]),       # a request that keeps nothing
    ((12, 2), 64, [150, 150, 7], 2, 0, False, 0, [150, 0, 7]),       # .. and has nothing else either
])
def test_pairs_at_their_edges(heads, q_len, docs, layers, prefix, self_block, rope_layout, kept):
    _both_paths(heads, q_len, _lens(sum(docs)), docs, layers, prefix, self_block, kept=kept, rope_layout=rope_layout, kernel=2)


@pytest.mark.parametrize("heads,q_len,docs,every", [((16, 2), 17, [340], 1), ((32, 8), 50, [70, 70], 3)])
def test_rows_of_pairs_out_of_range(heads, q_len, docs, every):
    lens = _lens(sum(docs))
    ends = np.cumsum(lens) - 1
    _, lse, _ = _both_paths(heads, q_len, lens, docs, peak=[int(e) for e in ends[5::40]], peak_every=every, kernel=2)
    assert float(lse.max()) > 60.0


@pytest.mark.parametrize("docs,length,layers", [([1] * 100, 20, 9), ([1, 2, 1] * 20, 97, 4)])
def test_many_units_in_a_share_of_a_pair(docs, length, layers):
    """Shares of some fifty units of one tile, or of a dozen of two and four: descriptions of segments and tiles lap their rings."""
    _both_paths((16, 4), 40, [length] * sum(docs), docs, layers, kernel=2)
