"""sage_compact_kv where its blocks and batches of moves have edges: one to all blocks of a cluster, columns that do not
fill the last round, paths longer than one group of 32 entries, more sequences than fit at once, and sequences that are
left alone.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_00523_b200 as sage
from helpers import dev_bf16, dev_i32, host_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,heads,batch,max_path", [(1, 1, 1, 9), (1, 8, 3, 64), (3, 5, 2, 40), (13, 8, 1, 9), (33, 7, 2, 17),
                                                          (80, 8, 2, 9), (2, 2, 70, 33)])
def test_compact_edges(layers, heads, batch, max_path):
    r = np.random.Generator(np.random.Philox(layers * 1000 + heads * 100 + batch))
    lens = r.integers(1, 200, batch)
    pages_b = [(int(l) + 64 + 63) // 64 for l in lens]
    n_pages, max_pages = sum(pages_b) + 2, max(pages_b)
    ids = r.permutation(n_pages)
    table = np.full((batch, max_pages), -1, np.int32)
    at = 0
    for b, n in enumerate(pages_b):
        table[b, :n] = ids[at:at + n]
        at += n
    shape = (layers, n_pages, heads, 64, 128)
    k, v = (r.integers(0, 1 << 16, shape, dtype=np.uint16) for _ in range(2))
    path = np.full((batch, max_path), -1, np.int32)
    plen = np.zeros(batch, np.int32)
    for b in range(batch):
        n = int(r.integers(1, max_path + 1)) if b else max_path       # the first sequence accepts a full path
        rest = np.sort(r.choice(np.arange(1, 64), n - 1, replace=False))
        path[b, :n], plen[b] = np.concatenate([[0], rest]), n
    dk, dv, dl, st = dev_bf16(k), dev_bf16(v), dev_i32(lens), sage.new_status()
    sage.sage_compact_kv(dk, dv, dev_i32(table), dl, dev_i32(path), dev_i32(plen), status=st)
    wk, wv, wl = oracle.compact_kv(k, v, table, lens.astype(np.int32), path, plen, 64)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    np.testing.assert_array_equal(host_bits(dk), wk)
    np.testing.assert_array_equal(host_bits(dv), wv)
    np.testing.assert_array_equal(dl.cpu().numpy(), wl)


@pytest.mark.parametrize("at,node,code", [(35, 20, sage.SAGE_STATUS_BAD_PATH), (0, 1, sage.SAGE_STATUS_BAD_PATH),
                                          (36, 64, sage.SAGE_STATUS_BAD_PATH), (None, None, sage.SAGE_STATUS_BAD_PAGE)])
def test_a_bad_entry_leaves_its_sequence_alone_and_no_other(at, node, code):
    r = np.random.Generator(np.random.Philox(5))
    k, v = (r.integers(0, 1 << 16, (2, 6, 4, 64, 128), dtype=np.uint16) for _ in range(2))
    table = np.array([[0, 1, 2], [3, 4, 5]], np.int32)
    lens = np.array([70, 60], np.int32)
    good = np.concatenate([[0], np.arange(2, 38)]).astype(np.int32)   # 37 entries, all but the first move
    path = np.stack([good, good])
    plen = np.array([37, 37], np.int32)
    if at is None:
        table[0, 1] = 6                                               # a page outside the pool
    else:
        path[0, at] = node
    dk, dv, dl, st = dev_bf16(k), dev_bf16(v), dev_i32(lens), sage.new_status()
    sage.sage_compact_kv(dk, dv, dev_i32(table), dl, dev_i32(path), dev_i32(plen), status=st)
    assert int(st.item()) == code
    wk, wv, wl = oracle.compact_kv(k, v, table[1:], lens[1:], path[1:], plen[1:], 64)
    np.testing.assert_array_equal(host_bits(dk), wk)
    np.testing.assert_array_equal(host_bits(dv), wv)
    np.testing.assert_array_equal(dl.cpu().numpy(), [70, wl[0]])
