"""sage_expand_topk at the edges of its chunks: vocabularies around one batch of a thread block, rows that take one,
two, four and eight blocks, ragged ends, candidates on both sides of a boundary, references that jump, and the
hand-over of tokens to several trees.  Against the fp64 oracle, with the tolerances of the other parity tests."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_00523_b200 as sage
from helpers import check_logits, dev_f32, dev_i32
from workloads import chain_tree, random_tree, star_tree

pytestmark = pytest.mark.gpu
BATCH = 4096                                     # elements of one batch of a thread block


def expand(lg, k, ke, **tree):
    """Rows padded to a stride of a multiple of four with values that must not be read."""
    rows, vocab = lg.shape
    buf = np.full((rows, (vocab + 3) // 4 * 4 + 4), 1e9, np.float32)
    buf[:, :vocab] = lg
    st = sage.new_status()
    o = sage.sage_expand_topk(dev_f32(buf)[:, :vocab], k, ke, status=st, **tree)
    torch.cuda.synchronize()
    return {n: t.cpu().numpy() for n, t in o.items()}, int(st.item())


# (rows, vocab): every number of blocks per row from 1 to 8, and the counts of the many-row cases
@pytest.mark.parametrize("rows,vocab", [(1, 1), (2, 3), (3, 5), (201, 9), (1, BATCH - 1), (1, BATCH + 1), (2, 2 * BATCH),
                                        (1, 4 * BATCH + 3), (30, 8 * BATCH - 2), (70, 3 * BATCH + 1), (120, 5 * BATCH),
                                        (200, 7 * BATCH + 2), (25, 15 * BATCH + 1), (601, 2 * BATCH + 5),
                                        (37, 9 * BATCH + 6), (45, 7 * BATCH - 1), (54, 5 * BATCH + 1), (90, 3 * BATCH),
                                        (150, 16 * BATCH + 3), (300, 16 * BATCH)])
@pytest.mark.parametrize("k", [1, 8, 9, 16])
def test_chunk_edges(rows, vocab, k):
    k = min(k, vocab)
    r = np.random.Generator(np.random.Philox(rows * 1000003 + vocab + k))
    lg = r.standard_normal((rows, vocab)).astype(np.float32) * 2
    for edge in range(BATCH, vocab, BATCH):      # peaks and ties on both sides of every batch boundary
        lg[:, edge - 1:edge + 1] = np.float32(9.0)
    lg[-1, -1] = 11.0                            # the last element of the last chunk
    got, st = expand(lg, k, max(1, min(k, 10)))
    assert st == 0
    check_logits(got, lg, k, max(1, min(k, 10)))


def test_reference_jumps_and_masked_tokens():
    V = 6 * BATCH + 2
    r = np.random.Generator(np.random.Philox(11))
    lg = r.standard_normal((6, V)).astype(np.float32)
    lg[0, 5 * BATCH + 17] = 40.0                 # far above everything before it
    lg[1] += np.linspace(0, 60, V).astype(np.float32)
    lg[2] += np.linspace(60, 0, V).astype(np.float32)
    lg[3, :4 * BATCH] = np.finfo(np.float32).min  # a masked prefix: whole blocks without weight
    lg[4, BATCH // 2:] = np.finfo(np.float32).min
    lg[5] = 7.5                                  # constant: the lowest indices, in order
    got, st = expand(lg, 10, 10)
    assert st == 0
    check_logits(got, lg, 10, 10)
    assert list(got["topk_idx"][5]) == list(range(10))


def test_tokens_go_to_the_children_in_every_tree_of_a_batch():
    r = np.random.Generator(np.random.Philox(12))
    trees = [random_tree(r, n, max_children=5) for n in (1, 2, 33, 40)] + [chain_tree(64), star_tree(6)] * 16
    offs = np.concatenate([[0], np.cumsum([len(t["parent"]) for t in trees])]).astype(np.int32)
    rows, V, k = int(offs[-1]) + 3, 2 * BATCH + 1, 6
    parent, rank = np.concatenate([t["parent"] for t in trees]), np.concatenate([t["rank"] for t in trees])
    root = r.integers(0, V, len(trees)).astype(np.int32)
    lg = r.standard_normal((rows, V)).astype(np.float32)
    kw = dict(parent=dev_i32(parent), rank=dev_i32(rank), node_offsets=dev_i32(offs), root_token=dev_i32(root))
    got, st = expand(lg, k, 4, **kw)
    assert st == 0
    np.testing.assert_array_equal(got["draft_token"], oracle.expand_gather(got["topk_idx"], parent, rank, offs, root))
    # a rank outside the candidates and a parent that is not before its child: reported, token -1, the others as before
    bad_rank, bad_parent = rank.copy(), parent.copy()
    a, b = int(offs[2]) + 7, int(offs[3]) + 9
    bad_rank[a], bad_parent[b] = k, 9
    kw.update(parent=dev_i32(bad_parent), rank=dev_i32(bad_rank))
    bad, st = expand(lg, k, 4, **kw)
    assert st == sage.SAGE_STATUS_BAD_TREE
    want = got["draft_token"].copy()
    want[[a, b]] = -1
    np.testing.assert_array_equal(bad["draft_token"], want)


@pytest.mark.parametrize("peaks,entropy_bound,logprob_bound", [(1, 4.3e-7, 1.2e-7), (8, 1.3e-7, 1.8e-7)])
def test_rows_with_peaks_are_as_exact_as_32_bit_sums_allow(peaks, entropy_bound, logprob_bound):
    """Root mean square errors against 64 bits, of rows cut into two chunks.  What counts is how the sums are taken: with one
    rounding per 16 elements and the largest element at the reference the entropies are off by 3.0e-7 and 1.0e-7, the first
    log-probabilities by 0.85e-7 and 0.92e-7; with one per two elements and a reference up to 8 lower by 6.1e-7 and 1.8e-7, 1.7e-7
    and 2.4e-7 (the bounds lie between).  A unit in the last place of these results is 1.2e-7 (entropies of 1 to 2) or less."""
    rows, V = 148, 152064
    r = np.random.Generator(np.random.Philox(13))
    lg = r.standard_normal((rows, V), dtype=np.float32)
    top = lg.max(axis=1)
    for i in range(peaks):
        at = r.integers(i * (V // peaks), (i + 1) * (V // peaks), rows)
        lg[np.arange(rows), at] = top + (6 + 4 * r.random(rows, dtype=np.float32) if peaks == 1 else np.float32(10 - i))
    got, st = expand(lg, 1, 1)
    assert st == 0
    H, lse = oracle.softmax_entropy(lg)
    rms = lambda e: float(np.sqrt((e ** 2).mean()))                                              # noqa: E731
    assert rms(got["entropy_full"] - H) <= entropy_bound
    assert rms(got["topk_logprob"][:, 0] - (lg.max(axis=1).astype(np.float64) - lse)) <= logprob_bound


@pytest.mark.parametrize("rows_more", [0, 148])
def test_rows_with_few_finite_logits_give_real_indices(rows_more):
    """Masks of -inf that leave fewer elements than candidates (allowed tokens of a grammar): the finite ones first, then the
    lowest of the masked indices.  Elements that are no number are never candidates; without any other the index is -1."""
    V, k = 6 * BATCH + 3, 10
    r = np.random.Generator(np.random.Philox(14))
    lg = np.full((8 + rows_more, V), -np.inf, np.float32)
    lg[1, [V - 1, 5, 2 * BATCH + 77]] = 3.0, 1.0, 2.0
    lg[2, [V - 2, BATCH]] = -1.0, 4.0
    lg[3, r.permutation(V)[:9]] = r.standard_normal(9)
    lg[4, 3 * BATCH:3 * BATCH + 9] = 2.5
    lg[5, -k:] = r.standard_normal(k)                # as many as are asked for
    lg[6, :BATCH] = r.standard_normal(BATCH)         # whole blocks without a finite element
    lg[7] = np.nan
    lg[7, [40, V - 1]] = 1.0, 2.0
    lg[8:] = r.standard_normal((rows_more, V))
    got, st = expand(lg, k, k)
    assert st == 0
    ok = np.arange(len(lg)) != 7
    np.testing.assert_array_equal(got["topk_idx"][ok], oracle.topk(lg[ok], k))
    assert list(got["topk_idx"][7]) == [V - 1, 40] + [-1] * 8
    some = ok & (np.arange(len(lg)) > 0)
    x = lg[some].astype(np.float64)
    lse = x.max(axis=1) + np.log(np.exp(x - x.max(axis=1, keepdims=True)).sum(axis=1))
    np.testing.assert_allclose(got["lse"][some], lse, rtol=1e-6, atol=1e-6)
    want = np.take_along_axis(x, got["topk_idx"][some].astype(np.int64), 1) - lse[:, None]
    np.testing.assert_allclose(got["topk_logprob"][some], want, rtol=1e-5, atol=1e-5)
    assert np.abs(got["alpha"][5:7] - oracle.confidence(lg[5:7], k)[1]).max() <= 1e-5


@pytest.mark.parametrize("rows,vocab", [(2, 12 * BATCH + 5), (160, 17 * BATCH), (600, 16 * BATCH + 2)])
@pytest.mark.parametrize("k", [1, 10, 16])
def test_plateaus_and_slopes_that_overflow_the_list(rows, vocab, k):
    """More elements reach the threshold than a thread block's list holds: equal values within, across and behind batches,
    steps up and down between them, values in order.  Of equal values the lowest index counts."""
    r = np.random.Generator(np.random.Philox(rows + k))
    batch_of = np.arange(vocab) // (BATCH // 2)
    kinds = [np.full(vocab, -2.0), batch_of % 5, -batch_of, batch_of, np.sort(r.standard_normal(vocab)),
             -np.sort(r.standard_normal(vocab)), r.integers(-3, 4, vocab), np.where(batch_of % 3, np.finfo(np.float32).min, 1.0),
             np.where(r.random(vocab) < 0.5, 0.0, -0.0), np.where(np.arange(vocab) < vocab // 2, r.standard_normal(vocab), np.finfo(np.float32).min)]
    lg = np.stack([kinds[i % len(kinds)] for i in range(rows)]).astype(np.float32)
    got, st = expand(lg, k, 1)
    assert st == 0
    want = oracle.topk(lg[:len(kinds)], k)
    np.testing.assert_array_equal(got["topk_idx"], np.stack([want[i % len(kinds)] for i in range(rows)]))


def test_masked_and_constant_rows_take_no_multiple_of_the_time():
    """Half of the vocabulary masked with the type's lowest value, or no preference at all.  With the elements that overflow a
    list taken one by one the calls below took 50 times as long as on normal rows; now they take the same."""
    x = torch.randn(600, 152064, device="cuda")
    masked = x.clone()
    masked[:, 152064 // 2:] = torch.finfo(torch.float32).min

    def us(lg):
        out = sage.sage_expand_topk(lg, 10, 10)
        ws = torch.empty(sage.sage_expand_topk_workspace_size(600, 152064), dtype=torch.uint8, device="cuda")
        times = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                sage.sage_expand_topk(lg, 10, 10, out=out, ws=ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    normal = us(x)
    assert us(masked) <= 4 * normal and us(torch.full_like(x, 0.5)) <= 4 * normal
