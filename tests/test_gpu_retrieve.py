"""GPU parity of top-1 retrieval against the oracle (bit-exact indices).

The kernel decides the argmax on fp32 scores, the oracle on exact double scores. The
cases are built so that both decisions are the same decision: either every score is a
small integer (exact in fp32, ties included), or the test asserts that the best exact
score leads the runner-up by far more than the fp32 accumulation error of a 768-term
dot product. Scores are then compared within that error.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _pg():
    import paper_2608_02560_gb300 as pg
    return pg


def _run(index, queries):
    import torch
    pg = _pg()
    Q = queries.shape[0]
    idx = torch.full((Q,), -7, dtype=torch.int64, device=index.device)
    score = torch.empty((Q,), dtype=torch.float32, device=index.device)
    pg.precog_retrieve(index, queries, idx, score)
    assert pg.precog_device_status()[0] == 0
    return idx.cpu().numpy(), score.cpu().numpy()


def _oracle_top1_blocked(index_np, q_np, block=65536):
    """Oracle top-1 over a large index, row block by row block; blocks are combined with
    the oracle's own rule (strictly greater replaces), so the lowest row still wins ties.
    Also returns the gap between the best and second-best exact scores."""
    best_i, best_s = -1, -np.inf
    top2 = np.array([-np.inf, -np.inf])
    for s in range(0, index_np.shape[0], block):
        blk = index_np[s:s + block].astype(np.float64)
        i, sc = oracle.retrieve(blk, q_np[None])
        if i[0] >= 0 and sc[0] > best_s:
            best_i, best_s = s + int(i[0]), float(sc[0])
        sc_all = blk @ q_np.astype(np.float64)
        top2 = np.sort(np.concatenate([top2, np.partition(sc_all, -2)[-2:]]))[-2:]
    return best_i, best_s, float(top2[1] - top2[0])


def test_tiny_planted(cuda_device):
    import torch
    w = synth.tiny_workload(0)
    index = torch.from_numpy(w.index).to(cuda_device)
    query = torch.from_numpy(w.query).to(cuda_device)
    idx, score = _run(index, query)
    ref_i, ref_s = oracle.retrieve(w.index, w.query)
    assert idx[0] == ref_i[0] == w.planted
    assert abs(score[0] - ref_s[0]) < 1e-6


@pytest.mark.parametrize("dtype_name", ["float16", "bfloat16", "float32"])
@pytest.mark.parametrize("M,Q", [(1, 1), (5, 3), (1000, 9), (4099, 2)])
def test_small_exact_integer_scores(cuda_device, dtype_name, M, Q):
    """Small-integer keys make every score exact in fp32: indices and scores must equal
    the oracle's bit for bit, including the many exact ties (lowest row wins). fp16 and
    bf16 keys run the tensor-core kernel (every 16-bit retrieval does, a single query
    included), fp32 keys the CUDA-core GEMV."""
    import torch
    dtype = getattr(torch, dtype_name)
    rng = np.random.default_rng(M * 7 + Q)
    dim = 64
    index = rng.integers(-2, 3, size=(M, dim)).astype(np.float32)
    queries = rng.integers(-2, 3, size=(Q, dim)).astype(np.float32)
    idx, score = _run(torch.from_numpy(index).to(cuda_device, dtype),
                      torch.from_numpy(queries).to(cuda_device, dtype))
    ref_i, ref_s = oracle.retrieve(index, queries)
    np.testing.assert_array_equal(idx, ref_i)
    np.testing.assert_array_equal(score.astype(np.float64), ref_s)


def test_ties_across_the_grid_and_nan_rows(cuda_device):
    """The same best key planted at rows far apart (different CTAs and warps): the lowest
    row wins. A NaN row never wins; an all-NaN index returns -1 and NaN."""
    import torch
    rng = np.random.default_rng(11)
    M, dim = 200_003, 768
    index = (rng.standard_normal((M, dim)) * 0.01).astype(np.float16)
    best = rng.standard_normal(dim).astype(np.float16)
    for r in (150_001, 70_000, 199_999, 70_001):
        index[r] = best
    index[5] = np.nan
    q = best.astype(np.float32)[None]
    idx, score = _run(torch.from_numpy(index).to(cuda_device),
                      torch.from_numpy(q.astype(np.float16)).to(cuda_device))
    assert idx[0] == 70_000
    nan_index = np.full((7, 64), np.nan, dtype=np.float32)
    idx, score = _run(torch.from_numpy(nan_index).to(cuda_device),
                      torch.ones((2, 64), device=cuda_device))
    assert list(idx) == [-1, -1] and np.all(np.isnan(score))


@pytest.mark.parametrize("dtype_name", ["float16", "bfloat16", "float32"])
def test_empty_index(cuda_device, dtype_name):
    """An index without rows has no comparable score: row -1 and a NaN score for every
    query (no sweep kernel runs; the merge alone writes the result)."""
    import torch
    dtype = getattr(torch, dtype_name)
    idx, score = _run(torch.empty((0, 64), dtype=dtype, device=cuda_device),
                      torch.ones((3, 64), dtype=dtype, device=cuda_device))
    assert list(idx) == [-1, -1, -1]
    assert np.isnan(score).all()


@pytest.mark.parametrize("Q", [1, 256])
def test_query_workload_full_index(cuda_device, Q):
    """1,000,000 unit-norm fp16 keys of dim 768; queries = random keys + N(0, 0.02^2)
    noise, renormalised. Every query must find its planted key; sampled queries are
    checked against the oracle over the whole index (exact fp64 scores)."""
    import torch
    index = synth.device_unit_index(synth.QUERY_INDEX_M, synth.QUERY_DIM, 0, cuda_device)
    queries, rows = synth.device_planted_queries(index, Q, synth.QUERY_NOISE, seed=Q)
    idx, score = _run(index, queries)
    np.testing.assert_array_equal(idx, rows.cpu().numpy())
    index_np = index.cpu().numpy()
    q_np = queries.float().cpu().numpy()
    for qi in sorted({0, Q - 1, Q // 2}):
        ref_i, ref_s = oracle.retrieve(index_np[rows[qi].item()][None], q_np[qi][None])
        assert abs(score[qi] - ref_s[0]) < 1e-5
        bi, bs, gap = _oracle_top1_blocked(index_np, q_np[qi])
        assert gap > 1e-4            # far above fp32 accumulation error: the top-1 is unique
        assert idx[qi] == bi and abs(score[qi] - bs) < 1e-5
    del index
    torch.cuda.empty_cache()


# ------------------------------------------------------------- tensor-core path (every 16-bit retrieval)


@pytest.mark.parametrize("dtype_name", ["float16", "bfloat16"])
@pytest.mark.parametrize("M,Q,dim", [(1, 5, 64), (127, 9, 64), (128, 130, 96), (129, 256, 768),
                                     (4099, 300, 96), (20000, 17, 136), (3000, 2, 64), (70000, 4, 768),
                                     (513, 127, 64), (513, 128, 64),
                                     (1000, 200, 96), (39161, 300, 136), (77824, 129, 64)])
def test_tensor_core_exact_integer_scores(cuda_device, dtype_name, M, Q, dim):
    """Every retrieval over a 16-bit index takes the tcgen05 path; these shapes stress
    its tiling. Small integer keys and queries make every score exact in fp32, so indices
    and scores must
    equal the oracle's bit for bit: ragged tiles (M), ragged and multi-pass query batches
    (Q > 128, Q > 256), a K tail (dim not a multiple of 64), many exact ties. A pass of
    more than 128 queries over an even grid runs on SM pairs (one M = 256 MMA per pair):
    4 tiles on 2 pairs (1000), 153 tiles on 76 pairs so that the first pair takes a third
    tile (39161), a second half of one query (77824, 129)."""
    import torch
    dtype = getattr(torch, dtype_name)
    rng = np.random.default_rng(M * 31 + Q * 7 + dim)
    index = rng.integers(-3, 4, size=(M, dim)).astype(np.float32)
    queries = rng.integers(-3, 4, size=(Q, dim)).astype(np.float32)
    idx, score = _run(torch.from_numpy(index).to(cuda_device, dtype),
                      torch.from_numpy(queries).to(cuda_device, dtype))
    ref_i, ref_s = oracle.retrieve(index, queries)
    np.testing.assert_array_equal(idx, ref_i)
    np.testing.assert_array_equal(score.astype(np.float64), ref_s)


def test_tensor_core_ties_and_nan_rows(cuda_device):
    """The tcgen05 path keeps the lowest row among equal best scores even when they sit
    in different tiles and CTAs, and never lets a NaN row win."""
    import torch
    rng = np.random.default_rng(5)
    M, dim, Q = 300_000, 768, 16
    index = (rng.standard_normal((M, dim)) * 0.01).astype(np.float16)
    best = rng.standard_normal((Q, dim)).astype(np.float16)
    planted = [(q, r) for q in range(Q) for r in (290_001 - 97 * q, 150_000 + 13 * q, 17 * q + 3)]
    for q, r in planted:
        index[r] = best[q]
    index[[1, 2, 299_999]] = np.nan
    idx, score = _run(torch.from_numpy(index).to(cuda_device), torch.from_numpy(best).to(cuda_device))
    for q in range(Q):
        assert idx[q] == min(r for qq, r in planted if qq == q)
    assert np.all(np.isfinite(score))


@pytest.mark.parametrize("dtype_name", ["float16", "bfloat16"])
@pytest.mark.parametrize("M,dim", [(1, 8), (63, 64), (65, 200), (130, 4096), (9729, 64), (38912, 72), (38913, 64),
                                   (50000, 64)])
@pytest.mark.parametrize("Q", [1, 32, 33, 129, 257])
def test_tile_heights(cuda_device, dtype_name, M, dim, Q):
    """Tiles of 16-bit keys are as tall as spreads the rows evenly over the rounds: one tile of
    64 rows, heights between the limits (of SM pairs too), CTAs without a tile, the last row
    of a round, A tiles of 32 and 128 rows and rings of every depth, several rounds of the
    ring and of the two accumulators. Small integers: exact scores and many ties."""
    import torch
    import paper_2608_02560_gb300 as pg
    rng = np.random.default_rng(M + dim + Q)
    index = rng.integers(-2, 3, size=(M, dim)).astype(np.float32)
    queries = rng.integers(-2, 3, size=(Q, dim)).astype(np.float32)
    dtype = getattr(torch, dtype_name)
    ix, qs = (torch.from_numpy(a).to(cuda_device, dtype) for a in (index, queries))
    scores = queries @ index.T                 # exact: |sum| <= 4 * 4096
    order = np.argsort(-scores, axis=1, kind="stable")
    i1 = torch.empty(Q, dtype=torch.int64, device=cuda_device)
    s1 = torch.empty(Q, dtype=torch.float32, device=cuda_device)
    pg.precog_retrieve(ix, qs, i1, s1)
    np.testing.assert_array_equal(i1.cpu().numpy(), order[:, 0])
    for k in (2, 5):
        i = torch.empty((Q, k), dtype=torch.int64, device=cuda_device)
        s = torch.empty((Q, k), dtype=torch.float32, device=cuda_device)
        pg.precog_retrieve_topk(ix, qs, k, i, s)
        m = min(k, M)
        np.testing.assert_array_equal(i.cpu().numpy()[:, :m], order[:, :m])
        np.testing.assert_array_equal(s.cpu().numpy()[:, :m], np.take_along_axis(scores, order[:, :m], axis=1))
        assert (i[:, m:] == -1).all()
    assert pg.precog_device_status()[0] == 0
