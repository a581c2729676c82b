"""The fused launches of an ordinary search against the same stages as
launches of their own (a search with stage timing), bit for bit: canonical
predicates, plan, fingerprint, alpha and w_f in one kernel, and the tables
straight from the conditioning, at the edges of their tiles."""
import numpy as np
import pytest

from paper_2607_22922_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ifvs():
    from paper_2607_22922_gb300 import build
    build.build()
    from paper_2607_22922_gb300 import ifvs as mod
    return mod


@pytest.mark.parametrize("M,K,ds", [(1, 256, 4), (5, 100, 8), (8, 256, 16), (12, 256, 8), (16, 1, 8), (16, 256, 8),
                                    (16, 255, 4), (24, 256, 16), (33, 16, 4), (120, 256, 8), (128, 100, 4)])
@pytest.mark.parametrize("cond", [True, False])
def test_fused_tables_equal_separate_stages(ifvs, M, K, ds, cond):
    rng = np.random.default_rng(M * K + ds)
    N, nq = 3001, 70
    codes = rng.integers(0, K, (N, M), dtype=np.uint8)
    attr = rng.integers(0, 1000, N, dtype=np.int32)
    Cpq = rng.standard_normal((M, K, ds)).astype(np.float32)
    bank = rng.standard_normal((64, M * 8)).astype(np.float32)
    W = (0.1 * rng.standard_normal((M, 8, K, ds))).astype(np.float32)
    g = ifvs.Index(codes, [attr], D=M * ds, K=K)
    g.load_codebooks(Cpq, **(dict(bank=bank, W=W, hash_seeds=np.array([3, 5], np.uint64)) if cond else {}))
    q = rng.standard_normal((nq, M * ds)).astype(np.float32)
    wz = rng.standard_normal((nq, M * ds)).astype(np.float32)
    p = synth.empty_predicates(nq)
    p["n_clauses"] = 1
    p["c"][:, 0]["op"] = synth.OP_LT
    p["c"][:, 0]["lo"] = rng.integers(0, 1100, nq)
    for n in (1, nq):
        for w in (None, wz):
            a = g.search(q[:n], p[:n], 10, wz=None if w is None else w[:n])
            b = g.search(q[:n], p[:n], 10, wz=None if w is None else w[:n], flags=ifvs.IFVS_F_STAGE_TIMING)
            for x, y in zip(a, b):
                np.testing.assert_array_equal(x, y)
    g.close()


@pytest.mark.parametrize("M,k", [(16, 10), (16, 100), (16, 200), (12, 32), (12, 33), (8, 1), (10, 64), (34, 10),
                                 (120, 128)])
def test_results_do_not_depend_on_the_split(ifvs, M, k):
    """Work items of any size, pairs or none, one query or more than a sorting
    segment per batch: the same ids, distances and counts."""
    rng = np.random.default_rng(M + k)
    N, nq, ds = 70_001, 2300, 4
    codes = rng.integers(0, 256, (N, M), dtype=np.uint8)
    attr = rng.integers(0, 1000, N, dtype=np.int32)
    other = rng.integers(0, 50, N).astype(np.int16)
    g = ifvs.Index(codes, [attr, other, attr], D=M * ds)
    g.load_codebooks(rng.standard_normal((M, 256, ds)).astype(np.float32))
    q = rng.standard_normal((nq, M * ds)).astype(np.float32)
    p = synth.empty_predicates(nq)
    for i in range(nq):
        lo = int(rng.integers(0, 1000))
        width = int(rng.choice([0, 1, 3, 30, 300, 1000]))       # empty to all rows
        synth.set_clause(p[i], 0, 0, synth.OP_RANGE, max(0, lo - width // 2), lo + width - width // 2)
        p[i]["n_clauses"] = 1
        if i % 5 == 0:                                            # the bitmap path
            synth.set_clause(p[i], 1, 1, synth.OP_LT, int(rng.integers(0, 60)))
            p[i]["n_clauses"] = 2
    p[1]["n_clauses"] = 0
    base = g.search(q, p, k, sub_batch=nq)
    few = slice(0, 40)
    for kw in (dict(sub_batch=152), dict(sub_batch=7), dict(chunk_blocks=1, sub_batch=300),
               dict(pair_min_rows=1, sub_batch=nq), dict(pair_min_rows=1, chunk_blocks=9),
               dict(flags=ifvs.IFVS_F_PLAIN_LOADS, sub_batch=600)):
        got = g.search(q, p, k, **kw)
        for x, y in zip(base, got):
            np.testing.assert_array_equal(x, y)
    one = [g.search(q[i:i + 1], p[i:i + 1], k) for i in range(nq)[few]]
    for j in range(3):
        np.testing.assert_array_equal(base[j][few], np.concatenate([o[j] for o in one]))
    g.close()


@pytest.mark.parametrize("M,k", [(12, 1), (12, 64), (16, 10), (16, 128), (12, 256), (16, 256)])
@pytest.mark.parametrize("lists", [True, False])
def test_bitmap_pairs_equal_single_queries(ifvs, M, k, lists):
    """Two bitmap queries per CTA (any density, an odd one out, ties in distance,
    an index that ends inside a block; with the sorted-copy scan off every
    query is one): bit for bit what one query per CTA returns."""
    rng = np.random.default_rng(M + k)
    N, nq, ds = 33_333, 61, 4
    codes = rng.integers(0, 256, (N, M), dtype=np.uint8)
    codes[20_000:24_000] = codes[:4_000]                          # equal rows: ids decide
    attr = rng.integers(0, 1000, N, dtype=np.int32)
    other = rng.integers(0, 50, N).astype(np.int16)
    other[8_192:16_384] = 49                                      # blocks few queries pass
    g = ifvs.Index(codes, [attr, other], D=M * ds)
    g.load_codebooks(rng.standard_normal((M, 256, ds)).astype(np.float32))
    q = rng.standard_normal((nq, M * ds)).astype(np.float32)
    p = synth.empty_predicates(nq)
    for i in range(nq):
        synth.set_clause(p[i], 0, 0, synth.OP_LT, int(rng.choice([0, 1, 5, 100, 500, 1001])))
        synth.set_clause(p[i], 1, 1, synth.OP_LT, int(rng.choice([2, 25, 49, 60])))
        p[i]["n_clauses"] = 2
    kw = dict(list_max_ppm=0 if lists else -1)
    base = g.search(q, p, k, pair_min_rows=-1, **kw)
    for more in (dict(pair_min_rows=1), dict(pair_min_rows=9000), dict(pair_min_rows=1, chunk_blocks=3),
                 dict(pair_min_rows=1, sub_batch=2), dict(pair_min_rows=1, flags=ifvs.IFVS_F_STAGE_TIMING)):
        for x, y in zip(base, g.search(q, p, k, **more, **kw)):
            np.testing.assert_array_equal(x, y)
    g.close()


def test_a_malformed_predicate_takes_no_other_results_away(ifvs):
    """One malformed predicate: IFVS_ERR_ARG, and the other queries' ids,
    distances and counts all the same, whether a host call is small (results
    in the index's page-locked block), larger, or device I/O."""
    import torch
    rng = np.random.default_rng(3)
    N, M, ds, nq, k = 5001, 16, 8, 9, 10
    g = ifvs.Index(rng.integers(0, 256, (N, M), dtype=np.uint8), [rng.integers(0, 1000, N, dtype=np.int32)], D=M * ds)
    g.load_codebooks(rng.standard_normal((M, 256, ds)).astype(np.float32))
    q = rng.standard_normal((nq, M * ds)).astype(np.float32)
    p = synth.empty_predicates(nq)
    p["n_clauses"] = 1
    p["c"][:, 0]["op"] = synth.OP_LT
    p["c"][:, 0]["lo"] = 500
    want = [x.copy() for x in g.search(q, p, k)]
    p[4]["reserved"] = 1
    want[0][4], want[1][4], want[2][4] = -1, np.inf, 0
    for kw in (dict(), dict(sub_batch=4), dict(flags=ifvs.IFVS_F_DEVICE_IO)):
        out = [np.full((nq, k), -7, np.int64), np.full((nq, k), -7, np.float32), np.full(nq, -7, np.int64)]
        args = [q, p.view(np.uint8).reshape(nq, -1)] + out
        if kw.get("flags"):
            args = [torch.from_numpy(x).cuda() for x in args]
        else:
            args[1] = p
        with pytest.raises(ifvs.IfvsError) as e:
            g.search(args[0], args[1], k, ids=args[2], dists=args[3], npass=args[4], **kw)
        assert e.value.code == ifvs.IFVS_ERR_ARG
        for x, y in zip(want, args[2:]):
            np.testing.assert_array_equal(x, y.cpu().numpy() if kw.get("flags") else y)
    g.close()


@pytest.mark.parametrize("M,ds", [(4, 8), (31, 8), (32, 8), (120, 8)])
@pytest.mark.parametrize("R", [1, 17, 256])
def test_rerank_of_many_queries_equals_few(ifvs, M, ds, R):
    """A batch on either side of the rule for the warps per query, at
    dimensions on either side of the candidates in flight: the same bits, and
    the exact order (the distances to a float32 sum's rounding, D 2^-24)."""
    rng = np.random.default_rng(M + R)
    N, nq, k, D = 2000, 650, min(R, 7), M * ds
    X = rng.standard_normal((N, D)).astype(np.float32)
    g = ifvs.Index(rng.integers(0, 256, (N, M), dtype=np.uint8), [np.zeros(N, np.int32)], vectors=X)
    q = rng.standard_normal((nq, D)).astype(np.float32)
    cand = np.stack([rng.permutation(N)[:R] for _ in range(nq)]).astype(np.int64)
    cand[rng.random((nq, R)) < 0.1] = -1
    cand[5] = -1
    ids, d = g.rerank(q, cand, k)
    for a in range(0, nq, 300):
        i2, d2 = g.rerank(q[a:a + 300], cand[a:a + 300], k)
        np.testing.assert_array_equal(ids[a:a + 300], i2)
        np.testing.assert_array_equal(d[a:a + 300], d2)
    for i in (0, 5, 649):
        ok = cand[i][cand[i] >= 0]
        e = np.sort(((q[i].astype(np.float64) - X[ok]) ** 2).sum(1))[:k]
        np.testing.assert_allclose(d[i, :len(e)], e, rtol=D * 2.0 ** -24)
        assert (ids[i, len(e):] == -1).all() and np.isinf(d[i, len(e):]).all()
    g.close()
