"""Selection and re-ranking at the lengths where their kernels change: the K
first pairs by (x desc, key asc) against numpy's sort, and the t largest |c|
by FP32 bounds against the same call without them (t near the number of
candidates takes the FP64 product of every candidate)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


@pytest.mark.parametrize("kind", ["ties", "wide", "equal"])
@pytest.mark.parametrize("n,K", [(1, 1), (31, 40), (33, 5), (2047, 2047), (2048, 100), (2049, 2049),
                                 (8193, 8193), (32_768, 32_768), (32_769, 30_000),
                                 (40_000, 1000), (140_000, 3000), (300_000, 1), (300_000, 2048),
                                 (300_000, 150_000)])
def test_select_pairs(n, K, kind):
    import paper_1506_03872_gb300 as mad
    rng = _rng(n + K)
    key = rng.choice(1 << 40, size=n, replace=False).astype(np.uint64)
    i, j = key >> np.uint64(20), key & np.uint64((1 << 20) - 1)
    if n > 100:   # indices that use all 32 bits
        i[:50] += np.uint64((1 << 32) - (1 << 21))
    x = {"ties": rng.integers(0, 4, n), "wide": rng.integers(-(1 << 61), 1 << 62, n),
         "equal": np.full(n, 7)}[kind].astype(np.int64)
    with mad.Context() as c:
        out, cnt = mad.mad_select_pairs(c.ctx, mad.encode_pairs(i, j, x), n, K)
    gi, gj, gx, _ = mad.decode_pairs(out, cnt)
    keys = mad.keys_of(i, j)
    pos = np.nonzero(x > 0)[0]
    order = pos[np.lexsort((keys[pos], -x[pos]))][:K]
    assert cnt == len(order)
    assert np.array_equal(gx, x[order])
    assert np.array_equal(mad.keys_of(gi, gj), keys[order])


@pytest.mark.parametrize("kind", ["factors", "ties", "tiny", "mixed_scales"])
@pytest.mark.parametrize("ta,tb,d", [(np.float32, np.float32, 100), (np.float64, np.float64, 33),
                                     (np.float64, np.float32, 1), (np.float32, np.float64, 1024)])
def test_bounded_rescore_equals_the_whole_one(kind, ta, tb, d):
    import paper_1506_03872_gb300 as mad
    rng = _rng(d)
    m, n = 700, 900
    A, B = rng.standard_normal((m, d)), rng.standard_normal((d, n))
    if kind == "ties":
        A, B = np.sign(A), np.sign(B)
    if kind == "tiny":         # FP32 products below its range, FP64 entries below it
        A[1:] *= 1e-30
        B[:, 1:] *= 1e-18
        if ta == np.float64:
            A[5:] *= 1e-40
    if kind == "mixed_scales":
        A *= np.exp(6 * rng.standard_normal((m, 1)))
        B *= np.exp(rng.standard_normal((1, n)))
    tA = torch.from_numpy(A.astype(ta)).cuda()
    tB = torch.from_numpy(B.astype(tb)).cuda()
    flat = rng.permutation(m * n)
    with mad.Context() as c:
        c.build(mad.dense(tA), mad.dense(tB), 1024, keep=(tA, tB))
        for ncand, t in ((4096, 1), (4097, 512), (20_000, 2049), (140_001, 700), (300_000, 5000)):
            q = flat[:ncand]
            if kind == "tiny":
                q = q[(q // n > 0) & (q % n > 0)]
            cand = mad.encode_pairs(q // n, q % n, np.arange(1, len(q) + 1))
            whole, nw = mad.mad_rescore(c.ctx, cand, len(q), len(q))
            for _ in range(2):
                top, nt = mad.mad_rescore(c.ctx, cand, len(q), t)
                assert nw == len(q) and nt == t
                assert torch.equal(top, whole[:t])


def test_a_long_candidate_list_is_sized_by_the_keys_there_are():
    """t' above the number of keys of X: the selection's lists (three of 24
    bytes an item and the sorted one) hold those keys, not X's slots (three
    and more per diamond of the budget)."""
    import paper_1506_03872_gb300 as mad
    rng = _rng(8)
    m, d, n, s = 20_000, 20, 3001, 1 << 22
    tA = torch.from_numpy(rng.standard_normal((m, d)).astype(np.float32)).cuda()
    tB = torch.from_numpy(rng.standard_normal((d, n)).astype(np.float32)).cuda()
    out = mad.new_pairs(s)
    with mad.Context() as c:
        c.build(mad.dense(tA), mad.dense(tB), s, keep=(tA, tB))
        mad.mad_sample(c.ctx, s, 3)
        st = mad.mad_stats(c.ctx)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        _, cnt = mad.mad_topk(c.ctx, s, out)
        used = free - torch.cuda.mem_get_info()[0]
        keys, vals, nx = mad.mad_export_x(c.ctx, cap=s)
    x = vals[:nx]
    assert st["distinct"] == nx and cnt == int((x > 0).sum())
    got = out[:cnt, 1]
    assert torch.equal(got, torch.sort(x[x > 0], descending=True).values)
    lists = 3 * 24 * nx + 24 * (1 << (nx - 1).bit_length())
    assert used <= lists + (64 << 20), (used, lists)


@pytest.mark.parametrize("ld,first", [(100, 0), (104, 0), (128, 4), (102, 0), (104, 2), (101, 1)])
def test_bounded_rescore_of_rows_in_a_wider_matrix(ld, first):
    """A leading dimension above d, rows on 16-byte boundaries or not."""
    import paper_1506_03872_gb300 as mad
    rng = _rng(ld + first)
    m, d, n, ncand, t = 700, 100, 900, 50_000, 300
    wide = torch.from_numpy(rng.standard_normal(m * ld + first + 8).astype(np.float32)).cuda()
    tA = wide[first:].as_strided((m, d), (ld, 1))
    tB = torch.from_numpy(rng.standard_normal((d, n)).astype(np.float32)).cuda()
    q = rng.permutation(m * n)[:ncand]
    cand = mad.encode_pairs(q // n, q % n, np.arange(1, ncand + 1))
    with mad.Context() as c:
        c.build(mad.dense(tA), mad.dense(tB), 1024, keep=(wide, tB))
        whole, nw = mad.mad_rescore(c.ctx, cand, ncand, ncand)
        top, nt = mad.mad_rescore(c.ctx, cand, ncand, t)
    assert nw == ncand and nt == t and torch.equal(top, whole[:t])
    A64, B64 = tA.double().cpu().numpy(), tB.double().cpu().numpy()
    gi, gj, _, gc = mad.decode_pairs(top, t)
    assert np.allclose(gc, np.einsum("ij,ji->i", A64[gi], B64[:, gj]), rtol=0, atol=1e-11)
