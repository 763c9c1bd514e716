"""The library steps of a sharded run (mad_export_x_by_owner,
mad_accumulate, mad_select_pairs) on one GPU, with the ranks emulated one
after another in one process (no collective: the owner segments are handed
over here): the partial X of the diamond ranges, merged by owner, equal the
X of one context that sampled every diamond, and Omega_t' and Omega_t equal
that context's and the oracle's bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from gpu_cases import Case  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _x_sorted(mad, ctx, cap):
    keys, vals, n = mad.mad_export_x(ctx, cap=cap)
    k = keys[:n].cpu().numpy().view(np.uint64)
    v = vals[:n].cpu().numpy()
    order = np.argsort(k)
    return k[order], v[order]


@pytest.mark.parametrize("name,world", [("dense_ragged_f32", 2), ("dense_factors_small", 3),
                                        ("chung_lu_small", 2), ("bipartite_binary", 4)])
def test_emulated_ranks_equal_one_run(name, world):
    import paper_1506_03872_gb300 as mad
    from paper_1506_03872_gb300.shard import LibraryOps, diamond_range
    s, seed, tprime, t = 240_000, 31, 1500, 40
    ranks = [Case(name, s_max=s) for _ in range(world)]
    one = Case(name, s_max=s)
    try:
        ops = [LibraryOps(c.ctx.ctx, export_cap=1 << 12) for c in ranks]
        for r in range(world):
            first, count = diamond_range(s, r, world)
            ops[r].sample(count, seed, first)
        parts = [ops[r].export_by_owner(world) for r in range(world)]
        # every partial key goes to exactly one owner
        total = sum(int(p[2][-1]) for p in parts)
        assert total == sum(len(_x_sorted(mad, c.ctx.ctx, s + 1)[0]) for c in ranks)
        cands = []
        for o in range(world):
            rk = torch.cat([k[int(off[o]):int(off[o + 1])] for k, _, off in parts])
            rv = torch.cat([v[int(off[o]):int(off[o + 1])] for _, v, off in parts])
            ops[o].reset()
            ops[o].accumulate(rk, rv)
            cand, nc = ops[o].topk(tprime)
            cands.append(cand[:nc])
        # The owners' X together are the one-run X, key for key.
        mad.mad_sample(one.ctx.ctx, s, seed)
        ok, ov = _x_sorted(mad, one.ctx.ctx, s + 1)
        merged = [_x_sorted(mad, c.ctx.ctx, s + 1) for c in ranks]
        mk = np.concatenate([k for k, _ in merged])
        mv = np.concatenate([v for _, v in merged])
        order = np.argsort(mk)
        assert np.array_equal(mk[order], ok) and np.array_equal(mv[order], ov)
        # Omega_t' from the gathered candidates, then Omega_t.
        allc = torch.cat(cands)
        sel, ns = ops[0].select(allc, allc.shape[0], tprime)
        ref_c, nref = mad.mad_topk(one.ctx.ctx, tprime)
        assert ns == nref
        assert np.array_equal(sel[:ns].cpu().numpy(), ref_c[:nref].cpu().numpy())
        res, nr = ops[0].rescore(sel, ns, t)
        ref, nrr = mad.mad_rescore(one.ctx.ctx, ref_c, nref, t)
        assert nr == nrr
        assert np.array_equal(res[:nr].cpu().numpy(), ref[:nrr].cpu().numpy())
        keys, c = one.oracle.run(s, seed, tprime, t)
        gi, gj, _, gc = mad.decode_pairs(res, nr)
        assert np.array_equal(mad.keys_of(gi, gj), keys)
        assert np.array_equal(gc.view(np.int64), c.view(np.int64))
    finally:
        for c in ranks + [one]:
            c.close()


def test_select_pairs_orders_and_filters():
    """x <= 0 is never selected; ties in x go to the smaller key; fewer
    positive pairs than K returns them all."""
    import paper_1506_03872_gb300 as mad
    c = Case("plain_small", s_max=1 << 16)
    try:
        i = np.array([5, 3, 9, 3, 1, 7])
        j = np.array([1, 2, 0, 1, 4, 7])
        x = np.array([4, 4, -2, 9, 0, 4])
        pairs = mad.encode_pairs(i, j, x)
        out, n = mad.mad_select_pairs(c.ctx.ctx, pairs, 6, 10)
        gi, gj, gx, _ = mad.decode_pairs(out, n)
        assert n == 4
        assert list(zip(gi.tolist(), gj.tolist(), gx.tolist())) == [
            (3, 1, 9), (3, 2, 4), (5, 1, 4), (7, 7, 4)]
        out, n = mad.mad_select_pairs(c.ctx.ctx, pairs, 6, 2)
        assert n == 2
    finally:
        c.close()


@pytest.mark.parametrize("name", ["chung_lu_small", "bipartite_binary"])
@pytest.mark.parametrize("first", [0, 30_000])
def test_binary_x_takes_more_pairs_than_its_budget_draws(name, first):
    """Partial X of other runs merged into a 0/1 context: the table, sized for
    the context's own diamonds, grows before the added pairs fill it."""
    import paper_1506_03872_gb300 as mad
    s = 60_000
    c = Case(name, s_max=s)
    try:
        ctx = c.ctx.ctx
        if first:
            mad.mad_sample(ctx, first, 5)
        own_k, own_v = _x_sorted(mad, ctx, s + 1)
        cap = mad.mad_stats(ctx)["hash_capacity"]
        rng = np.random.Generator(np.random.PCG64(1))
        flat = rng.permutation(c.m * c.n)
        i, j = flat // c.n, flat % c.n
        if c.flags & 2:
            i, j = i[i < j], j[i < j]
        n = s   # (what s_max / 0.6 slots hold)
        assert n > cap or name == "bipartite_binary"
        k = (i[:n].astype(np.uint64) << np.uint64(32)) | j[:n].astype(np.uint64)
        v = rng.integers(1, 9, n)
        for a in range(0, n, n // 3 + 1):   # in three calls
            b = a + n // 3 + 1
            mad.mad_accumulate(ctx, torch.from_numpy(k[a:b].view(np.int64).copy()).cuda(),
                               torch.from_numpy(v[a:b].copy()).cuda())
        want = dict(zip(own_k.tolist(), own_v.tolist()))
        for key, val in zip(k.tolist(), v.tolist()):
            want[key] = want.get(key, 0) + val
        gk, gv = _x_sorted(mad, ctx, 4 * cap)
        wk = np.array(sorted(want), dtype=np.uint64)
        assert np.array_equal(gk, wk)
        assert np.array_equal(gv, np.array([want[x] for x in wk.tolist()]))
        st = mad.mad_stats(ctx)
        assert st["device_error"] == 0 and st["distinct"] == len(wk)
        top, nt = mad.mad_topk(ctx, 50)
        assert nt == 50
        # The grown table serves the next run as the first one did.
        mad.mad_reset_hash(ctx)
        mad.mad_sample(ctx, s, 9)
        o = c.oracle
        assert o.sample(s, 9) == 0
        ok, ov = o.x()
        gk, gv = _x_sorted(mad, ctx, s + 1)
        assert np.array_equal(gk, ok) and np.array_equal(gv, ov)
    finally:
        c.close()


def test_binary_x_without_memory_to_grow(monkeypatch):
    """The growth is a service, not a need: where its memory is refused, pairs
    that the table holds are added all the same, and a table that fills up is
    reported."""
    import paper_1506_03872_gb300 as mad
    c = None
    for n in range(1, 100):
        monkeypatch.setenv("MAD_FAULT", f"oom:{n}")
        try:
            c = Case("chung_lu_small", s_max=60_000)   # (its allocations succeed; the next fails)
            break
        except mad.MadError as e:
            assert e.status == mad.MAD_ERR_OOM
    monkeypatch.delenv("MAD_FAULT")
    try:
        ctx = c.ctx.ctx
        cap = mad.mad_stats(ctx)["hash_capacity"]
        rng = np.random.Generator(np.random.PCG64(2))
        flat = rng.permutation(c.m * c.m)
        i, j = flat // c.m, flat % c.m
        i, j = i[i < j], j[i < j]
        k = (i.astype(np.uint64) << np.uint64(32)) | j.astype(np.uint64)
        n = cap // 2
        mad.mad_accumulate(ctx, torch.from_numpy(k[:n].view(np.int64).copy()).cuda(),
                           torch.ones(n, dtype=torch.int64, device="cuda"))
        st = mad.mad_stats(ctx)
        assert st["hash_capacity"] == cap and st["distinct"] == n and st["device_error"] == 0
        rest = k[n:2 * cap]
        mad.mad_accumulate(ctx, torch.from_numpy(rest.view(np.int64).copy()).cuda(),
                           torch.ones(len(rest), dtype=torch.int64, device="cuda"))
        with pytest.raises(mad.MadError) as e:
            mad.mad_topk(ctx, 10)
        assert e.value.status == mad.MAD_ERR_HASH_FULL
    finally:
        c.close()
