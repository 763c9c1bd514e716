"""X of dense Gram inputs whose row norms rise, fall or differ by orders of
magnitude along the row index (the order decides which regions of the hash
the keys start in), against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("order", ["rising", "falling", "one_heavy", "equal"])
@pytest.mark.parametrize("flags", [2, 2 | 4])
def test_x_of_ordered_norms(order, flags):
    import paper_1506_03872_gb300 as mad
    rng = np.random.Generator(np.random.PCG64(90))
    m, d, s = 701, 20, 150_000
    A = rng.standard_normal((m, d))
    scale = {"rising": np.exp(np.linspace(-2, 2, m)), "falling": np.exp(np.linspace(2, -2, m)),
             "one_heavy": np.where(np.arange(m) == 650, 300.0, 1.0), "equal": np.ones(m)}[order]
    A *= scale[:, None]
    B = np.ascontiguousarray(A.T)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    o = oracle.Oracle(oracle.Matrix(A), oracle.Matrix(B), flags, s)
    assert o.sample(s, 7) == 0
    keys, x = o.x()
    with mad.Context(flags) as c:
        c.build(mad.dense(tA), mad.dense(tB), s, keep=(tA, tB))
        mad.mad_sample(c.ctx, s // 2, 7)
        mad.mad_sample(c.ctx, s - s // 2, 7, s // 2)
        gk, gx, n = mad.mad_export_x(c.ctx, s)
    gk, gx = gk.cpu().numpy().view(np.uint64), gx.cpu().numpy()
    assert n == len(keys)
    a, b = np.argsort(gk), np.argsort(keys)
    assert np.array_equal(gk[a], np.asarray(keys, np.uint64)[b])
    assert np.array_equal(gx[a], np.asarray(x)[b])
