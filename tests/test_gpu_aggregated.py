"""Aggregated lists (sqrt of the mean squared score over the targets) against the oracle's whole ranking: a candidate
that a pair kernel loses or scores too low is missing here.  Target counts on both sides of the kernels' slots (4, 8,
16), sample counts that end in a ragged chunk, and on both sides of the two re-score kernels (N = 4096).

Tolerance 1e-5 of the score, as in test_gpu_parity.py: outside a band of twice that around the last score the lists
are the same sets."""
import numpy as np
import pytest

import __graft_entry__ as ge

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ge.build()
    import oracle
    from paper_2602_06986_gb300 import dse
    from paper_2602_06986_gb300 import workloads as W

    return torch, oracle, dse, W


@pytest.mark.parametrize("N,n0,dims", [(33, 7, 0), (257, 9, 2), (1001, 6, 0), (4096, 5, 0), (4099, 5, 2)])
@pytest.mark.parametrize("T", [2, 4, 5, 8, 9, 16])
def test_whole_ranking(env, N, n0, dims, T):
    torch, oracle, dse, W = env
    g = np.random.Generator(np.random.PCG64(50 + N + T))
    X = W._f32(g.lognormal(0.0, 0.5, size=(n0, N)))
    units = g.integers(-1, 2, size=(n0, dims)).astype(np.int32)
    Y = np.stack([X[t % n0] * X[(t + 1) % n0] / X[(t + 2) % n0] + 0.3 * g.standard_normal(N) for t in range(T)])
    k = 150
    sp = dse.Space(torch.from_numpy(X).cuda(), units, W.OPS_FULL, 2)
    orc = oracle.Space(X, units, W.OPS_FULL, 2)
    oids, osc, cnt = orc.screen(Y, k, mode="aggregated")
    oids, osc = np.asarray(oids[0]), np.asarray(osc[0])
    res = sp.screen(torch.from_numpy(Y).cuda(), k, mode=dse.MODE_AGGREGATED, precision=dse.PREC_FP32)
    ids, sc, eb = res.fetch(0)
    assert res.stats()["reasons"] == cnt and len(ids) == len(oids) == k and len(set(ids.tolist())) == k
    last = osc[-1]
    assert {int(i) for i, s in zip(oids, osc) if s > last * (1 + 2 * TOL)} <= {int(i) for i in ids}
    ref = np.sqrt(np.mean(orc.score_ids(Y, ids)[0] ** 2, axis=1))
    assert np.all(np.abs(sc - ref) <= TOL * ref) and np.all(np.abs(sc - ref) <= eb + 1e-12)
    assert np.all(np.diff(sc) <= 0) and np.all(ref >= last * (1 - 2 * TOL))
    # rank by rank (ties may swap ids, not scores)
    assert np.all(np.abs(sc - osc) <= TOL * osc)
