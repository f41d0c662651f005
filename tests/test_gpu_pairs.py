"""The CUDA-core pair kernels at the sizes where their tiles, sample chunks and
target blocks end: against the CPU FP64 oracle.

Tolerances as in test_gpu_parity.py (1e-5 relative, and the reported bounds);
FP64 screens 1e-9 (sums of up to 1001 products, condition numbers of the
centred sums below 1e4: 1001 * 1e4 * 1.1e-16)."""
import numpy as np
import pytest

import __graft_entry__ as ge

pytestmark = pytest.mark.gpu


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


def problem(W, N, n0, T, dims, seed):
    g = np.random.Generator(np.random.PCG64(900 + seed))
    X = W._f32(g.lognormal(0.0, 0.5, size=(n0, N)))
    units = g.integers(-1, 2, size=(n0, dims)).astype(np.int32)
    Y = np.stack([X[t % n0] * X[(t + 1) % n0] / X[(t + 2) % n0] + 0.05 * g.standard_normal(N) for t in range(T)])
    return X, units, Y


# chunks of 32 samples, odd and even tails; dims 0: every pair may be added (tiles), 2: the equal-unit pair list
@pytest.mark.parametrize("N,n0,dims", [(16, 5, 0), (31, 6, 2), (32, 7, 0), (33, 9, 0), (95, 8, 2), (257, 10, 0), (1001, 6, 0)])
@pytest.mark.parametrize("T", [1, 2, 4, 5, 8, 9])
def test_pair_kernels(env, N, n0, dims, T):
    torch, oracle, dse, W = env
    X, units, Y = problem(W, N, n0, T, dims, N + T)
    k = 40
    sp = dse.Space(torch.from_numpy(X).cuda(), units, W.OPS_FULL, 2)
    orc = oracle.Space(X, units, W.OPS_FULL, 2)
    Yd = torch.from_numpy(Y).cuda()
    oids, osc, cnt = orc.screen(Y, k)
    res = sp.screen(Yd, k, precision=dse.PREC_FP32, flags=dse.FLAG_DIRECT)
    st = res.stats()
    assert st["reasons"] == cnt and st["binary_path"] == dse.PATH_CUDA_CORE and st["reruns"] == 0
    for t in range(T):
        ids, sc, eb = res.fetch(t)
        ge._check_topk(ids, sc, eb, oids[t], osc[t], orc, Y, t)
    res.free()
    if T == 1:
        res = sp.screen(Yd, k, precision=dse.PREC_FP64)
        assert res.stats()["reasons"] == cnt
        ids, sc, eb = res.fetch(0)
        ge._check_topk(ids, sc, eb, oids[0], osc[0], orc, Y, 0, tol=1e-9)
    else:
        res = sp.screen(Yd, k, mode=dse.MODE_AGGREGATED, precision=dse.PREC_FP32)
        assert res.stats()["reasons"] == cnt
        ids, sc, eb = res.fetch(0)
        ref = np.sqrt(np.mean(orc.score_ids(Y, ids)[0] ** 2, axis=1))
        assert np.all(np.abs(sc - ref) <= 1e-5 * ref) and np.all(np.diff(sc) <= 0)


def test_pair_kernels_ranges(env):
    """Range screens (a part of the pair triangle) merge to the whole, FP32 and FP64."""
    torch, oracle, dse, W = env
    X, units, Y = problem(W, 130, 9, 1, 0, 3)
    sp = dse.Space(torch.from_numpy(X).cuda(), units, W.OPS_FULL, 2)
    Yd = torch.from_numpy(Y).cuda()
    for prec in (dse.PREC_FP32, dse.PREC_FP64):
        full = sp.screen(Yd, 30, precision=prec, flags=dse.FLAG_DIRECT).fetch(0)
        cuts = [0, 17, sp.n_stored + 5, sp.n_stored + sp.n_total // 3, sp.n_total]
        parts = [sp.screen(Yd, 30, precision=prec, flags=dse.FLAG_DIRECT, id_begin=a, id_end=b).fetch(0)
                 for a, b in zip(cuts, cuts[1:])]
        ids = np.concatenate([p[0] for p in parts])
        sc = np.concatenate([p[1] for p in parts])
        top = np.sort(sc)[::-1][:30]
        assert np.all(np.abs(top - full[1]) <= 2e-5 * full[1]) and set(full[0].tolist()) <= set(ids.tolist())
