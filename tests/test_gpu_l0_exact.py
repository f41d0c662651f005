"""The exhaustive search on targets and columns that a fast Gram matrix and a
fast bound get wrong: a constant target, columns of near-equal magnitudes over
many samples, columns whose bulk lies far below their largest value."""
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


def search(env, X, y, dim, top):
    """The search over the columns X themselves (primaries, each stored)."""
    torch, oracle, dse, W = env
    sp = dse.Space(torch.from_numpy(X).cuda(), None, W.mask(W.MUL), 1)
    assert sp.n_stored == len(X)
    out = sp.l0_search(torch.from_numpy(y).cuda(), np.arange(len(X), dtype=np.uint64), dim, top)
    sp.free()
    return out


def rmse_of(cols, y):
    A = np.column_stack([np.ones(len(y))] + list(cols))
    r = y - A @ np.linalg.lstsq(A, y, rcond=None)[0]
    return np.sqrt(np.mean(r * r))


def frame(g, N, count, spikes=()):
    """Orthonormal mean-free vectors of N samples: one along each sample of `spikes`, then `count` random ones."""
    A = np.zeros((N, 1 + len(spikes) + count))
    A[:, 0] = 1.0
    for k, s in enumerate(spikes):
        A[s, 1 + k] = 1.0
    A[:, 1 + len(spikes):] = g.standard_normal((N, count))
    return np.linalg.qr(A)[0].T[1:]


@pytest.mark.parametrize("dim", [1, 2, 3])
@pytest.mark.parametrize("value", [0.0, 3.0])
def test_constant_target(env, dim, value):
    """Every full-rank subset explains a constant target: RMSE 0, in the order of the positions, as the oracle has it."""
    torch, oracle, dse, W = env
    w = W.tiny(0)
    kw = dict(unit_check_addsub=w["unit_check_addsub"], explog_dimensionless=w["explog_dimensionless"])
    sp = dse.Space(torch.from_numpy(w["X"]).cuda(), w["units"], w["op_mask"], w["max_rung"], **kw)
    orc = oracle.Space(w["X"], w["units"], w["op_mask"], w["max_rung"], **kw)
    ids = np.sort(orc.screen(w["Y"][0], 40)[0][0]).astype(np.uint64)
    y = np.full(w["X"].shape[1], value)
    opos, orm = orc.l0_search(y, ids, dim, 10)
    pos, rm, cf = sp.l0_search(y, ids, dim, 10)
    assert len(pos) == len(opos) == 10 and np.all(rm == 0.0) and np.all(np.abs(orm) < 1e-12)
    assert np.all(cf[:, 0] == value) and np.all(cf[:, 1:] == 0.0)
    assert pos.tolist() == opos.tolist()
