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


def test_many_samples_of_one_magnitude(env):
    """A two-valued column over 300 000 samples: its squared sum is the largest that the digits' integer sums hold
    (several panels of samples).  It explains half of the target, 79 others 46 to 49%."""
    N, n, at = 300_000, 80, 41
    g = np.random.Generator(np.random.PCG64(5))
    X = np.empty((n, N))
    X[at] = np.where(np.arange(N) % 2, 2.998, 1.0)
    t = (X[at] - X[at].mean()) / X[at].std()
    w = g.standard_normal(N)
    w -= w.mean()
    w -= t * (w @ t) / N
    y = t + w / w.std()
    for k in range(n):
        if k != at:
            a = 0.46 + 0.03 * k / n
            X[k] = np.sqrt(a / 2) * y + np.sqrt(1 - a) * g.standard_normal(N)
    pos, rm, cf = search(env, X, y, 1, 16)
    ref = [rmse_of(X[k:k + 1], y) for k in range(n)]
    order = np.argsort(ref)
    assert pos[:, 0].tolist() == order[:16].tolist() and order[0] == at
    assert np.all(np.abs(rm - np.array(ref)[order[:16]]) <= 1e-9 * rm)


def test_bound_of_columns_with_a_far_value(env):
    """Two columns of which one sample each holds 40% of the squared norm explain slightly more (3e-6 of the target's
    square) than each of the 600 pairs around another column: the FP32 bound may not exclude them."""
    N, n, q = 60_000, 700, 2 * 0.68 ** 2 / 1.5
    g = np.random.Generator(np.random.PCG64(6))
    E0, E1, u, v0, v1, w, g2 = frame(g, N, 5, spikes=(1234, 45678))
    p = [np.sqrt(0.4) * E + np.sqrt(0.5) * u + np.sqrt(0.1) * v for E, v in ((E0, v0), (E1, v1))]
    c = 0.68
    y = c / np.sqrt(0.5) * u + np.sqrt(1 - 2 * c * c) * w
    a = q - 3e-6
    good = np.sqrt(a) * y + np.sqrt(1 - a) * g2
    X = np.empty((n, N))
    X[:] = g.standard_normal((n, N))
    X -= X.mean(1, keepdims=True)
    for b in (y, g2):
        X -= np.outer(X @ b, b)
    X[70] = good
    X[n - 2], X[n - 1] = (1.0001 * v / np.abs(v).max() for v in p)  # just above a power of two
    pos, rm, _ = search(env, X, y, 2, 8)
    found = [tuple(v) for v in pos.tolist()]
    assert (n - 2, n - 1) in found[:3]
    for (i, j), r in list(zip(found, rm))[:3]:
        ref = rmse_of(X[[i, j]], y)
        assert abs(r - ref) <= 1e-9 * ref


def test_near_equal_columns_with_a_far_value(env):
    """Two columns that one sample dominates and whose angle is 6e-7 explain 98% of the target: their squared sine,
    4e-13, has to survive the Gram matrix's rounding."""
    N, n = 20_000, 20
    g = np.random.Generator(np.random.PCG64(7))
    E0, z, w = frame(g, N, 2, spikes=(777,))
    X = g.standard_normal((n, N))
    x = E0 + 0.01 * (X[0] / np.linalg.norm(X[0]))
    x *= 1.0001 / np.abs(x).max()
    X[3], X[11] = x, x + np.sqrt(4e-13) * np.linalg.norm(x) * z
    y = np.sqrt(0.98) * z + np.sqrt(0.02) * w
    pos, rm, _ = search(env, X, y, 2, 4)
    assert pos[0].tolist() == [3, 11]
    assert abs(rm[0] / y.std() - np.sqrt(0.02)) <= 0.01


@pytest.mark.parametrize("dim", [1, 2, 3])
def test_little_memory(env, dim):
    """Where the first allocation fails, the search does without the FP32 copy and with short panels: the same subsets."""
    torch, oracle, dse, W = env
    N, n = 700, 130 if dim < 3 else 40
    g = np.random.Generator(np.random.PCG64(8))
    X = g.lognormal(0.0, 0.7, size=(n, N))
    y = X[3] / X[3].std() + 0.7 * X[n // 2] / X[n // 2].std() + 0.5 * g.standard_normal(N)
    ref = search(env, X, y, dim, 12)
    sp = dse.Space(torch.from_numpy(X).cuda(), None, W.mask(W.MUL), 1)
    yd, ids = torch.from_numpy(y).cuda(), torch.arange(n, dtype=torch.int64, device="cuda")
    try:
        dse.debug_fail_alloc(0)
        got = sp.l0_search(yd, ids, dim, 12)
    finally:
        dse.debug_fail_alloc(-1)
    assert len(ref[0]) == 12
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
