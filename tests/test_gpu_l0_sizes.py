"""The exhaustive search at the sizes where its Gram tiles (128 x 64 columns),
digit blocks (512 samples) and panels end, against numpy in FP64.

The best subsets' RMSEs agree to 1e-9 (least squares of up to three columns of
condition below 1e4: 1e4 * N * 1.1e-16 < 2e-9 of the norm, squared in the
RMSE); columns with one sign and near-equal values make every digit product of
a block add up."""
import itertools

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
    from paper_2602_06986_gb300 import dse
    from paper_2602_06986_gb300 import workloads as W

    return torch, dse, W


def rmse_of(cols, y):
    A = np.column_stack([np.ones(len(y))] + list(cols))
    r = y - A @ np.linalg.lstsq(A, y, rcond=None)[0]
    return np.sqrt(np.mean(r * r))


@pytest.mark.parametrize("N,n,dim", [(17, 3, 1), (17, 3, 3), (511, 63, 2), (512, 64, 2), (513, 65, 2), (1300, 129, 2),
                                     (1300, 30, 3), (600, 200, 1)])
@pytest.mark.parametrize("values", ["mixed", "flat"])
def test_sizes(env, N, n, dim, values):
    torch, dse, W = env
    g = np.random.Generator(np.random.PCG64(N + n + dim))
    n0 = 12
    X = g.lognormal(0.0, 0.7, size=(n0, N)) * 10.0 ** g.integers(-6, 7, size=(n0, 1))
    if values == "flat":  # one step: centred columns of two near-equal magnitudes
        X = np.where(g.random((n0, N)) < 0.5, 1.0, 3.0) + 1e-3 * g.random((n0, N))
    sp = dse.Space(torch.from_numpy(X).cuda(), None, W.mask(W.MUL, W.DIV, W.ADD), 2)
    ids = np.sort(g.choice(sp.n_stored, n, replace=False)).astype(np.uint64)
    vals = np.stack([_column(sp, X, int(i)) for i in ids])
    y = vals[0] / vals[0].std() + vals[n // 2] / vals[n // 2].std() + 0.3 * g.standard_normal(N)
    pos, rm, cf = sp.l0_search(y, ids, dim, 8)
    subsets = list(itertools.combinations(range(n), dim))
    Z = vals - vals.mean(1, keepdims=True)
    Z = Z / np.linalg.norm(Z, axis=1, keepdims=True)
    yc = (y - y.mean()) / np.linalg.norm(y - y.mean())
    G, b = Z @ Z.T, Z @ yc
    S = np.array(subsets)
    sub = G[S[:, :, None], S[:, None, :]] + 1e-13 * np.eye(dim)
    q = np.einsum("ki,ki->k", b[S], np.linalg.solve(sub, b[S][..., None])[..., 0])
    best = np.argsort(-q)[:40]
    ref = np.sort([rmse_of(vals[list(subsets[k])], y) for k in best])[:len(rm)]
    assert np.all(np.abs(rm - ref) <= 1e-9 * ref + 1e-12), (rm, ref)
    for p, r, c in zip(pos, rm, cf):
        assert abs(rmse_of(vals[p], y) - r) <= 1e-9 * r + 1e-12
        assert abs(np.sqrt(np.mean((y - c[0] - c[1:] @ vals[p]) ** 2)) - r) <= 1e-9 * r + 1e-12


def _column(sp, X, i):
    rung, op, a, b = sp.decode(i)
    if rung == 0:
        return X[a]
    u, v = _column(sp, X, a), _column(sp, X, b)
    return u * v if op == 8 else u / v if op == 9 else v / u if op == 10 else u + v
