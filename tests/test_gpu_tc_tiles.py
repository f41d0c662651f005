"""The tensor-core screen's tile shapes (16 x 8, 8 x 16 and 4 x 32 rows): id
ranges whose last row block holds 1 to 16 rows, and a first or last row taken
in part, against the CPU FP64 oracle (tolerances of test_gpu_parity.py)."""
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

    g = np.random.Generator(np.random.PCG64(77))
    X = W._f32(g.uniform(0.3, 4.0, size=(4, 67)))
    Y = np.stack([X[t % 4] * X[(t + 1) % 4] / X[(t + 2) % 4] + 0.1 * g.standard_normal(67) for t in range(17)])
    units = np.zeros((4, 0), np.int32)
    sp = dse.Space(torch.from_numpy(X).cuda(), units, W.OPS_FULL, 2)
    orc = oracle.Space(X, units, W.OPS_FULL, 2)
    return torch, dse, sp, orc, Y


def first_id(sp, row, j):
    """Id of the first slot of pair (row, j) of the last rung (full operator library, 4 primaries stored first)."""
    n, o = sp.n_stored, 4
    pairs = row * (row - 1) // 2 - o * (o - 1) // 2 + j
    return n + 6 * (n - o) + 6 * pairs


@pytest.mark.parametrize("rows", [1, 2, 4, 5, 8, 9, 12, 13, 16, 17, 21])
@pytest.mark.parametrize("cut", [0, 3])
def test_row_blocks(env, rows, cut):
    torch, dse, sp, orc, Y = env
    i0 = 20
    begin = first_id(sp, i0, 0) + 5 * cut            # cut: part of the first and of the last row
    end = first_id(sp, i0 + rows, 0) - 11 * cut
    res = sp.screen(torch.from_numpy(Y).cuda(), 25, precision=dse.PREC_BF16X3, id_begin=begin, id_end=end)
    oids, osc, cnt = orc.screen(Y, 25, id_begin=begin, id_end=end)
    st = res.stats()
    assert st["binary_path"] == dse.PATH_TENSOR and st["reasons"] == cnt and st["screened"] == end - begin
    for t in range(len(Y)):
        ids, sc, eb = res.fetch(t)
        ge._check_topk(ids, sc, eb, oids[t], osc[t], orc, Y, t)


def test_first_tiles_leave_room():
    """20 M candidates in full tiles: the tiles scored before the first thresholds exist must not fill the buffers
    (a list that overflows is screened a second time)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ge.build()
    from paper_2602_06986_gb300 import dse
    from paper_2602_06986_gb300 import workloads as W

    w = W.precision(seed=0)
    X, Y = np.ascontiguousarray(w["X"][:, :64]), np.ascontiguousarray(w["Y"][:, :64])
    sp = dse.Space(torch.from_numpy(X).cuda(), w["units"], w["op_mask"], 3)
    begin = sp.n_stored + 6 * sp.n_stored + w["block_seed"]
    st = sp.screen(torch.from_numpy(Y).cuda(), 1000, precision=dse.PREC_BF16X3, id_begin=begin,
                   id_end=begin + 20_000_000).stats()
    assert st["binary_path"] == dse.PATH_TENSOR and st["screened"] == 20_000_000 and st["reruns"] == 0
