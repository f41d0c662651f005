"""The multi-target Gram kernel's three tile widths (4, 8 and 16 target slots,
15, 9 and 6 b-features): target counts on both sides of each line, one sample
chunk to several accumulation blocks, and feature counts that leave a ragged
last b-block, against the CPU FP64 oracle (tolerances of test_gpu_parity.py)."""
import numpy as np
import pytest

import __graft_entry__ as ge

pytestmark = pytest.mark.gpu


def data(N, n0, seed):
    from paper_2602_06986_gb300 import workloads as W

    g = np.random.Generator(np.random.PCG64(seed))
    X = W._f32(g.uniform(0.3, 4.0, size=(n0, N)))
    X[1] = W._f32(X[1] - 2.0)  # both signs: quotients and logarithms of it are refused or escalated
    Y = np.stack([X[t % n0] * X[(t + 1) % n0] / X[(t + 2) % n0] + 0.1 * g.standard_normal(N) for t in range(16)])
    return X, Y


@pytest.mark.parametrize("T", [2, 3, 4, 5, 7, 8, 9, 16])
@pytest.mark.parametrize("N,n0", [(16, 3), (33, 4), (513, 3), (1100, 4)])
def test_target_slots(T, N, n0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ge.build()
    import oracle
    from paper_2602_06986_gb300 import dse
    from paper_2602_06986_gb300 import workloads as W

    X, Y = data(N, n0, 100 * T + N)
    Y = Y[:T]
    units = np.zeros((n0, 0), np.int32)
    sp = dse.Space(torch.from_numpy(X).cuda(), units, W.OPS_FULL, 2)
    orc = oracle.Space(X, units, W.OPS_FULL, 2)
    total = sp.n_total
    for begin, end in ((0, total), (sp.n_stored + (total - sp.n_stored) // 3, total - 7)):
        res = sp.screen(torch.from_numpy(Y).cuda(), 40, precision=dse.PREC_BF16X3, id_begin=begin, id_end=end)
        oids, osc, cnt = orc.screen(Y, 40, id_begin=begin, id_end=end)
        st = res.stats()
        assert st["binary_path"] == dse.PATH_GRAM_MT and st["reasons"] == cnt and st["screened"] == end - begin
        for t in range(T):
            ids, sc, eb = res.fetch(t)
            ge._check_topk(ids, sc, eb, oids[t], osc[t], orc, Y, t)
