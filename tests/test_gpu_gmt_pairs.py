"""The multi-target Gram kernel in clusters of two CTAs (b-images of 1 GB and more) against one CTA a tile: the same
lists and counts for every slot width, with odd numbers of feature blocks and tiles, whole screens and id ranges.  The
sums of a tile do not depend on the launch, so the lists are equal to the bit."""
import numpy as np
import pytest

import __graft_entry__ as ge

pytestmark = pytest.mark.gpu


# stored rows: 6 n0 (unary) + 6 n0 (n0 - 1) / 2 (pairs) + n0, full library
@pytest.mark.parametrize("T,n0,N", [(4, 20, 17_009), (8, 20, 12_500), (16, 17, 12_100), (16, 17, 8_000)])
def test_pairs_and_single_blocks_agree(T, n0, N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ge.build()
    from paper_2602_06986_gb300 import dse
    from paper_2602_06986_gb300 import workloads as W

    g = np.random.Generator(np.random.PCG64(60 + T))
    X = W._f32(g.lognormal(0.0, 0.5, size=(n0, N)))
    Y = np.stack([X[t % n0] * X[(t + 1) % n0] / X[(t + 2) % n0] + 0.1 * g.standard_normal(N) for t in range(T)])
    sp = dse.Space(torch.from_numpy(X).cuda(), None, W.OPS_FULL, 2)
    rows, slots = sp.n_stored, {4: 15, 8: 9, 16: 6}[T]
    images = -(-rows // slots) * -(-N // 32) * (28 if T == 16 else 24) * 1024
    assert images >= 1 << 30  # (below it one CTA a tile is taken: test_gpu_gmt_targets.py)
    Yd = torch.from_numpy(Y).cuda()
    for begin, end in ((0, sp.n_total), (sp.n_stored + (sp.n_total - sp.n_stored) // 3, sp.n_total - 1001)):
        got = []
        try:
            for ctas in (1, 2):
                dse.set_tuning({"gmt_cluster": ctas})
                res = sp.screen(Yd, 300, precision=dse.PREC_BF16X3, id_begin=begin, id_end=end)
                st = res.stats()
                assert st["binary_path"] == dse.PATH_GRAM_MT and st["screened"] == end - begin
                got.append((st["reasons"], [res.fetch(t) for t in range(T)]))
                res.free()
        finally:
            dse.set_tuning(None)
        assert got[0][0] == got[1][0]
        for a, b in zip(got[0][1], got[1][1]):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
    sp.free()
