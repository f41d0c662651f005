"""Lists fetched into host and device memory, in any order and from several threads."""
import ctypes as C
import threading

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


K = 30


@pytest.fixture(scope="module")
def batch(env):
    torch, dse, W = env
    g = np.random.Generator(np.random.PCG64(31))
    X = W._f32(g.lognormal(0.0, 0.5, size=(6, 80)))
    rows = [np.sort(g.choice(80, 64, replace=False)).astype(np.int64) for _ in range(41)]
    spaces = [dse.Space(torch.from_numpy(X).cuda(), None, W.OPS_FULL, 2, sample_idx=r) for r in rows]
    Y = [X[0, r] * X[1, r] + 0.1 * g.standard_normal(64) for r in rows]
    return dse.Batch(spaces, Y, K), [y[::-1].copy() for y in Y]


def direct(env, b, i):
    """List i through device memory: no copy of other lists is involved."""
    torch, dse, W = env
    out = [torch.zeros(K, dtype=t, device="cuda") for t in (torch.int64, torch.float64, torch.float64)]
    n = C.c_int64()
    assert dse.lib().dse_batch_fetch(b._h, i, *(t.data_ptr() for t in out), K, C.byref(n)) == dse.OK
    return [t[:n.value].cpu().numpy() for t in out]


def same(a, b):
    return all(np.array_equal(x.astype(y.dtype), y) for x, y in zip(a, b))


def test_batch_lists_in_any_order(env, batch):
    torch, dse, W = env
    b, other = batch
    n = len(b.spaces)
    g = np.random.Generator(np.random.PCG64(32))
    for new in (False, True):
        if new:
            b.rescreen(torch.from_numpy(np.concatenate(other)).cuda())
        first = b.fetch(0)  # (before any other list)
        ref = [direct(env, b, i) for i in range(n)]
        assert same(first, ref[0]) and all(len(r[0]) == K for r in ref)
        for order in (range(n), reversed(range(n)), g.permutation(n), [5, 6, 7, 3, 8, 9, 10, 11, 40, 0, 1, 2]):
            for i in order:
                assert same(b.fetch(int(i)), ref[i]), i


def test_batch_lists_from_several_threads(env, batch):
    """Each of four threads fetches every list, from another start on."""
    b, _ = batch
    n = len(b.spaces)
    ref = [direct(env, b, i) for i in range(n)]
    wrong = []

    def work(t):
        for _ in range(20):
            for i in range(n):
                j = (i + 11 * t) % n
                if not same(b.fetch(j), ref[j]):
                    wrong.append((t, j))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("shift", [0, 1, 4, 8])
def test_device_arrays_of_any_alignment(env, shift):
    """A list of a screen into device bytes at any offset: the values of the host fetch, and nothing beyond them."""
    torch, dse, W = env
    w = W.tiny(0)
    sp = dse.Space(torch.from_numpy(w["X"]).cuda(), w["units"], w["op_mask"], w["max_rung"])
    res = sp.screen(torch.from_numpy(w["Y"]).cuda(), K)
    ref = res.fetch(0)
    out = [torch.full((8 * K + 32,), 0x5A, dtype=torch.uint8, device="cuda") for _ in range(3)]
    n = C.c_int64()
    assert dse.lib().dse_topk_fetch(res._h, 0, *(t.data_ptr() + shift for t in out), K, C.byref(n)) == dse.OK
    torch.cuda.synchronize()
    assert n.value == len(ref[0]) > 0
    for t, r in zip(out, ref):
        b = t.cpu().numpy()
        assert b[shift:shift + 8 * n.value].tobytes() == r.tobytes()
        assert np.all(b[:shift] == 0x5A) and np.all(b[shift + 8 * n.value:] == 0x5A)
