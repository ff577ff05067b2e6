"""Residual histories longer than the pinned buffer that comes with a solve's verdict, and a max_iter that
is large only in case: its residuals have room on the device, not in pinned host memory."""
import numpy as np
import pytest

from test_gpu_parity import OM, to_dev
from test_gpu_parity import dgp, torch_dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu
N, BOX, A, WSPLIT = 16, 16.0, 0.1, 0.82  # a splitting that converges slowly on this field


def _delta():
    rng = np.random.default_rng(1)
    d = np.exp(rng.normal(0, 0.6, (N, N, N)))
    return d / d.mean() - 1.0


@pytest.mark.parametrize("max_iter", [63, 64, 65, 300])
def test_long_history_follows_the_oracle(dgp, torch_dev, max_iter):
    """FP64 to 1e-11: the residuals agree to 1e-6 of themselves down to 1e-8, which is far above the rounding floor."""
    from oracle import field as ofield
    torch, dev = torch_dev
    delta = _delta()
    want = np.asarray(ofield.solve_phi(delta, A, BOX, OM, 1.0, tol=1e-11, max_iter=max_iter, w=WSPLIT)[3]["history"])
    assert len(want) > 63
    ctx = dgp.dgp_init(BOX, N, 1.0, OM, w=WSPLIT, precision=dgp.DGP_FP64, max_iter=max_iter, tol=1e-11)
    try:
        st, info = dgp.dgp_solve_phi(ctx, A, to_dev(torch_dev, delta, torch.float64), None, 1e-11)
        got = dgp.dgp_solve_history(ctx)
    finally:
        dgp.dgp_destroy(ctx)
    m = min(len(got), len(want))
    assert abs(len(got) - len(want)) <= 1
    sel = want[:m] > 1e-8
    assert sel.sum() >= min(max_iter + 1, 70)
    assert np.max(np.abs(got[:m][sel] / want[:m][sel] - 1)) < 1e-6
    assert got[info["iters"]] == info["norm_res"]


def test_long_histories_of_a_class(dgp, torch_dev):
    """Every member's history ends with the residual its step reports (tol within reach of FP32)."""
    torch, dev = torch_dev
    count, n, t = 3, N, []
    for k in range(count):  # particles on mesh points: delta as rough as the counts
        rng = np.random.default_rng(k)
        cell = np.repeat(np.arange(n ** 3), rng.poisson(30.0 * np.exp(0.6 * rng.normal(size=(n, n, n)))).reshape(-1))
        pos = [to_dev(torch_dev, c * (BOX / n), torch.float32) for c in (cell // (n * n), cell // n % n, cell % n)]
        t.append(pos + [torch.zeros(cell.size, device=dev) for _ in range(3)])
    torch.cuda.synchronize()
    plist = [dgp.params(BOX, n, 1.0, w=0.84, precision=dgp.DGP_FP32, tol=1e-6, max_iter=400)] * count
    b, ctxs = dgp.dgp_batch_create(plist, OM)
    try:
        assert dgp.dgp_batch_classes(b, count)[1] == 1
        infos = dgp.dgp_batch_step(b, [dgp.particles(*m) for m in t], [A] * count, [2.0 ** -50] * count)
        hist = [dgp.dgp_solve_history(c) for c in ctxs]
        for c, p in zip(ctxs, t):  # each member's solve of the same field from rest
            d = torch.empty((n, n, n), device=dev)
            dgp.dgp_deposit(c, dgp.particles(*p), d)
            dgp.dgp_reset(c)
            dgp.dgp_solve_phi(c, A, d, None, 1e-6)
            hist.append(dgp.dgp_solve_history(c))
    finally:
        dgp.dgp_batch_destroy(b)
    assert max(len(h) for h in hist) > 64
    for h in hist:
        assert np.all(np.isfinite(h)) and np.all(h > 0) and h[-1] == h.min()
    for i, h in zip(infos, hist):
        assert h[i["iters"]] == i["norm_res"]


def test_large_max_iter_pins_no_host_memory(dgp, torch_dev):
    """2e7 residuals are 160 MB."""
    import os

    def resident():
        with open("/proc/self/statm") as f:
            return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")

    torch, dev = torch_dev
    dgp.dgp_destroy(dgp.dgp_init(BOX, N, 1.0, OM, precision=dgp.DGP_FP32))
    before = resident()
    ctx = dgp.dgp_init(BOX, N, 1.0, OM, precision=dgp.DGP_FP32, max_iter=20000000)
    try:
        assert resident() - before < 40e6
    finally:
        dgp.dgp_destroy(ctx)
