"""A member of a class that stops on its patience returns the iterate of its lowest residual, which the
class regenerates by replaying that member's iterations alone.  The replay must give the bits of the
iterate the class examined.

Two runs of the same class: the first with tol = 0, so that its members stop on patience after their
best iterate b; the second with each member's max_iter = b, so that the member ends on iterate b itself, with
nothing to replay.  The solves see the same field to the bit: the particles sit at cell midpoints (CIC
weights 1/8, whose sums are exact in any order) and a step of some ulp of a moves none of them.  A step
makes two solves (forces before and after the drift); where the first one's best iterate comes after b
the second run starts its second solve elsewhere, which its residuals show: those members are left out."""
import ctypes

import numpy as np
import pytest

from test_gpu_parity import OM
from test_gpu_parity import dgp, torch_dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def _particles(torch, dev, n, seed):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    rate = 4.0 * torch.exp(0.6 * torch.randn((n, n, n), generator=g, device=dev))
    num = torch.poisson(rate, generator=g).long().reshape(-1)
    cell = torch.repeat_interleave(torch.arange(n ** 3, device=dev), num)
    pos = [(c.float() + 0.5) * 2.0 for c in (cell // (n * n), cell // n % n, cell % n)]
    return [p.contiguous() for p in pos] + [torch.zeros(cell.numel(), device=dev) for _ in range(3)]


def _run(dgp, torch, dev, n, prec, plane, seed, max_iter):
    """One class step: (best iterates, residual histories, accepted solutions)."""
    count, a, da = len(max_iter), 0.5, 2.0 ** -50
    t = [_particles(torch, dev, n, seed + k) for k in range(count)]
    start = [[v.clone() for v in m[:3]] for m in t]
    parts = (dgp.Particles * count)(*[dgp.particles(*m) for m in t])
    plist = [dgp.params(2.0 * n, n, 0.8 + 0.05 * k, precision=prec, tol=0.0, max_iter=m)
             for k, m in enumerate(max_iter)]
    torch.cuda.synchronize()
    b, ctxs = dgp.dgp_batch_create(plist, OM)
    try:
        dgp.dgp_batch_set_plane_pass(b, plane)
        assert dgp.dgp_batch_classes(b, count)[1] == 1
        infos = (dgp.SolveInfo * count)()
        assert dgp.lib.dgp_batch_step(b, parts, (ctypes.c_double * count)(*[a] * count),
                                      (ctypes.c_double * count)(*[da] * count), infos, None) == dgp.DGP_OK
        sol = []
        for c in ctxs:
            sol.append(torch.empty((n, n, n), device=dev))
            dgp.dgp_get_solution(c, sol[-1])
        torch.cuda.synchronize()
        hist = [dgp.dgp_solve_history(c) for c in ctxs]
    finally:
        dgp.dgp_batch_destroy(b)
    assert all(torch.equal(x, y) for m, s in zip(t, start) for x, y in zip(m, s))
    return [i.iters for i in infos], hist, sol


@pytest.mark.parametrize("n,prec,plane", [(16, "DGP_FP32", True), (32, "DGP_MIXED_EFT", True),
                                          (48, "DGP_FP32", True), (48, "DGP_FP32", False),
                                          (48, "DGP_MIXED_F32R", True), (48, "DGP_MIXED_EFT", False),
                                          (64, "DGP_MIXED", True), (96, "DGP_MIXED_EFT", True)])
def test_replayed_member_holds_the_iterate_it_reports(dgp, torch_dev, n, prec, plane):
    torch, dev = torch_dev
    prec, count = getattr(dgp, prec), 16 if n < 96 else 8
    same, differ = [], []
    for seed in range(100 * n, 100 * n + 3 * count, count):  # three sets of fields
        best, hist, sol = _run(dgp, torch, dev, n, prec, plane, seed, [100] * count)
        _, hist2, sol2 = _run(dgp, torch, dev, n, prec, plane, seed, best)
        sel = [k for k in range(count) if 0 < best[k] < len(hist[k]) - 1
               and np.array_equal(hist2[k], hist[k][:best[k] + 1])]
        same += [seed + k for k in sel]
        differ += [seed + k for k in sel if not torch.equal(sol[k], sol2[k])]
    assert same
    assert not differ, (same, differ)
