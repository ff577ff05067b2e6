"""Edges of the estimator, sort, initial-condition and adjoint kernels: magnitudes far from one,
shell counts and angle counts that do not fill a launch, pointers that are not 16-byte aligned, and
every row split of the relaxation pass and of the adjoint's fused z pass.

Tolerances: scaling a field by a power of two is exact in every step, so spectra scale exactly;
a shorter list of shells and angles taken one at a time use the same sums, so they are equal; an
unaligned pointer changes only how values are moved.  The FP32 adjoint (both solves to 1e-6) against
FP64 (1e-12): the bound of the FP32 comparison with the oracle, 1e-4."""
import math

import numpy as np
import pytest

from test_gpu_parity import OM, rel_l2
from test_gpu_parity import dgp, torch_dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def _field(torch, dev, n, seed):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return torch.randn((n, n, n), generator=g, device=dev)


@pytest.mark.parametrize("n", [16, 48, 64])
@pytest.mark.parametrize("e", [-60, -31, 40])
def test_spectra_scale_with_the_field(dgp, torch_dev, n, e):
    """|delta_k|^2 of these fields leaves the FP32 range without the per-CTA scale."""
    torch, dev = torch_dev
    d = _field(torch, dev, n, n)
    ctx = dgp.dgp_init(100.0, n, 1.0, OM, precision=dgp.DGP_FP32)
    try:
        k0, p0, c0 = dgp.power_spectrum(ctx, d, n // 2)
        k1, p1, c1 = dgp.power_spectrum(ctx, d * 2.0 ** e, n // 2)
        kf = 2 * math.pi / 100.0
        th = [0.3, 1.1, 2.0]
        b0, q0 = dgp.bispectrum(ctx, d, 3 * kf, 4 * kf, th)
        b1, q1 = dgp.bispectrum(ctx, d * 2.0 ** e, 3 * kf, 4 * kf, th)
    finally:
        dgp.dgp_destroy(ctx)
    assert np.array_equal(k0, k1) and np.array_equal(c0, c1)
    assert np.all(p0 > 0) and np.array_equal(p1, p0 * 2.0 ** (2 * e))
    assert np.array_equal(b1, b0 * 2.0 ** (3 * e))
    assert np.allclose(q1, q0 * 2.0 ** -e, rtol=1e-14, atol=0)


@pytest.mark.parametrize("n,nbins", [(16, 1), (32, 7), (96, 33), (128, 63)])
def test_fewer_shells_are_the_first_of_all(dgp, torch_dev, n, nbins):
    torch, dev = torch_dev
    d = _field(torch, dev, n, 3)
    ctx = dgp.dgp_init(100.0, n, 1.0, OM, precision=dgp.DGP_FP32)
    try:
        full = dgp.power_spectrum(ctx, d, n // 2)
        part = dgp.power_spectrum(ctx, d, nbins)
    finally:
        dgp.dgp_destroy(ctx)
    for a, b in zip(full, part):
        assert np.array_equal(a[:nbins], b)


@pytest.mark.parametrize("n,ntheta", [(16, 1), (16, 7), (16, 8), (16, 20), (32, 16)])
def test_angles_in_groups_equal_angles_one_by_one(dgp, torch_dev, n, ntheta):
    """The sums of an angle are read back in groups of up to n / 2."""
    torch, dev = torch_dev
    d = _field(torch, dev, n, 5)
    kf = 2 * math.pi / 100.0
    th = [0.05 + 3.0 * i / ntheta for i in range(ntheta)]
    ctx = dgp.dgp_init(100.0, n, 1.0, OM, precision=dgp.DGP_FP32)
    try:
        b, q = dgp.bispectrum(ctx, d, 2 * kf, 3 * kf, th)
        one = [dgp.bispectrum(ctx, d, 2 * kf, 3 * kf, [t]) for t in th]
    finally:
        dgp.dgp_destroy(ctx)
    assert np.array_equal(b, [v[0][0] for v in one]) and np.array_equal(q, [v[1][0] for v in one])


@pytest.mark.parametrize("prec", ["DGP_FP32", "DGP_FP64"])
@pytest.mark.parametrize("npart", [1, 255, 4097])
def test_sort_into_an_unaligned_cell_start(dgp, torch_dev, prec, npart):
    torch, dev = torch_dev
    n, box = 16, 50.0
    td = torch.float64 if prec == "DGP_FP64" else torch.float32
    g = torch.Generator(device=dev)
    g.manual_seed(npart)
    v = torch.rand((6, npart), generator=g, device=dev, dtype=td) * (box * 0.999)
    ctx = dgp.dgp_init(box, n, 1.0, OM, precision=getattr(dgp, prec))
    try:
        got = []
        for off in (0, 1):
            t = [c.clone() for c in v]
            cells = torch.full((n ** 3 + 1 + off,), -1, dtype=torch.int32, device=dev)[off:]
            dgp.dgp_sort_particles(ctx, dgp.particles(*t), cells)
            got.append((cells.clone(), torch.stack(t)))
    finally:
        dgp.dgp_destroy(ctx)
    assert torch.equal(got[0][0], got[1][0]) and int(got[0][0][-1]) == npart
    for cells, t in got:  # the same particles, the six values of each kept together
        a, b = t.cpu().numpy(), v.cpu().numpy()
        assert np.array_equal(a[:, np.lexsort(a)], b[:, np.lexsort(b)])


@pytest.mark.parametrize("n", [16, 48])
def test_zeldovich_on_unaligned_arrays(dgp, torch_dev, n):
    torch, dev = torch_dev
    d = _field(torch, dev, n, 7) * 0.3
    ctx = dgp.dgp_init(80.0, n, 1.0, OM, precision=dgp.DGP_FP32)
    try:
        runs = []
        for off in (0, 1):
            t = [torch.zeros(n ** 3 + off, device=dev)[off:] for _ in range(6)]
            dgp.dgp_zeldovich(ctx, d, 0.4, dgp.particles(*t))
            back = torch.empty((n, n, n), device=dev)
            dgp.dgp_zeldovich_adjoint(ctx, dgp.particles(*t), 0.4, back)
            torch.cuda.synchronize()
            runs.append([v.clone() for v in t] + [back])
    finally:
        dgp.dgp_destroy(ctx)
    assert all(torch.equal(a, b) for a, b in zip(*runs))


@pytest.mark.parametrize("n", [16, 32, 48, 64, 96, 128])
def test_fp32_adjoint_follows_fp64(dgp, torch_dev, n):
    torch, dev = torch_dev
    box, a = 100.0 * n / 64, 0.6
    f = _field(torch, dev, n, 11).double() * 0.25
    delta = torch.exp(f)
    delta = (delta / delta.mean() - 1.0).float().double()
    cot = _field(torch, dev, n, 12).double()
    out = {}
    for prec, tol, td in (("DGP_FP64", 1e-12, torch.float64), ("DGP_FP32", 1e-6, torch.float32)):
        ctx = dgp.dgp_init(box, n, 1.0, OM, precision=getattr(dgp, prec), tol=tol, max_iter=200)
        try:
            st, _ = dgp.dgp_solve_phi(ctx, a, delta.to(td), None, tol)
            assert st == dgp.DGP_OK
            bar = torch.empty((n, n, n), dtype=td, device=dev)
            st, info = dgp.dgp_solve_adjoint(ctx, cot.to(td), bar, tol)
            assert st == dgp.DGP_OK and info["iters"] >= 1
            torch.cuda.synchronize()
            out[prec] = bar.double().cpu().numpy()
        finally:
            dgp.dgp_destroy(ctx)
    assert rel_l2(out["DGP_FP32"], out["DGP_FP64"]) < 1e-4


@pytest.mark.parametrize("prec", ["DGP_FP32", "DGP_MIXED", "DGP_MIXED_EFT", "DGP_MIXED_F32R"])
@pytest.mark.parametrize("n", [16, 32, 48, 64, 96])
def test_relaxation_row_splits_follow_fp64(dgp, torch_dev, n, prec):
    """Every row split of the relaxation pass in every arithmetic: forces of FP32-data solves to 1e-6
    against an FP64 solve to 1e-12; the bound of the FP32-data paths, 1e-5."""
    torch, dev = torch_dev
    delta = torch.exp(_field(torch, dev, n, 21).double() * 0.25)
    delta = (delta / delta.mean() - 1.0).float().double()
    out = []
    for p, tol, td in (("DGP_FP64", 1e-12, torch.float64), (prec, 1e-6, torch.float32)):
        ctx = dgp.dgp_init(100.0 * n / 64, n, 1.0, OM, precision=getattr(dgp, p), tol=tol, max_iter=200)
        try:
            g = [torch.empty((n, n, n), dtype=td, device=dev) for _ in range(4)]  # phi and the forces
            st, _ = dgp.dgp_solve_forces(ctx, 0.6, delta.to(td), *g, tol)
            assert st == dgp.DGP_OK
            torch.cuda.synchronize()
            out.append(torch.stack(g[1:]).double().cpu().numpy())
        finally:
            dgp.dgp_destroy(ctx)
    assert rel_l2(out[1], out[0]) < 1e-5
