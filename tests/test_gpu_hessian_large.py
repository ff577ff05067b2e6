"""The Hessian and relaxation passes of the largest meshes on content up to and on the Nyquist planes: the eight-column
x tile, the y pass that reads its rows again, the two TMA boxes along kz (the second one clipped) and the four-row
CTAs exist at 512^3 only, and the other 512^3 test has its content at the lowest modes.

A 32^3 density with content in every mode is repeated n / 32 times along each axis.  Its modes lie on the multiples of
n / 32, its Nyquist index on n / 2, so the n^3 solve is the repeated 32^3 solve, which the oracle makes.

Tolerances: those of the same comparison on the smaller meshes, FP64 (both sides to 1e-11) 1e-9, FP32 data (to 1e-6) 1e-5."""
import numpy as np
import pytest

from test_gpu_parity import OM
from test_gpu_parity import dgp, torch_dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu
M = 32


def _small():
    rng = np.random.default_rng(7)
    delta = rng.normal(0.0, 0.25, (M, M, M))
    s = 1.0 - 2.0 * (np.arange(M) % 2)
    c = np.cos(2 * np.pi * np.arange(M) / M)
    delta += 0.2 * (s[:, None, None] * c[None, :, None] * np.roll(c, 3)[None, None, :] +
                    c[:, None, None] * s[None, :, None] * c[None, None, :] +
                    np.roll(c, 1)[:, None, None] * c[None, :, None] * s[None, None, :] +
                    s[:, None, None] * s[None, :, None] * c[None, None, :])
    delta = np.exp(delta)
    return (delta / delta.mean() - 1.0).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,prec,tol,bound", [(256, "DGP_MIXED_F32R", 1e-6, 1e-5), (256, "DGP_FP64", 1e-11, 1e-9),
                                              (512, "DGP_MIXED_F32R", 1e-6, 1e-5), (512, "DGP_MIXED_EFT", 1e-6, 1e-5),
                                              (512, "DGP_FP64", 1e-11, 1e-9)])
def test_repeated_nyquist_content_matches_the_small_mesh(dgp, torch_dev, n, prec, tol, bound):
    from oracle import field as ofield
    torch, dev = torch_dev
    delta, box, a = _small(), 1.5 * M, 0.5
    phi_o, g_o, D_o, oinfo = ofield.solve_phi(delta, a, box, OM, 1.0, tol=min(tol, 1e-9) * 0.1)
    assert oinfo["converged"]
    td = torch.float64 if prec == "DGP_FP64" else torch.float32
    rep = n // M
    ctx = dgp.dgp_init(box * rep, n, 1.0, OM, precision=getattr(dgp, prec), tol=tol, max_iter=200)
    try:
        d = torch.as_tensor(delta).to(dev, td).repeat(rep, rep, rep).contiguous()
        out = [torch.empty((n, n, n), dtype=td, device=dev) for _ in range(5)]
        st, info = dgp.dgp_solve_forces(ctx, a, d, *out[:4], tol)
        assert st == dgp.DGP_OK
        dgp.dgp_get_solution(ctx, out[4])
        torch.cuda.synchronize()
        for got, want in zip(out, (phi_o, *g_o, D_o)):
            w = torch.as_tensor(np.ascontiguousarray(want)).to(dev)
            err = got.double().reshape(rep, M, rep, M, rep, M) - w[None, :, None, :, None, :]
            assert float(err.norm()) / (float(w.norm()) * rep ** 1.5) < bound
            del err
    finally:
        dgp.dgp_destroy(ctx)
