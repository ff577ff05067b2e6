"""The Hessian passes of the field solve (x pass with three outputs, y pass forming the six second
derivatives and N) against the oracle on a field with content in every mode, the Nyquist planes
included, where the off-diagonal multipliers are |k_i k_j| / k^2: every mesh the oracle can do in
reasonable time (all splits N = N1 N2: equal, unequal, with 3 and 6), FP64 and FP32 data, with
and without the non-local terms.

Tolerances: FP64, both sides converged to <|R|>/eps < 1e-11, so D agrees to a small multiple of
that (1e-9); FP32, the solve's tolerance 1e-6 and FP32 rounding give a few 1e-6 (1e-5)."""
import numpy as np
import pytest

from test_gpu_parity import OM, rel_l2, to_dev  # noqa: F401
from test_gpu_parity import dgp, torch_dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol,bound", [("DGP_FP64", 1e-11, 1e-9), ("DGP_MIXED_F32R", 1e-6, 1e-5)])
@pytest.mark.parametrize("n,local", [(16, False), (32, False), (48, False), (64, True), (96, False), (128, False)])
def test_solve_with_nyquist_content_matches_oracle(dgp, torch_dev, n, local, prec, tol, bound):
    from oracle import field as ofield
    torch, dev = torch_dev
    if n == 128 and prec == "DGP_FP64":
        pytest.skip("the FP32 case covers this mesh")
    rng = np.random.default_rng(n)
    delta = rng.normal(0.0, 0.25, (n, n, n))
    # pure Nyquist waves along single axes and pairs of axes
    s = 1.0 - 2.0 * (np.arange(n) % 2)
    c = np.cos(2 * np.pi * np.arange(n) / n)
    delta += 0.2 * (s[:, None, None] * c[None, :, None] * np.roll(c, 3)[None, None, :] +
                    c[:, None, None] * s[None, :, None] * c[None, None, :] +
                    np.roll(c, 1)[:, None, None] * c[None, :, None] * s[None, None, :] +
                    s[:, None, None] * s[None, :, None] * c[None, None, :])
    delta = np.exp(delta)  # a density: delta >= -1, where the equation has a solution
    delta = (delta / delta.mean() - 1.0).astype(np.float32).astype(np.float64)
    box, a = 1.5 * n, 0.5
    phi_o, g_o, D_o, oinfo = ofield.solve_phi(delta, a, box, OM, 1.0, tol=min(tol, 1e-9) * 0.1, local_only=local)
    assert oinfo["converged"]
    td = torch.float64 if prec == "DGP_FP64" else torch.float32
    ctx = dgp.dgp_init(box, n, 1.0, OM, precision=getattr(dgp, prec), tol=tol, max_iter=200, local_only=local)
    try:
        out = [torch.empty((n, n, n), dtype=td, device=dev) for _ in range(5)]
        st, info = dgp.dgp_solve_forces(ctx, a, to_dev(torch_dev, delta, td), *out[:4], tol)
        assert st == dgp.DGP_OK
        dgp.dgp_get_solution(ctx, out[4])
        torch.cuda.synchronize()
        got = [v.double().cpu().numpy() for v in out]
    finally:
        dgp.dgp_destroy(ctx)
    assert rel_l2(got[4], D_o) < bound
    assert rel_l2(got[0], phi_o) < bound
    for i in range(3):
        assert rel_l2(got[1 + i], g_o[i]) < bound
