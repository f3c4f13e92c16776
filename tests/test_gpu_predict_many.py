"""Predictions at many new inputs (one CTA per input) against dense linear algebra, and against the two-column path on the
same inputs (few of them at a time).

Bounds: with C = K + nugget I of condition number kappa, |mu - mu_ref| and |var - var_ref| / tau2 are at most 8 kappa u plus
what C~ differs from C by (n eps kappa / ||C||, eps the cross approximation's tolerance); the two paths share C~ and its
factor, so between them 8 kappa u is all."""
import numpy as np
import pytest

from paper_2006_06537_gb300.inputs import uniform_sine
from tests.gpu_util import build_lib, dev, host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

build_lib()
from paper_2006_06537_gb300 import fifa  # noqa: E402

U = 2.0 ** -53


@pytest.mark.parametrize("n,B,m,mean", [(40, 64, 9, True), (1000, 33, 200, True), (2500, 128, 17, False), (3001, 32, 160, True)])
def test_many_inputs(n, B, m, mean):
    rho, nug, eps, tau2 = 0.1, 1e-3, 1e-12, 1.7
    x, y = uniform_sine(n, 7)
    g = np.random.default_rng(8)
    xs = g.uniform(-0.2, 1.2, m)
    f = np.sin(5 * x)
    ctx = fifa.Context(leaf_size=B, aca_tol=eps, rank_cap=32, arena_bytes=1 << 30)
    xd, fd, xsd = dev(x, torch), dev(f, torch), dev(xs, torch)
    C = fifa.fifa_assemble(ctx.h, xd, n, fifa.fifa_hyper(0, 1.0, rho, 1.0, nug))
    W = fifa.fifa_factor(ctx.h, C)
    mu, var = (torch.full((m,), np.nan, dtype=torch.float64, device="cuda") for _ in range(2))
    fifa.fifa_predict(ctx.h, C, W, xd, fd, xsd, m, tau2, mu if mean else None, var)
    mu2, var2 = torch.empty_like(mu), torch.empty_like(var)
    for j in range(0, m, 4):  # few at a time: two columns per sweep
        k = min(4, m - j)
        fifa.fifa_predict(ctx.h, C, W, xd, fd, xsd[j:j + k], k, tau2, mu2[j:j + k], var2[j:j + k])
    torch.cuda.synchronize()
    K = np.exp(-0.5 * ((x[:, None] - x[None]) / rho) ** 2) + nug * np.eye(n)
    c = np.exp(-0.5 * ((x[:, None] - xs[None]) / rho) ** 2)
    w = np.linalg.eigvalsh(K)
    kappa = w[-1] / w[0]
    sol = np.linalg.solve(K, np.column_stack([f, c]))
    tol = 8 * kappa * U
    full = tol + n * eps / w[0]
    amp = np.linalg.norm(sol[:, 0]) * np.sqrt(n)  # |c . alpha| is at most this
    v_ref = tau2 * (1 - (c * sol[:, 1:]).sum(0))
    assert np.max(np.abs(host(var) - v_ref)) <= tau2 * full
    assert np.max(np.abs(host(var) - host(var2))) <= tau2 * tol
    if mean:
        assert np.max(np.abs(host(mu) - c.T @ sol[:, 0])) <= full * amp
        assert np.max(np.abs(host(mu) - host(mu2))) <= tol * amp
