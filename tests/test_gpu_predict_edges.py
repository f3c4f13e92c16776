"""Predictions at many new inputs: the Matern kernel against dense linear algebra, and both sides of the size where a
column no longer fits one SM's shared memory, against the two-column path.

Bounds as in test_gpu_predict_many.py: 8 kappa u between the two paths, n eps / lambda_min more against the dense solution;
at the large sizes kappa <= (n + nugget) / nugget (unit kernel), and |c . alpha| <= |C^-1 f| sqrt(n) <= n max|f| / nugget."""
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


def _predict(n, B, m, kind, rho, nug, eps, tau2, few):
    """(x, f, xs, mu, var, mu and var of the first `few` inputs, four at a time)"""
    x, _ = uniform_sine(n, 7)
    xs = np.random.default_rng(8).uniform(-0.2, 1.2, m)
    f = np.sin(5 * x)
    ctx = fifa.Context(leaf_size=B, aca_tol=eps, rank_cap=32, arena_bytes=2 << 30)
    xd, fd, xsd = dev(x, torch), dev(f, torch), dev(xs, torch)
    C = fifa.fifa_assemble(ctx.h, xd, n, fifa.fifa_hyper(kind, 1.0, rho, 1.0, nug))
    W = fifa.fifa_factor(ctx.h, C)
    _, code = fifa.fifa_logdet(ctx.h, W)
    assert code == fifa.FIFA_OK
    mu, var = (torch.full((m,), np.nan, dtype=torch.float64, device="cuda") for _ in range(2))
    fifa.fifa_predict(ctx.h, C, W, xd, fd, xsd, m, tau2, mu, var)
    mu2, var2 = torch.empty_like(mu[:few]), torch.empty_like(var[:few])
    for j in range(0, few, 4):
        k = min(4, few - j)
        fifa.fifa_predict(ctx.h, C, W, xd, fd, xsd[j:j + k], k, tau2, mu2[j:j + k], var2[j:j + k])
    torch.cuda.synchronize()
    ctx.close()
    return x, f, xs, host(mu), host(var), host(mu2), host(var2)


def test_matern():
    n, m, rho, nug, eps, tau2 = 1501, 70, 0.1, 1e-3, 1e-12, 1.7
    x, f, xs, mu, var, mu2, var2 = _predict(n, 33, m, 1, rho, nug, eps, tau2, m)

    def k(a, b):
        t = np.sqrt(5.0) * np.abs(a[:, None] - b[None]) / rho
        return (1 + t + t * t / 3) * np.exp(-t)

    K, c = k(x, x) + nug * np.eye(n), k(x, xs)
    w = np.linalg.eigvalsh(K)
    kappa = w[-1] / w[0]
    sol = np.linalg.solve(K, np.column_stack([f, c]))
    tol = 8 * kappa * U
    full = tol + n * eps / w[0]
    amp = np.linalg.norm(sol[:, 0]) * np.sqrt(n)
    assert np.max(np.abs(var - tau2 * (1 - (c * sol[:, 1:]).sum(0)))) <= tau2 * full
    assert np.max(np.abs(mu - c.T @ sol[:, 0])) <= full * amp
    assert np.max(np.abs(var - var2)) <= tau2 * tol
    assert np.max(np.abs(mu - mu2)) <= tol * amp


@pytest.mark.parametrize("beyond", [0, 1])
def test_around_the_largest_column(beyond):
    # a column, its rows' leaves and the sweep's buffers: 10 bytes a row, 10240, and 1024 left to the kernel's own
    optin = torch.cuda.get_device_properties(0).shared_memory_per_block_optin
    n = (optin - 1024 - 10240) // 10 + beyond
    m, nug, tau2 = n // 256 + 5, 1e-2, 1.3
    x, f, xs, mu, var, mu2, var2 = _predict(n, 64, m, 1, 0.05, nug, 1e-10, tau2, 12)
    tol = 8 * (n + nug) / nug * U
    assert np.all(np.isfinite(mu)) and np.all(np.isfinite(var)) and np.all(var <= tau2 * (1 + tol))
    assert np.max(np.abs(var[:12] - var2)) <= tau2 * tol
    assert np.max(np.abs(mu[:12] - mu2)) <= tol * n / nug
