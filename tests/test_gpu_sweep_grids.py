"""The fused sweeps and products over their grids (one CTA, a cluster of independent contexts, grids of several row counts
per CTA, the per-level kernels of independent contexts above 8192 rows) through the identities of the factor, and between
the two kinds of context.

Bound: with A = C~ + I and kappa = n + 2 >= cond(A) (unit kernel), every application is off by at most a modest multiple of
kappa u per tree level: 8 (L + 1) kappa u in norm, L + 1 <= 12 for these sizes."""
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
# rows per CTA: 30; 65; 128 and 160..161 (staging sizes); 257; 512..513; 1024 (largest cluster); the first size beyond it; both sides of 2^15
CASES = [(30, 64), (129, 64), (1024, 32), (1285, 40), (2057, 33), (4099, 100), (8192, 32), (8193, 64), (32767, 32), (32769, 128)]


def _near(a, b, tol, what):
    a, b = host(a), host(b)
    err = np.linalg.norm(a - b, axis=-1) / np.linalg.norm(b, axis=-1)
    assert np.all(err <= tol), (what, err, tol)


@pytest.mark.parametrize("n,B", CASES)
def test_sweeps_and_products(n, B):
    x, _ = uniform_sine(n, 3)
    xd = dev(x, torch)
    v = dev(np.random.default_rng(4).standard_normal((2, n)), torch)
    L = max(0, int(np.ceil(np.log2(n / B))))
    tol = 8 * (L + 1) * (n + 2) * U
    seen = []
    for indep in (0, 1):
        ctx = fifa.Context(leaf_size=B, aca_tol=1e-10, rank_cap=16, prec=fifa.FIFA_MIXED, refine_tol=1e-10, refine_max=6,
                           arena_bytes=1 << 30, independent_ctas=indep)
        C = fifa.fifa_assemble(ctx.h, xd, n, fifa.fifa_hyper(0, 1.0, 0.1, 1.0, 1e-6))
        A = fifa.fifa_shift_scale(ctx.h, C, 1.0)
        F = fifa.fifa_factor(ctx.h, A)
        new = lambda: torch.full((2, n), np.nan, dtype=torch.float64, device="cuda")  # noqa: E731
        one = lambda: torch.full((1, n), np.nan, dtype=torch.float64, device="cuda")  # noqa: E731
        out = {}
        for name, op in (("A", None), ("W", (0, 0)), ("Wi", (0, 1)), ("Wt", (1, 0)), ("Wti", (1, 1))):
            two, single = new(), one()
            for src, dst, k in ((v, two, 2), (v[1:].contiguous(), single, 1)):
                if op is None:
                    fifa.fifa_matvec(ctx.h, A, src, dst, k)
                else:
                    fifa.fifa_apply_W(ctx.h, F, *op, src, dst, k)
            _near(single, two[1:], tol, name + " one vector")
            out[name] = two
        back, t = new(), new()
        fifa.fifa_apply_W(ctx.h, F, 0, 0, out["Wt"], back, 2)
        _near(back, out["A"], tol, "W W^T v = A v")
        fifa.fifa_apply_W(ctx.h, F, 0, 1, out["W"], t, 2)
        _near(t, v, tol, "W^-1 W v = v")
        fifa.fifa_apply_W(ctx.h, F, 1, 1, out["Wt"], t, 2)
        _near(t, v, tol, "W^-T W^T v = v")
        z = new()
        fifa.fifa_solve(ctx.h, F, v, z, 2)  # conjugate gradients: products and the FP32 copy's sweeps
        fifa.fifa_matvec(ctx.h, A, z, t, 2)
        _near(t, v, 2e-10 + tol, "A z = v")
        torch.cuda.synchronize()
        seen.append(out)
    for name in seen[0]:
        _near(seen[1][name], seen[0][name], tol, name + " between the contexts")
