"""The leaf factor's kernels (column by column up to 32 rows, blocks of eight columns above; columns shared by one, two or
four CTAs) at ragged leaf sizes, with more ancestor columns than one pass takes.

A = W W^T with W built from the leaf factors and L^-1 applied to the ancestor bases, so the check is W W^T x = A x as a
normwise backward error (a Cholesky factor and substitutions: at most a few times their inner dimension in u; 64 L B u in
all) and W^-1 W x = x within 8 kappa(A) u; the leaf factors themselves against numpy's: || L_i L_i^T - D_i || <= 8 B u || D_i ||."""
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

CASES = [
    # n, B, rho, eps: leaves of
    (300, 33, 0.1, 1e-12),     # 18 and 19 rows
    (65, 33, 0.1, 1e-12),      # 32 and 33
    (1300, 41, 0.05, 1e-12),   # 40 and 41, many columns
    (2000, 64, 0.02, 1e-14),   # 62 and 63, more columns than a pass
    (4000, 127, 0.02, 1e-12),  # 125
    (20400, 128, 0.02, 1e-10),  # 79 and 80 in 256 leaves: one CTA each
    (130, 128, 0.3, 1e-10),    # 65
    (100, 100, 0.3, 1e-10),    # one leaf, no ancestors
]


@pytest.mark.parametrize("case", CASES)
def test_leaf_factors(case):
    n, B, rho, eps = case
    x, _ = uniform_sine(n, 4)
    ctx = fifa.Context(leaf_size=B, aca_tol=eps, rank_cap=32, arena_bytes=1 << 30)
    C = fifa.fifa_assemble(ctx.h, dev(x, torch), n, fifa.fifa_hyper(0, 1.0, rho, 1.0, 1e-5))
    ex = fifa.fifa_hmat_export(ctx.h, C, bases=False)
    L, Bm = ex["L"], ex["Bm"]
    v = np.random.default_rng(6).standard_normal(n)
    vd = dev(v, torch)
    for s in (None, 20.0):
        M = C if s is None else fifa.fifa_shift_scale(ctx.h, C, s)
        F = fifa.fifa_factor(ctx.h, M)
        _, code = fifa.fifa_logdet(ctx.h, F)
        assert code == fifa.FIFA_OK
        fx = fifa.fifa_fact_export(ctx.h, F, fifa.fifa_hmat_dims(C))
        for D0, Lt in zip(ex["leaves"], fx["leaves"]):
            m = int((np.diag(D0) != 0).sum())
            D = D0[:m, :m] if s is None else s * D0[:m, :m] + np.eye(m)
            Li = Lt.T[:m, :m]
            assert np.all(np.triu(Li, 1) == 0)
            assert np.linalg.norm(Li @ Li.T - D) <= 8 * Bm * U * np.linalg.norm(D)
        a, b, t = (torch.empty_like(vd) for _ in range(3))
        fifa.fifa_matvec(ctx.h, M, vd, a, 1)
        fifa.fifa_apply_W(ctx.h, F, 1, 0, vd, t, 1)
        fifa.fifa_apply_W(ctx.h, F, 0, 0, t, b, 1)
        one, row = torch.ones_like(vd), torch.empty_like(vd)
        fifa.fifa_matvec(ctx.h, M, one, row, 1)
        torch.cuda.synchronize()
        norm = float(row.max())  # SE entries are positive: the largest row sum
        assert np.linalg.norm(host(a) - host(b)) <= 64 * max(1, L) * Bm * U * norm * np.linalg.norm(v)
        fifa.fifa_apply_W(ctx.h, F, 0, 0, vd, t, 1)
        fifa.fifa_apply_W(ctx.h, F, 0, 1, t, b, 1)
        torch.cuda.synchronize()
        kappa = norm / (1e-5 if s is None else 1.0)
        assert np.linalg.norm(host(b) - v) <= max(1e-10, 8 * kappa * U) * np.linalg.norm(v)
