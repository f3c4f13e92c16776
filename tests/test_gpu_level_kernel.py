"""The factorization's level kernels at the sizes where their paths meet: cluster and group nodes, resident and streamed
rows, ranks at the edges of the buckets, ragged sides.

Checks, each against the matrix the factor was made from (exported leaves and bases, written out densely):
* W W^T x = A x as a normwise backward error.  Every step (leaf Cholesky, two-pass CholeskyQR, capacitance, row updates)
  is backward stable with a constant of at most a few times its inner dimension, so the bound is 64 L B u ||A|| ||x||
  (L levels, leaves of B rows), ||A|| by its largest absolute row sum;
* log det A against numpy's slogdet of the same dense matrix: both have absolute error at most about n kappa(A) u.
"""
import numpy as np
import pytest

from paper_2006_06537_gb300.inputs import clustered, uniform_sine
from tests.gpu_util import build_lib, dev, host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

build_lib()
from paper_2006_06537_gb300 import fifa  # noqa: E402

U = 2.0 ** -53

CASES = [
    # n, B, kind, rho, eps, cap, data, (least, largest) rank wanted
    (130, 32, 0, 0.3, 1e-13, 32, "sine", (5, 16)),       # one-cluster nodes, tiny sides
    (500, 32, 0, 0.1, 1e-12, 32, "sine", (5, 16)),
    (2047, 64, 0, 0.1, 1e-12, 32, "sine", (5, 16)),
    (2049, 64, 0, 0.05, 1e-12, 32, "sine", (9, 32)),     # past the cluster's row limit: groups at the top
    (4100, 33, 1, 0.02, 1e-10, 32, "sine", (2, 8)),      # ragged leaves, Matern, ranks of both buckets
    (4100, 64, 0, 0.005, 1e-14, 40, "sine", (17, 40)),   # ranks above 16 next to smaller ones
    (5000, 128, 0, 0.01, 1e-10, 16, "cluster", (4, 16)), # cap 16: exchanges of few columns
    (3000, 32, 0, 0.1, 1e-3, 4, "sine", (1, 4)),         # low ranks, small cap; C~ itself is indefinite
]


def _dense(ex, n):
    A = np.zeros((n, n))
    L, B = ex["L"], ex["Bm"]
    bounds = [np.array([0, n])]
    for _ in range(L):
        b = bounds[-1]
        nxt = [0]
        for i in range(len(b) - 1):
            nxt += [b[i] + (b[i + 1] - b[i]) // 2, b[i + 1]]
        bounds.append(np.array(nxt))
    for i in range(ex["nleaf"]):
        s, e = bounds[L][i], bounds[L][i + 1]
        A[s:e, s:e] = ex["leaves"][i, :e - s, :e - s].T
    for lvl in range(L):
        for i in range(1 << lvl):
            s, e = bounds[lvl][i], bounds[lvl][i + 1]
            h = bounds[lvl + 1][2 * i + 1]
            r = ex["ranks"][(1 << lvl) - 1 + i]
            blk = ex["bases"][lvl, :r, s:h].T @ ex["bases"][lvl, :r, h:e]
            A[s:h, h:e] = blk
            A[h:e, s:h] = blk.T
    return A


@pytest.mark.parametrize("indep", [0, 1])
@pytest.mark.parametrize("case", CASES)
def test_factor_identity_and_logdet(case, indep):
    n, B, kind, rho, eps, cap, data, (rlo, rhi) = case
    x, _ = clustered(n, 2) if data == "cluster" else uniform_sine(n, 0)
    ctx = fifa.Context(leaf_size=B, aca_tol=eps, rank_cap=cap, arena_bytes=1 << 30, independent_ctas=indep)
    xd = dev(x, torch)
    C = fifa.fifa_assemble(ctx.h, xd, n, fifa.fifa_hyper(kind, 1.0, rho, 1.0, 1e-4))
    ex = fifa.fifa_hmat_export(ctx.h, C)
    assert rlo <= ex["ranks"].max() <= rhi, ex["ranks"].max()
    A0 = _dense(ex, n)
    v = np.random.default_rng(3).standard_normal(n)
    vd = dev(v, torch)
    for s in (None, 30.0):
        A, M = (A0, C) if s is None else (s * A0 + np.eye(n), fifa.fifa_shift_scale(ctx.h, C, s))
        F = fifa.fifa_factor(ctx.h, M)
        low = np.linalg.eigvalsh(A)[0]
        ld, code = fifa.fifa_logdet(ctx.h, F, allow=(fifa.FIFA_ERR_NOT_SPD,))
        if low < 0:  # the compression made it indefinite: reported, not factored
            assert code == fifa.FIFA_ERR_NOT_SPD, (s, low)
            continue
        assert code == fifa.FIFA_OK, (s, low)
        t = torch.empty_like(vd)
        fifa.fifa_apply_W(ctx.h, F, 1, 0, vd, t, 1)
        fifa.fifa_apply_W(ctx.h, F, 0, 0, t, t, 1)
        torch.cuda.synchronize()
        norm = np.abs(A).sum(1).max()
        err = np.linalg.norm(host(t) - A @ v) / (norm * np.linalg.norm(v))
        assert err <= 64 * max(1, ex["L"]) * B * U, (s, err)
        sign, ref = np.linalg.slogdet(A)
        kappa = norm / low
        assert sign == 1 and abs(ld - ref) <= n * kappa * U, (s, ld, ref)
