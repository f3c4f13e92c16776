"""Leaf factors whose ancestor columns take more than one pass (64 columns for leaves of up to 64 rows, 32 above), in CTAs
that have a leaf alone and in CTAs that share one: the checks and bounds of test_gpu_leaf_factor.py at sizes where, by the
exported ranks, the later passes run."""
import numpy as np
import pytest

from paper_2006_06537_gb300.inputs import uniform_sine
from tests.gpu_util import build_lib, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

build_lib()
from paper_2006_06537_gb300 import fifa  # noqa: E402
from tests import test_gpu_leaf_factor as leaf_factor  # noqa: E402


@pytest.mark.parametrize("n,B,rho,eps,share,passes", [
    (10001, 50, 0.02, 1e-14, 1, 2),   # leaves of 39 and 40 rows, a CTA each
    (5001, 64, 0.02, 1e-12, 2, 1),    # of 39 and 40, two CTAs each
    (20400, 128, 0.02, 1e-10, 1, 3),  # of 79 and 80, a CTA each
    (10001, 128, 0.02, 1e-12, 2, 2),  # of 78 and 79, two CTAs each
])
def test_columns_beyond_a_pass(n, B, rho, eps, share, passes):
    x, _ = uniform_sine(n, 4)
    ctx = fifa.Context(leaf_size=B, aca_tol=eps, rank_cap=32, arena_bytes=1 << 30)
    C = fifa.fifa_assemble(ctx.h, dev(x, torch), n, fifa.fifa_hyper(0, 1.0, rho, 1.0, 1e-5))
    ex = fifa.fifa_hmat_export(ctx.h, C, bases=False, leaves=False)
    L, rk = ex["L"], ex["ranks"]
    cols = np.array([sum(int(rk[(1 << lvl) - 1 + (i >> (L - lvl))]) for lvl in range(L)) for i in range(1 << L)])
    a_pass = 64 if B <= 64 else 32
    assert share == (1 if 2 * len(cols) > 304 else 2)  # a second CTA per leaf while all of them are at most two to an SM
    assert np.all(cols // share > (passes - 1) * a_pass)
    ctx.close()
    leaf_factor.test_leaf_factors((n, B, rho, eps))
