"""Contexts with independent CTAs run the sweeps and products of small problems in one thread-block cluster, whose CTAs
are scheduled together: nothing there polls, so opts.wait_polls cannot make such a context time out.  With a limit of one
poll every result is the default context's, bit for bit, and every status is FIFA_OK."""
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


# clusters of two, four and eight CTAs; the largest such problem
@pytest.mark.parametrize("n,B", [(70, 64), (250, 64), (1025, 32), (8192, 64)])
def test_one_poll_is_enough(n, B):
    x, _ = uniform_sine(n, 3)
    xd = dev(x, torch)
    v = dev(np.random.default_rng(5).standard_normal((2, n)), torch)
    seen = []
    for polls in (0, 1):
        ctx = fifa.Context(leaf_size=B, aca_tol=1e-10, rank_cap=32, prec=fifa.FIFA_MIXED, refine_tol=1e-10, refine_max=6,
                           arena_bytes=1 << 29, independent_ctas=1, wait_polls=polls)
        C = fifa.fifa_assemble(ctx.h, xd, n, fifa.fifa_hyper(0, 1.0, 0.1, 1.0, 1e-6))
        A = fifa.fifa_shift_scale(ctx.h, C, 1.0)
        F = fifa.fifa_factor(ctx.h, A)
        out = []
        for k in (1, 2):
            o = torch.full((7, k, n), np.nan, dtype=torch.float64, device="cuda")
            fifa.fifa_matvec(ctx.h, A, v, o[0], k)
            for i, (trans, inv) in enumerate(((0, 0), (0, 1), (1, 0), (1, 1))):
                fifa.fifa_apply_W(ctx.h, F, trans, inv, v, o[1 + i], k)
            fifa.fifa_apply_precond(ctx.h, F, v, o[5], k)
            fifa.fifa_solve(ctx.h, F, v, o[6], k)
            out.append(host(o))
        _, code = fifa.fifa_logdet(ctx.h, F, allow=(fifa.FIFA_ERR_TIMEOUT,))
        code_h = fifa.fifa_hmat_export(ctx.h, A, allow=(fifa.FIFA_ERR_TIMEOUT,), bases=False, leaves=False)["status"]
        assert (code, code_h) == (fifa.FIFA_OK, fifa.FIFA_OK), polls
        seen.append(out)
        ctx.close()
    for a, b in zip(*seen):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)
