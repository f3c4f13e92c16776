"""The additive model at sizes where the blocks' ACA and level kernels work in groups of CTAs that wait on each other, and
all blocks' groups together exceed what the GPU holds at once, so that one launch takes them with smaller groups.

* The bases of an accepted proposal, which that launch assembled, equal the same block's assembled by itself, bit for bit
  (they are looked up in the model's arena by their first values).
* Sweeps agree with a context of independent CTAs, which takes the blocks one at a time: with kappa <= (n + nugget) /
  nugget (unit kernel), 8 kappa u for what passes through one factor, ten times that for the trace, a hundred times for
  the components (the tolerances of test_gpu_additive.py)."""
import math

import numpy as np
import pytest

from paper_2006_06537_gb300.inputs import additive4
from tests.gpu_util import build_lib, dev, host, rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

build_lib()
from paper_2006_06537_gb300 import fifa  # noqa: E402

B, EPS, CAP, RHO0, NUG, SWEEPS = 32, 1e-10, 32, 0.1, 1e-2, 3


def _run(X, y, indep, share):
    n, d = X.shape
    o = fifa.fifa_opts(B, EPS, CAP, fifa.FIFA_FP64, 1e-12, 3, indep, 0, share)
    ctx = fifa.Context(leaf_size=B, aca_tol=EPS, rank_cap=CAP, arena_bytes=int(1.2 * d * fifa.fifa_chain_bytes(o, n)) + (64 << 20),
                       stream=torch.cuda.Stream(), independent_ctas=indep, coresident_share=share)
    vy = float(np.var(y))
    pr = fifa.fifa_prior(1.0, 1.0, 1.0, 1.0, math.log(RHO0), 1.0, 0.01)  # small steps: most proposals are accepted
    Xd, yd = dev(X.T, torch), dev(y, torch)
    torch.cuda.synchronize()
    m = fifa.fifa_additive_create(ctx.h, Xd, yd, n, d, fifa.fifa_hyper(0, vy / d, RHO0, 0.5 * vy, NUG), pr, 3)
    tr = np.zeros((SWEEPS, fifa.fifa_additive_trace_fields(d)))
    fifa.fifa_additive_sweep(ctx.h, m, SWEEPS, tr)
    F = torch.empty((d, n), dtype=torch.float64, device="cuda")
    _, hyp = fifa.fifa_additive_get(ctx.h, m, d, F)
    torch.cuda.synchronize()
    return ctx, m, tr, host(F), hyp


@pytest.mark.parametrize("n,d,share", [(20001, 2, 8), (20001, 3, 8), (65539, 4, 1)])
def test_groups_of_several_blocks(n, d, share):
    X, y = additive4(n, seed=5)
    X = np.ascontiguousarray(X[:, :d])
    # the cross-approximation kernel's CTAs the GPU holds at once: four to an SM
    cores = 4 * torch.cuda.get_device_properties(0).multi_processor_count // share
    o = fifa.fifa_opts(B, EPS, CAP, fifa.FIFA_FP64, 1e-12, 3, 0, 0, share)
    plan = fifa.fifa_plan_describe(o, n, cores, (cores, cores, cores))
    assert 0 < plan["info"].aca_grouped_ctas <= cores < d * plan["info"].aca_grouped_ctas
    assert np.any(plan["groups"][:, : max(1, int(math.log2(n / 2048)))] > d)  # levels beyond clusters: groups for every block

    ctx, model, tr, F, hyp = _run(X, y, 0, share)
    assert np.all(tr[:, 3] == 0)
    accepted = [k for k in range(d) if hyp[k].rho != RHO0]
    assert accepted
    words = ctx.arena[: ctx.arena.numel() // 8 * 8].view(torch.int64)
    for k in accepted[:2]:
        one = fifa.Context(leaf_size=B, aca_tol=EPS, rank_cap=CAP, arena_bytes=1 << 30, independent_ctas=1)
        xk = dev(np.sort(X[:, k]), torch)
        H = fifa.fifa_assemble(one.h, xk, n, fifa.fifa_hyper(0, 1.0, hyp[k].rho, 1.0, NUG))
        ex = fifa.fifa_hmat_export(one.h, H, leaves=False)
        one.close()
        L, rk, bits = ex["L"], ex["ranks"], ex["bases"].view(np.int64)
        head = bits[0, 0, :64]
        places = [int(p) for p in torch.nonzero(words == int(head[0])).flatten().cpu()
                  if np.array_equal(host(words[int(p):int(p) + 64]), head)]
        assert places, k
        same = False
        for p in places:
            got = host(words[p:p + bits.size]).reshape(bits.shape)
            ok = True
            for lvl in range(L):
                for i in range(1 << lvl):
                    off = (1 << lvl) - 1 + lvl + i
                    s, e, r = plan["bounds"][off], plan["bounds"][off + 1], rk[(1 << lvl) - 1 + i]
                    ok = ok and np.array_equal(got[lvl, :r, s:e], bits[lvl, :r, s:e])
            same = same or ok
        assert same, k
    fifa.fifa_destroy_additive(ctx.h, model)
    ctx.close()

    ctx, model, tr1, F1, hyp1 = _run(X, y, 1, 0)
    tol = max(1e-10, 8 * (n + NUG) / NUG * 2.0 ** -53)
    assert np.array_equal(tr1[:, 5 + 2 * d:], tr[:, 5 + 2 * d:])
    assert np.allclose(tr1[:, 5 + d:5 + 2 * d], tr[:, 5 + d:5 + 2 * d], rtol=1e-12, atol=0)
    for c in [1, 2] + list(range(5, 5 + d)):
        assert np.all(np.abs(tr1[:, c] - tr[:, c]) <= 10 * tol * np.abs(tr[:, c])), c
    assert rel(F, F1) <= 100 * tol
    fifa.fifa_destroy_additive(ctx.h, model)
    ctx.close()
