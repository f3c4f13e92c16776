"""The ACA kernels' launch forms (clusters of several sizes, one CTA, one warp, groups; U and V kept in shared memory or
not) against the oracle, bit for bit: ranks, pivots and bases do not depend on how a block is split."""
import numpy as np
import pytest

from paper_2006_06537_gb300.inputs import clustered, uniform_sine
from tests.gpu_util import build_lib, dev, oracle_bases, oracle_hmat, used_mask

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

build_lib()
from paper_2006_06537_gb300 import fifa  # noqa: E402

CASES = [
    # n, B, kind, rho, eps, cap, data
    (33, 32, 0, 0.2, 1e-12, 32, "sine"),       # one block of 16 x 17
    (257, 16, 1, 0.1, 1e-10, 32, "sine"),      # warp-sized blocks by clusters, one of 128 x 129 by a solo launch
    (1500, 40, 0, 0.3, 1e-14, 6, "sine"),      # the rank cap stops every large block
    (3000, 2, 0, 0.05, 1e-10, 16, "sine"),     # more small blocks than the GPU holds CTAs: one warp each
    (3500, 32, 0, 0.05, 1e-10, 32, "sine"),    # large and small blocks in one launch, clusters of four
    (6001, 100, 1, 0.02, 1e-10, 32, "cluster"),  # groups at the top, clusters below
    (9000, 64, 0, 0.002, 1e-12, 40, "sine"),   # many steps: U and V beyond the kept ones
]


@pytest.mark.parametrize("indep", [0, 1])
@pytest.mark.parametrize("case", CASES)
def test_bases_bit_exact(case, indep):
    n, B, kind, rho, eps, cap, data = case
    x, _ = clustered(n, 2) if data == "cluster" else uniform_sine(n, 1)
    ctx = fifa.Context(leaf_size=B, aca_tol=eps, rank_cap=cap, arena_bytes=1 << 30, independent_ctas=indep)
    H = fifa.fifa_assemble(ctx.h, dev(x, torch), n, fifa.fifa_hyper(kind, 1.0, rho, 1.0, 1e-6))
    ex = fifa.fifa_hmat_export(ctx.h, H)
    Ho = oracle_hmat(x, B, kind, rho, 1e-6, eps, cap)
    for lvl in range(Ho.tree.L):
        for i in range(1 << lvl):
            nid = (1 << lvl) - 1 + i
            r = Ho.rank(lvl, i)
            assert ex["ranks"][nid] == r, (lvl, i)
            assert list(ex["row_piv"][nid, :r]) == Ho.row_piv[(lvl, i)]
            assert list(ex["col_piv"][nid, :r]) == Ho.col_piv[(lvl, i)]
    assert (ex["status"] == fifa.FIFA_ERR_RANK_CAP) == any(Ho.hit_cap.values())
    mask = used_mask(ex["ranks"], Ho.tree, cap)
    assert np.array_equal(ex["bases"][mask].view(np.uint64), oracle_bases(Ho, n, cap)[mask].view(np.uint64))
