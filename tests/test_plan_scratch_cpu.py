"""Scratch of a plan (no GPU): an arena that held a problem goes on holding it.  The bounds are what the same plans took
when fused sweeps had two slots of partials in all and clusters had none; regions belong to the CTAs that exchange through
them, so neither the levels without groups nor a context whose launches are one cluster take more."""
import os
import shutil

import pytest

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="nvcc not available to build the library")

BYTES = {  # (independent_ctas, n): scratch bytes at leaf 32, rank cap 32, mixed precision
    (0, 1024): 840192, (0, 4096): 3716352, (0, 8192): 7813888, (0, 8193): 15352320, (0, 20000): 32728832,
    (0, 131072): 97599232, (0, 1 << 20): 727965440,
    (1, 1024): 545792, (1, 4096): 2274816, (1, 8192): 4667648, (1, 8193): 8536064, (1, 20000): 18045696,
    (1, 131072): 82875136, (1, 1 << 20): 713241344,
}


@pytest.mark.parametrize("indep,n", sorted(BYTES))
def test_scratch_is_no_larger(indep, n):
    from paper_2006_06537_gb300 import build

    build.build()
    from paper_2006_06537_gb300 import fifa

    o = fifa.fifa_opts(32, 1e-10, 32, fifa.FIFA_MIXED, 1e-12, 3, indep)
    assert fifa.fifa_plan_describe(o, n, 608, (608, 456, 152))["info"].scratch_bytes <= BYTES[indep, n]
