"""The cross approximation of blocks whose rows and columns fill a CTA's slices beyond what it keeps in shared memory
(2048 to a CTA), beside groups and beside nothing else, against the oracle bit for bit: as test_gpu_aca_paths.py, at sizes
on both sides of that line."""
import pytest

from tests import test_gpu_aca_paths as paths
from tests.gpu_util import build_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

build_lib()


@pytest.mark.parametrize("n,B,rho,eps,cap,indep", [
    (16384, 128, 0.01, 1e-10, 32, 1),   # independent contexts: the root in a cluster of eight, 2048 to a CTA
    (16400, 128, 0.01, 1e-10, 32, 1),   # 2050
    (70001, 128, 0.02, 1e-10, 32, 0),   # groups down to 4375 rows, then 480 blocks of 2188 rows and less, a CTA each
    (60001, 128, 0.02, 1e-10, 3, 1),    # the rank cap stops blocks in mid-course, 30001 to a CTA
])
def test_bases_bit_exact(n, B, rho, eps, cap, indep):
    paths.test_bases_bit_exact((n, B, 0, rho, eps, cap, "sine"), indep)
