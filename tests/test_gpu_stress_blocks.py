"""The stress and the lapse at numbers of zones around the blocks of their kernels (runs of 12 zones; warps of a
ray's zones up to 256) and with few groups, against the oracle with the measures of tests/test_gpu_stress.py."""
import pytest

from paper_1809_05608_gb300 import problems
from tests import small_problems as SP
from tests import test_gpu_stress as stress

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module', autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_1809_05608_gb300 import mgfld
    mgfld.lib()
    stress.M = mgfld


@pytest.mark.parametrize('n_r', [2, 11, 12, 13, 31, 32, 33, 64, 255, 256, 257])
@pytest.mark.parametrize('n_e', [1, 2, 5])
def test_block_edges(n_r, n_e):
    inp = SP.strong(n_ray=3, n_r=n_r, n_e=n_e, kabs=1e3, kscat=1e3, nes=3.0, lapse=True)
    p, m = problems.stress_inputs(inp)
    stress.check(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'], p, m)
