"""The FP64 substitution of the pair systems on both sides of the lines between the ring-fed kernel and the thread per row
(chosen by the number of systems, two per ray, and the block width 2 n_e).  Both do the same operations on an entry in the
same order, so rays of a large launch end with the bits they have in a launch of their own."""
import numpy as np
import pytest

from paper_1809_05608_gb300 import problems
from tests import small_problems as SP

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module')
def M():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_1809_05608_gb300 import mgfld
    mgfld.lib()
    return mgfld


def _step(M, inp):
    st = M.Stepper(inp, M.MGFLD_FP64, tol=1e-11, max_iter=40)
    psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], inp['T0'])
    assert st.step(psi, ye, T) == M.MGFLD_OK
    return [t.cpu().numpy() for t in (psi, ye, T)]


@pytest.mark.parametrize('n_e,n_ray', [(1, 305), (3, 304), (3, 305), (6, 305), (8, 456), (8, 457), (9, 228), (9, 229),
                                       (13, 76), (13, 77), (13, 153), (16, 77), (17, 152), (17, 153), (20, 153), (21, 76),
                                       (21, 77), (24, 77)])
def test_launches_agree(M, n_e, n_ray):
    inp = SP.strong(n_ray=n_ray, n_r=5, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0, pair=1.0)
    many = _step(M, inp)
    for some in ([0, 1], list(range(n_ray - 100, n_ray)) if n_ray > 200 else [n_ray - 1]):
        few = _step(M, problems.subset_rays(inp, some))
        for a, b in zip(many, few):
            assert np.array_equal(a[some], b)
