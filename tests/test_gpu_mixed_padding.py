"""The mixed path at the group counts around the padded block sizes 4, 8, 12, 16, 20, 24 and 32 that no other
test takes.  28 groups are the one multiple of 4 that is not a padded size itself: blocks of 28 rows run padded
to 32, with flags.  On both sides of the line between a warp per half-system and several (1216 systems, 608
of blocks below 16 rows).

The converged step is compared with the oracle's.  The mixed path iterates to tol = 1e-11 with each
correction at most a tenth of the one before, so what is left is below 1e-11 of max(|psi|, 1) plus the
FP64 floor of the problem (fp64_tolerance); the gate 1e-10 covers both where the floor does."""
import numpy as np
import pytest

from oracle import mgfld_oracle as O
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


@pytest.mark.parametrize('n_e,n_ray,n_r', [(3, 3, 21), (10, 3, 21), (22, 3, 21), (26, 3, 21), (27, 3, 21), (28, 3, 21),
                                           (29, 3, 21), (10, 153, 6), (22, 305, 6), (28, 305, 6)])
def test_block_sizes(M, n_e, n_ray, n_r):
    inp = SP.strong(n_ray=n_ray, n_r=n_r, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0)
    st = M.Stepper(inp, M.MGFLD_MIXED, tol=1e-11, max_iter=60)
    psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], inp['T0'])
    assert st.step(psi, ye, T) == M.MGFLD_OK
    ref = O.step(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'])
    gate = max(1e-10, SP.fp64_tolerance(inp))
    err = np.abs(psi.cpu().numpy() - ref['psi'])
    assert np.max(np.max(err, axis=(2, 3)) / np.max(np.abs(ref['psi']), axis=(2, 3))) < gate
    assert np.max(np.abs(T.cpu().numpy() / ref['T'] - 1.0)) < gate
