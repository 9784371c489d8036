"""The mixed path's FP32 factors on both sides of the line between a warp per half-system and several
half-systems per warp (1216 systems, 608 of blocks below 16 rows), for whole and padded blocks, with a ray whose
blocks cannot be eliminated where the factor keeps flags.

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


@pytest.mark.parametrize('n_e,n_ray', [(20, 304), (20, 305), (13, 304), (13, 305), (9, 152), (9, 153), (12, 153)])
def test_both_sides(M, n_e, n_ray):
    inp = SP.strong(n_ray=n_ray, n_r=6, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0)
    ref = O.step(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'])
    gate = max(1e-10, SP.fp64_tolerance(inp))
    bad = n_ray - 2
    for poison in (False, True):
        T0 = np.array(inp['T0'])
        if poison:
            T0[bad, 4] = np.nan
        st = M.Stepper(inp, M.MGFLD_MIXED, tol=1e-11, max_iter=60)
        psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], T0)
        assert st.step(psi, ye, T) == (M.MGFLD_ENAN if poison else M.MGFLD_OK)
        good = np.arange(n_ray) != (bad if poison else -1)
        err = np.max(np.abs(psi.cpu().numpy() - ref['psi']), axis=(2, 3)) / np.max(np.abs(ref['psi']), axis=(2, 3))
        assert np.max(err[good]) < gate
        assert np.max(np.abs(T.cpu().numpy() / ref['T'] - 1.0)[good]) < gate
        assert (st.report['ray_status'].cpu().numpy() == M.MGFLD_OK).tolist() == good.tolist()
