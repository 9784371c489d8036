"""The mixed path's ring-fed substitution where its rings can go wrong: halves of no zone, of one, and
around whole groups of zones; block sizes of every padded width, with rows that fill it (16-byte
pieces), even and odd ones (bulk copies that start and end inside the 16-byte pieces they move).

The converged step is compared with the oracle's.  The mixed path iterates to tol = 1e-11 with each
correction at most a tenth of the one before, so what is left is below 1e-11 of max(|psi|, 1) plus the
FP64 floor of the problem (fp64_tolerance); the path's gate 1e-10 covers both where the floor does."""
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


def _check(M, inp):
    st = M.Stepper(inp, M.MGFLD_MIXED, tol=1e-11, max_iter=60)
    psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], inp['T0'])
    assert st.step(psi, ye, T) == M.MGFLD_OK
    ref = O.step(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'])
    gate = max(1e-10, SP.fp64_tolerance(inp))
    err = np.abs(psi.cpu().numpy() - ref['psi'])
    assert np.max(np.max(err, axis=(2, 3)) / np.max(np.abs(ref['psi']), axis=(2, 3))) < gate
    assert np.max(np.abs(T.cpu().numpy() / ref['T'] - 1.0)) < gate


@pytest.mark.parametrize('n_r', [1, 2, 3, 4, 15, 16, 17, 18, 19, 33, 35])
@pytest.mark.parametrize('n_e', [13, 20])
def test_group_edges(M, n_r, n_e):
    _check(M, SP.strong(n_ray=2, n_r=n_r, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0))


@pytest.mark.parametrize('n_e', [1, 2, 5, 6, 7, 9, 11, 14, 16, 17, 19, 21, 23, 24, 25, 30, 31, 32])
def test_block_sizes(M, n_e):
    _check(M, SP.strong(n_ray=3, n_r=21, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0))
