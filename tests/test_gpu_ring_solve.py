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


def _check(M, inp, tol=1e-11):
    st = M.Stepper(inp, M.MGFLD_MIXED, tol=tol, max_iter=60)
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


@pytest.mark.parametrize('n_e', [7, 8, 9, 10, 12, 13, 15, 18, 20, 22, 24, 25])
def test_incremental_residual(M, n_e):
    """The later residual passes for group counts that the kernel is compiled for and their neighbours,
    with a last block of fewer zones; from an empty state, so that the first corrections are as large as
    the occupations and their sums are formed again."""
    inp = SP.strong(n_ray=3, n_r=7, n_e=n_e, kabs=1e13, kscat=1e13, nes=5.0)
    _check(M, dict(inp, psi0=1e-3 * inp['psi0']))


@pytest.mark.parametrize('n_e,pair', [(13, False), (10, False), (5, True), (20, True)])
def test_a_failed_factor_stays_with_its_ray(M, n_e, pair):
    """A ray whose blocks cannot be eliminated (a NaN temperature in one zone) is done again with
    partial pivoting, fails on its own and leaves the other rays' results as they are without it."""
    inp = SP.strong(n_ray=3, n_r=11, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0, pair=1.0 if pair else 0.0)
    got = []
    for poison in (False, True):
        T0 = np.array(inp['T0'])
        if poison:
            T0[1, 4] = np.nan
        st = M.Stepper(inp, M.MGFLD_MIXED, tol=1e-11, max_iter=60)
        psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], T0)
        code = st.step(psi, ye, T)
        assert code == (M.MGFLD_ENAN if poison else M.MGFLD_OK)
        got.append((psi.cpu().numpy(), st.report['ray_status'].cpu().numpy()))
    assert got[1][1].tolist() == [M.MGFLD_OK, M.MGFLD_ENAN, M.MGFLD_OK]
    for ray in (0, 2):
        assert np.array_equal(got[0][0][ray], got[1][0][ray])


@pytest.mark.parametrize('n_r', [1, 2, 5, 9])
@pytest.mark.parametrize('n_e', [3, 4, 13, 16, 18, 20, 23, 24])
def test_pair_block_sizes(M, n_e, n_r):
    _check(M, SP.strong(n_ray=2, n_r=n_r, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0, pair=1.0))
