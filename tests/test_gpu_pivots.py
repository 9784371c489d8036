"""The mixed path's FP32 factor of padded and pair blocks eliminates without row exchanges and does a system again
with partial pivoting where its pivot blocks are not an M-matrix's.  An iterate with occupations outside
[0, 1] can make a leading 2 x 2 block singular while the system is well conditioned: without the second
elimination the first Newton step has no correct digit.

One outer iteration from such an iterate is compared with the FP64 path's, whose correction has the exact factors.  The
outer iteration asks of its FP32 factors that the error of a correction be at most a tenth of it (refactor_ratio's
default: what contracts by less takes new factors), and so does the test."""
import numpy as np
import pytest

from oracle import mgfld_oracle as O
from paper_1809_05608_gb300 import problems
from tests import small_problems as SP

torch = pytest.importorskip('torch')
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings('ignore::RuntimeWarning')]


@pytest.fixture(scope='module')
def M():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_1809_05608_gb300 import mgfld
    mgfld.lib()
    return mgfld


def singular_start(n_e, seed, pair, n_ray, n_r=4):
    """The strong-coupling problem with random changes of the electron neutrinos' occupations in the first
    zone of ray 0, scaled so that the first 2 x 2 block of the Jacobian there is singular."""
    inp = SP.strong(n_ray=n_ray, n_r=n_r, n_e=n_e, kabs=1e12, kscat=1e13, nes=200.0, pair=pair)
    one = problems.subset_rays(inp, [0])
    d = np.random.default_rng(seed).uniform(-1.0, 1.0, n_e)

    def at(t):
        psi = one['psi0'].copy()
        psi[0, 0, 0] += t * d
        f = O.setup_step(one['problem'], psi, one['ye0'], one['T0'])
        return np.linalg.det(O.jacobian(f, psi, one['ye0'])[0][0, 0, :2, :2]), psi
    ts = np.linspace(0.0, 1.5, 31)
    for a, b in zip(ts, ts[1:]):
        va = at(a)[0]
        if va * at(b)[0] < 0.0:
            for _ in range(60):
                mid = 0.5 * (a + b)
                if at(mid)[0] * va > 0.0:
                    a = mid
                else:
                    b = mid
            psi0 = inp['psi0'].copy()
            psi0[0] = at(a)[1][0]
            return dict(inp, psi0=psi0)
    raise AssertionError('no singular block on the way')


# (153 rays: beyond 608 systems several half-systems share a warp)
@pytest.mark.parametrize('n_ray', [1, 153])
@pytest.mark.parametrize('n_e,seed,pair', [(5, 1, 0.0), (5, 8, 0.0), (7, 2, 0.0), (7, 7, 0.0), (7, 10, 0.0), (5, 0, 5.0),
                                           (7, 4, 5.0)])
def test_first_step_from_a_singular_pivot(M, n_e, seed, pair, n_ray):
    inp = singular_start(n_e, seed, pair, n_ray)
    got = []
    for precision in (M.MGFLD_FP64, M.MGFLD_MIXED):
        st = M.Stepper(inp, precision, tol=1e-11, max_iter=1)
        psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], inp['T0'])
        assert st.step(psi, ye, T) == M.MGFLD_ENOCONV
        got.append(psi.cpu().numpy() - inp['psi0'])
    err = np.max(np.abs(got[1] - got[0]), axis=(1, 2, 3)) / np.max(np.abs(got[0]), axis=(1, 2, 3))
    print(f'n_e {n_e}, pair {pair}, {n_ray} rays: correction of the singular ray off by {err[0]:.1e}, of the others by '
          f'{np.max(err[1:], initial=0.0):.1e}')
    assert np.all(err <= 0.1)
