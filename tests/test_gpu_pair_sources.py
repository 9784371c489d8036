"""The final sources of the mixed pair path where the last correction is not small: a ray stopped by max_iter, and
a step converged to a loose tolerance.  T follows from the sources at the psi and Ye that the step returns (Eq. a62b), so
it is compared with the oracle's sources at those.

The tolerance is a bound on FP64 rounding: the sums of n_e products each within (2 n_e + 40) eps of the sum of their
terms' magnitudes, the emissivity's exponent (mu - eps)/T within a few eps of its terms, the energies within a few eps."""
import numpy as np
import pytest

from oracle import mgfld_oracle as O
from tests import small_problems as SP

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope='module')
def M():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_1809_05608_gb300 import mgfld
    mgfld.lib()
    return mgfld


def _temperature(inp, psi, ye):
    """T of Eq. a62b from the sources at (psi, Ye), and the rounding bound of it."""
    f = O.setup_step(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'])
    S, _, j, _, _ = O.sources(f, psi, ye)
    mu_q, _ = O.species_mu(f.rho, f.T_n, ye, f.eos)
    p = np.abs(psi)
    bar = p[:, O.PAIR_PARTNER]

    def rows(kernel, x):
        return O.C_NES * np.einsum('rikm,rim,rqim->rqik', kernel, f.w, x)
    terms = f.kappa_abs * p + (1.0 + p) * rows(f.phi_in, p) + p * rows(f.phi_out, 1.0 + p)
    terms = terms + (1.0 + p) * rows(f.pair_p, 1.0 + bar) + p * rows(f.pair_a, bar)
    arg = (np.abs(mu_q)[..., None] + f.eps[:, None]) / f.T_n[:, None, :, None]
    dS = EPS * ((2 * f.n_e + 40) * terms + (40.0 + 8.0 * arg) * j * (1.0 + p))
    to_e = (f.lapse * O.C_LIGHT * f.dt) * O.FOUR_PI_HC3 * (f.eos.m_b / f.rho)
    sums = [to_e * np.einsum('q,rik,rqik->ri', O.STAT_WEIGHT, f.w * f.eps, x) for x in (S, dS)]
    e = f.e_n - sums[0]
    T = O.temperature_from_e(f.rho, e, ye, f.eos)
    cold = np.abs(O.e_int(f.rho, np.zeros_like(T), ye, f.eos))
    slope = (O.e_int(f.rho, T, ye, f.eos) - O.e_int(f.rho, np.zeros_like(T), ye, f.eos)) / T
    return T, (sums[1] + 16.0 * EPS * (np.abs(f.e_n) + np.abs(sums[0]) + cold)) / slope


@pytest.mark.parametrize('n_e', [5, 8, 20])
@pytest.mark.parametrize('tol,max_iter', [(1e-11, 1), (1e-11, 2), (1e-2, 40), (1e-11, 60)])
def test_temperature_follows_the_returned_state(M, n_e, tol, max_iter):
    inp = SP.strong(n_ray=3, n_r=9, n_e=n_e, kabs=1e14, kscat=1e14, nes=10.0, pair=10.0)
    inp = dict(inp, psi0=1e-3 * inp['psi0'])
    st = M.Stepper(inp, M.MGFLD_MIXED, tol=tol, max_iter=max_iter)
    psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], inp['T0'])
    assert st.step(psi, ye, T) == (M.MGFLD_ENOCONV if max_iter < 40 else M.MGFLD_OK)
    ref, bound = _temperature(inp, psi.cpu().numpy(), ye.cpu().numpy())
    err = np.abs(T.cpu().numpy() - ref)
    print(f'n_e {n_e}, tol {tol}, max_iter {max_iter}: at most {np.max(err / bound):.2e} of the rounding bound, '
          f'{np.max(err / np.abs(ref)):.2e} relative')
    assert np.all(err <= bound)
