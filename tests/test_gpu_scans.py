"""The scans along a ray at the edges of their runs: the neutrinosphere's 32 chunks of zones (zone widths in
shared memory up to 2048 zones, from the edges beyond), the stress in runs of zones with the edge before
them, the lapse's runs per thread, and right-hand sides longer than the scaling kernel keeps in
registers (16384 entries).  Bounds: those of the stress parity tests (1e-13 of an edge's terms, lapse
1e-12) and the mixed step's gate 1e-10 (or the problem's FP64 floor)."""
import numpy as np
import pytest

from oracle import mgfld_oracle as O
from paper_1809_05608_gb300 import problems
from tests import small_problems as SP
from tests import test_gpu_stress as TS

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module', autouse=True)
def M():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_1809_05608_gb300 import mgfld
    mgfld.lib()
    TS.M = mgfld
    return mgfld


@pytest.mark.parametrize('n_r,n_e', [(2, 1), (11, 3), (12, 32), (13, 20), (24, 7), (25, 24), (300, 5), (2100, 4)])
def test_stress_and_lapse_runs(n_r, n_e):
    inp = SP.strong(n_ray=2, n_r=n_r, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0, lapse=True)
    p, m = problems.stress_inputs(inp)
    TS.check(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'], p, m)


@pytest.mark.parametrize('n_r,n_e', [(31, 9), (33, 9), (2049, 8), (2100, 8)])
def test_mixed_step_on_long_rays(M, n_r, n_e):
    inp = SP.strong(n_ray=1, n_r=n_r, n_e=n_e, kabs=1e12, kscat=1e13, nes=2.0)
    st = M.Stepper(inp, M.MGFLD_MIXED, tol=1e-11, max_iter=60)
    psi, ye, T = st.state_to_device(inp['psi0'], inp['ye0'], inp['T0'])
    assert st.step(psi, ye, T) == M.MGFLD_OK
    ref = O.step(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'])
    gate = max(1e-10, SP.fp64_tolerance(inp))
    err = np.abs(psi.cpu().numpy() - ref['psi'])
    assert np.max(np.max(err, axis=(2, 3)) / np.max(np.abs(ref['psi']), axis=(2, 3))) < gate
    assert np.max(np.abs(T.cpu().numpy() / ref['T'] - 1.0)) < gate
