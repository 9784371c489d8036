"""The FP64 elimination and substitution over their routes: one or two block rows per lane (chosen by
the number of systems), blocks that fill their padded size and blocks that do not, factors on and off
the 16-byte boundaries that bulk copies start on, rhs and solution in one array.  Every route does the
same operations on an entry in the same order, so the results are compared bit for bit."""
import numpy as np
import pytest

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


def _system(n_ray, n_r, n_e):
    """Random diagonally dominant blocks that need row exchanges, and couplings."""
    g = np.random.default_rng(100 * n_r + n_e)
    shape = (n_ray, 4, n_r, n_e)
    diag = g.standard_normal(shape + (n_e,))
    perm = g.permutation(n_e)
    diag[..., np.arange(n_e), perm] += 3.0 * n_e * np.where(g.random(shape) < 0.5, 1.0, -1.0)
    lower, upper = g.standard_normal(shape), g.standard_normal(shape)
    lower[:, :, 0] = 0.0
    upper[:, :, -1] = 0.0
    rhs = g.standard_normal(shape)
    return {k: torch.as_tensor(v, device='cuda') for k, v in
            dict(diag=diag, lower=lower, upper=upper, rhs=rhs).items()}


def _solve(M, s, offset=0, alias=False):
    n_ray, _, n_r, n_e = s['rhs'].shape
    d = M.Dims(n_ray, n_r, n_e, 4)
    f = torch.empty(s['diag'].numel() + offset, dtype=torch.float64, device='cuda')[offset:]
    assert M.mgfld_factor(d, s, M.MGFLD_FP64, f) == M.MGFLD_OK
    rhs = s['rhs'].clone()
    x = rhs if alias else torch.full_like(rhs, np.nan)
    assert M.mgfld_solve(d, s, M.MGFLD_FP64, f, rhs, x) == M.MGFLD_OK
    torch.cuda.synchronize()
    return f.clone(), x


@pytest.mark.parametrize('n_r', [1, 2, 3, 9])
@pytest.mark.parametrize('n_e,n_ray', [(3, 700), (4, 700), (7, 400), (12, 170), (13, 170), (20, 80), (21, 80), (24, 80),
                                       (31, 80), (32, 80)])
def test_routes_agree(M, n_e, n_ray, n_r):
    many = _system(n_ray, n_r, n_e)                       # two rows per lane
    f, x = _solve(M, many)
    few = {k: v[-3:].contiguous() for k, v in many.items()}
    f1, x1 = _solve(M, few)                               # one row per lane
    assert torch.equal(f.reshape(many['diag'].shape)[-3:], f1.reshape(few['diag'].shape))
    assert torch.equal(x[-3:], x1)
    _, off = _solve(M, few, offset=1)                     # factors off the 16-byte boundaries
    assert torch.equal(off, x1)
    _, same = _solve(M, few, alias=True)
    assert torch.equal(same, x1)
    # and they solve the system: each block row's residual within rounding of the size of its terms
    D, lo, up, b = (many[k] for k in ('diag', 'lower', 'upper', 'rhs'))
    r = (D * x[..., None, :]).sum(-1) - b
    t = (D * x[..., None, :]).abs().sum(-1) + b.abs()
    if n_r > 1:
        r[:, :, 1:] += lo[:, :, 1:] * x[:, :, :-1]
        r[:, :, :-1] += up[:, :, :-1] * x[:, :, 1:]
        t[:, :, 1:] += (lo[:, :, 1:] * x[:, :, :-1]).abs()
        t[:, :, :-1] += (up[:, :, :-1] * x[:, :, 1:]).abs()
    # the explicit inverses of well-conditioned blocks (cond < ~10): n_e eps a dot product, a few of them
    assert float((r.abs() / t.amax(dim=-1, keepdim=True)).max()) < 100 * n_e * 2.2e-16
