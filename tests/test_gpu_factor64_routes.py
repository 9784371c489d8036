"""The FP64 elimination and substitution on both sides of the lines between their kernels, which the number of
systems and the block width choose: one or two block rows per lane of k_factor64, a thread per row (k_factor) for
many systems, the ring-fed substitution or a thread per row (k_solve).  Every route does the same operations on an entry in
the same order, so systems of a large launch end with the bits they have in a small one."""
import numpy as np
import pytest

from tests import test_gpu_factor64 as routes

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module')
def M():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_1809_05608_gb300 import mgfld
    mgfld.lib()
    return mgfld


# n_ray of the large launch (4 systems a ray):
# 8 rows: a thread per row from 1217 systems; 12: from 609 (two halves of 12 a warp); 16: from 609; 20: where its whole
# waves are fewer (k_factor<20> at 1200, 1216 and 2400, k_factor64<20, 2> at 400 and 1220 systems); 24: two rows per lane from 305,
# a thread per row from 609; 32: two rows per lane from 305.  The substitution: 1217 systems and more by a thread per row.
@pytest.mark.parametrize('n_r', [2, 5])
@pytest.mark.parametrize('n_e,n_ray', [(5, 305), (8, 304), (8, 305), (9, 153), (12, 152), (12, 153), (16, 153), (17, 305),
                                       (20, 100), (20, 300), (20, 304), (20, 305), (20, 600), (21, 80), (23, 160), (24, 152),
                                       (24, 153), (24, 305), (26, 160), (28, 80), (32, 160)])
def test_large_and_small_launches(M, n_e, n_ray, n_r):
    many = routes._system(n_ray, n_r, n_e)
    f, x = routes._solve(M, many)
    few = {k: v[-3:].contiguous() for k, v in many.items()}
    f1, x1 = routes._solve(M, few)
    assert torch.equal(f.reshape(many['diag'].shape)[-3:], f1.reshape(few['diag'].shape))
    assert torch.equal(x[-3:], x1)
    assert bool(torch.isfinite(x).all())


@pytest.mark.parametrize('n_e', [1, 2, 3, 4])
def test_thread_per_row_blocks_of_up_to_four(M, n_e):
    """Blocks of up to 4 rows take k_factor at any number of systems: against the inverse of the first zone's
    block and the residual of the solution, within the rounding of well-conditioned blocks (cond < ~10)."""
    s = routes._system(2, 3, n_e)
    f, x = routes._solve(M, s)
    inv = torch.linalg.inv(s['diag'][:, :, 0])
    got = f.reshape(s['diag'].shape)[:, :, 0]
    assert float(((got - inv).abs().amax((-1, -2)) / inv.abs().amax((-1, -2))).max()) < 100 * n_e * 2.2e-16
    r = (s['diag'] * x[..., None, :]).sum(-1) - s['rhs']
    t = (s['diag'] * x[..., None, :]).abs().sum(-1) + s['rhs'].abs()
    for a, b, c in ((slice(1, None), slice(None, -1), 'lower'), (slice(None, -1), slice(1, None), 'upper')):
        r[:, :, a] += s[c][:, :, a] * x[:, :, b]
        t[:, :, a] += (s[c][:, :, a] * x[:, :, b]).abs()
    assert float((r.abs() / t.amax(dim=-1, keepdim=True)).max()) < 100 * n_e * 2.2e-16
