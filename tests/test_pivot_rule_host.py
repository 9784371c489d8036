"""The rule by which the mixed path's unpivoted FP32 elimination (2 x 2 pivot blocks) is taken as it is or done again with
partial pivoting, restated in float32 on the oracle's Jacobian blocks: determinant and diagonal entries of each pivot
block positive, none above 4 times the raw diagonal entry.  Blocks of occupations between 0 and 1 are
M-matrices and always taken, those of the pair process with the antineutrinos' rows and columns
included; of the others, whatever is taken is as good a factor as the outer iteration asks (it contracts by 0.1)."""
import numpy as np
import pytest

from oracle import mgfld_oracle as O
from tests import small_problems as SP

F = np.float32


def eliminate(block):
    """The inverse by Gauss-Jordan with 2 x 2 pivot blocks in float32, and whether the rule takes it."""
    n = len(block)
    a = np.eye(n + n % 2, dtype=F)
    a[:n, :n] = block
    top = F(4.0) * np.diag(a)
    taken = True
    for p in range(0, len(a), 2):
        q = a[p:p + 2, p:p + 2].copy()
        det = F(np.float64(q[0, 0]) * q[1, 1] - F(q[0, 1] * q[1, 0]))
        taken = taken and det > 0 and all(0 < q[i, i] <= top[p + i] for i in (0, 1))
        if not taken:
            return None, False
        inv = np.array([[q[1, 1], -q[0, 1]], [-q[1, 0], q[0, 0]]], dtype=F) * (F(1.0) / det)
        f = (a[:, p:p + 2] @ inv).astype(F)
        f[p:p + 2] = np.eye(2, dtype=F) - inv
        rows = a[p:p + 2].copy()
        for i in (0, 1):
            a = (a - f[:, i:i + 1] * rows[i:i + 1]).astype(F)
        a[:, p:p + 2] = -f
        a[p:p + 2, p:p + 2] = inv
    return a[:n, :n], True


@pytest.mark.parametrize('n_e', [3, 5, 9, 13, 21])
@pytest.mark.parametrize('nes,pair', [(2.0, 0.0), (300.0, 0.0), (30.0, 10.0)])
@pytest.mark.parametrize('amp', [0.0, 0.1, 1.0])
def test_what_the_rule_takes(n_e, nes, pair, amp):
    inp = SP.strong(n_ray=1, n_r=6, n_e=n_e, kabs=1e12, kscat=1e13, nes=nes, pair=pair)
    f = O.setup_step(inp['problem'], inp['psi0'], inp['ye0'], inp['T0'])
    g = np.random.default_rng(n_e)
    width = 2 * n_e if pair else n_e
    counts = [0, 0]
    for _ in range(10):
        shape = inp['psi0'].shape
        psi = g.uniform(0.0, 1.0, shape) if amp == 0.0 else inp['psi0'] + g.uniform(-amp, amp, shape)
        A = O.jacobian(f, psi, inp['ye0'])[0][0]
        for block in [a[:width, :width] for a in A]:
            inv, taken = eliminate(block)
            counts[taken] += 1
            if taken:
                assert np.max(np.abs(np.linalg.eigvals(np.eye(width) - inv @ block))) <= 0.1
    print(f'{counts[1]} blocks taken, {counts[0]} done again')
    assert counts[1] > 0 and (amp > 0.0 or counts[0] == 0)
