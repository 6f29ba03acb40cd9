"""The 4-wide tile of the complex64 strip solve and its output pass at their edges: strip widths
at and beside multiples of the 16-row warp tile up to the widest strip, full and partial tiles
of right-hand sides, groups of one to three separators and the single-chunk solve, one strip
and two (the transfer between them).

Bar, as for the other mixed-precision parity tests: 2e-4 relative against the CPU oracle
(complex64 factors, condition x 2^-24 with margin; 10 points per wavelength).  A lone strip may
be near a resonance, where complex64 misses the bar on every path; there the tile is held to
twice the error of the single-right-hand-side path on the same factors.
"""
import numpy as np
import pytest

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu


def _check(n, w_o, w_s, J, P, G, B):
    c = media.smooth_medium(n, 3.0, 1.0, 2.0, 9)
    h = 1.0 / 32
    omega = media.omega_for(c, h, 10.0)
    g = helm.HelmDD(c, h, omega, w_o, w_s, J, "mixed", chunks=P, sep_groups=G).factor()
    o = HelmholtzDD(c, h, omega, w_o, w_s, J).factor()
    f = media.random_rhs((B,) + g.shape, 31)
    Pf = g.apply_precond(f)
    for b in range(B):
        ref = o.apply_precond(f[b])
        single = np.linalg.norm(g.apply_precond(f[b:b + 1])[0] - ref)
        assert np.linalg.norm(Pf[b] - ref) <= max(2e-4 * np.linalg.norm(ref), 2 * single), (b, g.strip_widths())
    g.close()


@pytest.mark.parametrize("W,B", [(15, 2), (16, 4), (17, 3), (31, 5), (32, 2), (33, 4), (47, 3), (48, 18), (49, 2),
                                 (63, 4), (64, 7)])
def test_one_strip_widths(W, B):
    _check((W - 8, 31), 4, 3, 1, 7, 3, B)       # 39 rows: 6 separators in groups of 2, 1, 1


@pytest.mark.parametrize("P,G", [(1, 1), (2, 1), (3, 1), (5, 2), (12, 3)])
def test_two_strips_partitions(P, G):
    _check((44, 45), 5, 6, 2, P, G, 6)          # widths 34 and 33; a full tile and a pair
