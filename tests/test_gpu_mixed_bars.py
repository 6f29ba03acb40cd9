"""Mixed precision against bars that do not depend on the code under test: the 4-wide tile of the
complex64 strip solve over its widths, and the 2-D factorisation below and above the line of two
CTAs per SM.

Bars: the largest condition number over the sub-blocks that the partitioned elimination inverts
(runs of rows of a chunk from either end to its middle, and whole chunks; from the oracle's strip
operators) times the complex64 roundoff 2^-24, and 2e-4, the bar of the other mixed-precision parity
tests, where that is larger: 350 .. 1900 for the widths (1.1e-4), 3.1e4 and 3.8e4 (1.9e-3, 2.3e-3)
for the 40 strips of 170 columns in 7 and 8 chunks, which have a chunk near a resonance, 2400 in
19, 110 for the 8 strips of 222.
"""
import numpy as np
import pytest
import torch

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu


def _problem(n):
    c = media.smooth_medium(n, 3.0, 1.0, 2.0, 9)
    h = 1.0 / 32
    return c, h, media.omega_for(c, h, 10.0)


@pytest.mark.parametrize("nx,B", [(8, 2), (10, 3), (40, 4), (42, 5), (56, 18), (70, 6), (72, 7), (74, 2), (100, 3),
                                  (102, 4), (104, 17)])
def test_panel_widths(nx, B):
    c, h, omega = _problem((nx, 45))
    g = helm.HelmDD(c, h, omega, 5, 6, 2, "mixed", chunks=12, sep_groups=3).factor()
    assert g.strip_widths() == [nx // 2 + 12, nx // 2 + 11]
    o = HelmholtzDD(c, h, omega, 5, 6, 2).factor()
    f = media.random_rhs((B,) + g.shape, 31)
    Pf = g.apply_precond(f)
    for b in range(B):
        ref = o.apply_precond(f[b])
        assert np.linalg.norm(Pf[b] - ref) <= 2e-4 * np.linalg.norm(ref), b
    g.close()


@pytest.mark.parametrize("n,w_s,J,runs", [((170, 86), 3, 40, [(7, 1, 1.9e-3), (8, 1, 2.3e-3), (19, 9, 2e-4)]),
                                          ((222, 118), 8, 8, [(38, 1, 2e-4), (39, 1, 2e-4), (50, 3, 2e-4)])])
def test_factor_grids(n, w_s, J, runs):
    line = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    c, h, omega = _problem(n)
    o = HelmholtzDD(c, h, omega, 5, w_s, J).factor()
    f = media.random_rhs((1,) + tuple(reversed(o.N)), 31)
    ref = o.apply_precond(f[0])
    above = []
    for P, G, bar in runs:
        g = helm.HelmDD(c, h, omega, 5, w_s, J, "mixed", chunks=P, sep_groups=G).factor()
        above.append(g.chunks() * J > line)
        assert np.linalg.norm(g.apply_precond(f)[0] - ref) <= bar * np.linalg.norm(ref), (P, G)
        g.close()
    assert any(above) and not all(above)
