"""The 2-D factorisation on grids of more CTAs than two per SM, where the complex64 kernels for
strips of up to 48 columns are built for three: chunk grids just above and below that line,
with the separator groups on either side of it.

Bar, as for the other mixed-precision parity tests: 2e-4 relative against the CPU oracle
(complex64 factors, condition x 2^-24 with margin; 10 points per wavelength), or twice the error
of a partition that stays below the line where that one misses it too.
"""
import numpy as np
import pytest
import torch

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,w_o,w_s,J,groups", [((170, 86), 5, 3, 40, 9), ((222, 118), 5, 8, 8, 3)])
def test_grids_beyond_two_per_sm(n, w_o, w_s, J, groups):
    line = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    c = media.smooth_medium(n, 3.0, 1.0, 2.0, 9)
    h = 1.0 / 32
    omega = media.omega_for(c, h, 10.0)
    o = HelmholtzDD(c, h, omega, w_o, w_s, J).factor()
    f = media.random_rhs((1, n[1] + 2 * w_o, n[0] + 2 * w_o), 31)
    ref = o.apply_precond(f[0])
    below = line // J
    err = []
    for P, G in ((below, 1), (below + 1, 1), (below + 12, groups)):
        g = helm.HelmDD(c, h, omega, w_o, w_s, J, "mixed", chunks=P, sep_groups=G).factor()
        assert g.chunks() == P and max(g.strip_widths()) <= 48
        assert (g.chunks() * J > line) == (P > below)
        err.append(np.linalg.norm(g.apply_precond(f)[0] - ref) / np.linalg.norm(ref))
        g.close()
    assert max(err[1:]) <= max(2e-4, 2 * err[0]), err
