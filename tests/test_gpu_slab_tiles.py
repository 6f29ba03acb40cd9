"""The 3-D strip solve at the edges of its tiles and of its two elimination chains: grids of
1 to 4 rows along y (no chain, one chain, uneven and even chains), blocks below, at and just
above the 64-row tile of the block layout and the 128-row tile of the products, and every
width of the right-hand-side tile (1, 2-4, 5-8, 9-16 and a remainder).

Bars, as for the other 3-D parity tests: 1e-10 relative in FP64, 2e-4 in mixed precision
(complex64 blocks, condition x 2^-24 with margin), against the CPU oracle.
"""
import numpy as np
import pytest

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu

# (n = (n_x, n_y, n_z), w_outer, w_sub, J, right-hand sides)
CASES = [
    ((9, 1, 5), 0, 2, 2, 1),        # one row: the middle row only
    ((9, 2, 5), 0, 2, 2, 3),        # two rows: only the bottom chain has a row of its own
    ((9, 3, 5), 0, 2, 2, 2),        # blocks of 35 and 30 unknowns: one column chunk of the tile
    ((10, 4, 8), 0, 2, 2, 6),       # uneven chains; blocks of 64 and 56: one full 64-row tile
    ((15, 5, 5), 1, 3, 2, 16),      # blocks around 85: the second half tile is partial
    ((14, 6, 9), 2, 3, 2, 17),      # blocks of 169 and 156: two row tiles; tiles of 16 and 1
    ((13, 3, 14), 1, 3, 2, 9),      # two rows below a full chunk of columns
]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 2e-4)])
@pytest.mark.parametrize("case", CASES)
def test_slab_tiles_match_oracle(case, prec, tol):
    n, w_o, w_s, J, B = case
    c = media.smooth_medium(n, 2.0, 1.0, 2.0, 11)
    h = 1.0 / 24
    omega = media.omega_for(c, h, 8.0)
    g = helm.HelmDD(c, h, omega, w_o, w_s, J, prec).factor()
    o = HelmholtzDD(c, h, omega, w_o, w_s, J).factor()
    f = media.random_rhs((B,) + g.shape, 23)
    Pf = g.apply_precond(f)
    for b in range(B):
        ref = o.apply_precond(f[b])
        assert np.linalg.norm(Pf[b] - ref) <= tol * np.linalg.norm(ref), (b, B)
    g.close()
