"""The 3-D strip solve on large blocks with several right-hand sides: the vector gathered from many
row tiles, many ring slots to a step, and the narrower tiles taken where the 16-wide one (own
entries of a CTA) and the 8-wide one (shared memory) do not fit.

Bar, as for the other 3-D mixed-precision parity tests: 2e-4 relative against the CPU oracle
(complex64 blocks, condition x 2^-24 with margin).
"""
import numpy as np
import pytest

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,blocks", [((40, 2, 52), 2, [1860, 1800]),     # tiles of 16, 8 and 4
                                        ((44, 2, 90), 2, [3234, 3136]),     # 25 row tiles: 8 wide at most
                                        ((42, 1, 72), 1, [4000])])          # 1000 columns to a chunk: 4 at most
def test_large_blocks(n, J, blocks):
    c = media.smooth_medium(n, 2.0, 1.0, 2.0, 7)
    h = 1.0 / 24
    omega = media.omega_for(c, h, 8.0)
    g = helm.HelmDD(c, h, omega, 4, 6, J, "mixed").factor()
    assert [w * g.N[2] for w in g.strip_widths()] == blocks
    o = HelmholtzDD(c, h, omega, 4, 6, J).factor()
    f = media.random_rhs((16,) + g.shape, 19)
    ref = np.stack([o.apply_precond(f[b]) for b in range(16)])
    for B in (1, 3, 8, 16):
        Pf = g.apply_precond(f[:B])
        for b in range(B):
            assert np.linalg.norm(Pf[b] - ref[b]) <= 2e-4 * np.linalg.norm(ref[b]), (B, b)
    g.close()
