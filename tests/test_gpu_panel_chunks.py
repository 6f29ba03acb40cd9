"""The built-in chunk count of a panel set before the factorisation.  Complex128 panels run one
right-hand side to a CTA, so their P + 1 CTAs per right-hand side fill whole rounds of the SMs;
the count is raised again where the longer chunks would not fit a strip solve's shared memory."""
import numpy as np
import pytest
import torch

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import autotune, helm, media

pytestmark = pytest.mark.gpu


def _problem(n, w_o, w_s, J, panel):
    c = media.smooth_medium(n, 3.0, 1.0, 2.0, 5)
    h = 1.0 / 32
    omega = media.omega_for(c, h, 8.0)
    return (helm.HelmDD(c, h, omega, w_o, w_s, J, "fp64", panel=panel).factor(),
            HelmholtzDD(c, h, omega, w_o, w_s, J).factor())


@pytest.mark.parametrize("panel", [5, 8, 9, 16, 50])
def test_complex128_panel_fills_whole_rounds(panel):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    g, o = _problem((60, 500), 6, 5, 4, panel)
    P, P0 = g.chunks(), autotune.builtin_chunks(g.N[1])
    assert (P0 + 5) // 6 <= P < P0
    # the last round of one-wide CTAs is nearly full: one more chunk would begin another
    assert (P + 1) * panel <= -(-(P + 1) * panel // nsm) * nsm < (P + 2) * panel
    B = min(panel, 9)
    f = media.random_rhs((B,) + g.shape, 21)
    Pf = g.apply_precond(f)
    for b in range(B):
        ref = o.apply_precond(f[b])
        assert np.linalg.norm(Pf[b] - ref) <= 1e-10 * np.linalg.norm(ref)
    g.close()


@pytest.mark.parametrize("panel", [8, 32])
def test_lowered_count_still_fits(panel):
    # one strip of 50 columns: a strip solve holds chunks of about 27 rows in complex128
    g, _ = _problem((42, 700), 4, 3, 1, panel)
    assert g.strip_widths() == [50] and g.chunks() < autotune.builtin_chunks(g.N[1])
    f = media.random_rhs((1,) + g.shape, 21)
    assert np.linalg.norm(g.matvec(g.apply_precond(f)) - f) <= 1e-8 * np.linalg.norm(f)   # one strip: P = A^-1
    g.close()
