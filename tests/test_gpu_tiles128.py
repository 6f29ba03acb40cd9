"""Tiles of the complex128 strip solve: one right-hand side per CTA while the one-wide CTAs take
a few rounds of the SMs, four beyond (eight rounds where a solve has the GPU to itself, four
and a half with three streams).  The rule at both sides of its line, and the 4-wide tile at the
edges of its 16-row warps, with full tiles and remainders of one to three.

Bar, as for the other complex128 parity tests: 1e-10 relative against the CPU oracle.
"""
import numpy as np
import pytest
import torch

from oracle.helm_oracle import HelmholtzDD
from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sweep,streams,rounds", [("double", 1, 8.0), ("concurrent", 3, 4.5)])
def test_tile_width_rule(sweep, streams, rounds):
    n = (63, 61)
    g = helm.HelmDD(np.ones(tuple(reversed(n))), 1.0 / 64, 20.0, 5, 6, 4, "fp64", sweep=sweep)
    assert g.tile_width(4) == 0                      # not factored yet
    g.factor()
    ctas = g.chunks() + (1 if g.sep_groups() > 1 else 0)
    line = rounds * torch.cuda.get_device_properties(0).multi_processor_count / (ctas * streams)
    assert [g.tile_width(b) for b in (1, 2, int(line), int(line) + 1, 4 * int(line))] == [1, 1, 1, 4, 4]
    g.close()
    m = helm.HelmDD(np.ones(tuple(reversed(n))), 1.0 / 64, 20.0, 5, 6, 4, "mixed", sweep=sweep).factor()
    assert [m.tile_width(b) for b in (1, 2, 64)] == [1, 4, 4]
    m.close()


def _check(n, w_o, w_s, J, P, G, B, sweep):
    c = media.smooth_medium(n, 3.0, 1.0, 2.0, 9)
    h = 1.0 / 32
    omega = media.omega_for(c, h, 10.0)
    g = helm.HelmDD(c, h, omega, w_o, w_s, J, "fp64", chunks=P, sep_groups=G, sweep=sweep).factor()
    assert g.tile_width(B) == 4 and g.chunks() == P
    o = HelmholtzDD(c, h, omega, w_o, w_s, J, sweep=sweep).factor()
    f = media.random_rhs((B,) + g.shape, 31)
    Pf = g.apply_precond(f)
    for b in range(B):
        ref = o.apply_precond(f[b])
        assert np.linalg.norm(Pf[b] - ref) <= 1e-10 * np.linalg.norm(ref), (b, g.strip_widths())
    g.close()


@pytest.mark.parametrize("nx,B", [(8, 13), (10, 14), (40, 15), (42, 12), (56, 13), (70, 14)])
def test_widths_concurrent(nx, B):
    _check((nx, 45), 5, 6, 2, 20, 4, B, "concurrent")   # widths nx/2 + 12 and one less


@pytest.mark.parametrize("P,G,B", [(47, 6, 30), (24, 1, 55)])
def test_double_sweep(P, G, B):
    _check((44, 85), 5, 6, 2, P, G, B, "double")
