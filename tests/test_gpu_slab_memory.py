"""The 3-D complex64 factorisation with little device memory left: it inverts the blocks of up to
eight strips side by side and takes fewer when the scratch of all does not fit, with the same
factors (the strips do not depend on each other)."""
import numpy as np
import pytest
import torch

from paper_1208_3956_gb300 import helm, media

pytestmark = pytest.mark.gpu


def test_factor_with_little_memory_left():
    n, w_o, w_s, J = (64, 5, 71), 2, 5, 8     # eight strips, blocks of up to 1425 unknowns
    c = media.smooth_medium(n, 2.0, 1.0, 2.0, 7)
    h = 1.0 / 24

    def make():
        return helm.HelmDD(c, h, media.omega_for(c, h, 8.0), w_o, w_s, J, "mixed")

    g = make().factor()
    f = torch.as_tensor(media.random_rhs((1,) + g.shape, 3), device="cuda")
    ref = g.apply_precond(f)
    nmax = max(g.strip_widths()) * g.N[2]
    g.close()
    torch.cuda.empty_cache()
    block = 8 * nmax * nmax
    padded = -(-nmax // 64) * 64 * nmax * 8   # a stored block
    g = make()
    # what stays with the handle, and 10.5 blocks for the factorisation: eight strips side by side
    # take sixteen and their panels
    keep = J * g.N[1] * padded + (16 << 20)
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - keep - 21 * block // 2, dtype=torch.uint8, device="cuda")
    g.factor()
    del fill
    torch.cuda.empty_cache()
    err = float(torch.linalg.norm(g.apply_precond(f) - ref) / torch.linalg.norm(ref))
    assert err <= 1e-6, err   # complex64 rounding of one P
    g.close()
