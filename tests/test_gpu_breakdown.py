"""A Krylov basis that overflows to NaN is never taken for a converged one: start blocks
of finite but huge entries (1e36) overflow the FP32 solves of a mixed handle whose earlier
local stage left valid Ritz values behind; the subdomains fall back to the cold start as
with any start that leads nowhere, with the eigenvalues (1e-5, the bar of the mixed
precision) and residuals of a cold run."""
import numpy as np
import pytest

from parity_util import assert_eigs
from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu


def test_overflowing_start_block_falls_back_to_cold_start():
    import torch
    from paper_2211_13893_gb300 import MSGFEM
    cfg = get_config("t2")
    ang = element_angles(cfg)
    m = MSGFEM.from_config(cfg, ang, seed=3, precision=1)
    cold = m.local_spaces(cfg.n_loc).copy()
    torch.manual_seed(1)
    blocks = {}
    for j in range(m.N):
        n2, nw = m.warm_sizes(j, cfg.n_loc)
        if nw > 0:
            blocks[j] = 1e36 * torch.rand((n2, 8), dtype=torch.float32, device="cuda")
            m.set_start_block(j, blocks[j], 8, 8)
    assert blocks
    lam = m.local_spaces(cfg.n_loc)
    for j in range(m.N):
        assert m.info(j)["cold_restart"] == (1 if j in blocks else 0), j
        assert_eigs(lam[j], cold[j], 1e-5, j)
        phi, _ = m.basis(j)
        assert np.all(np.isfinite(phi))
    assert max(m.info(j)["residual"] for j in range(m.N)) <= 1e-5
    m.close()
