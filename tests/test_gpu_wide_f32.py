"""FP32 layers of 1,536 to about 2,000 DoFs, the widest that the inverse form's solves hold
in shared memory (four rows per stage, eight warps that share each row group): against the
block Cholesky, with the bars of the oracle parity tests for mixed precision (1e-5; 1e-7
for the particular functions)."""
from dataclasses import replace

import numpy as np
import pytest

from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu


# layers of 45 (ny + 1) and 42 (ny + 1) DoFs
@pytest.mark.parametrize("ny,nz", [(34, 2), (36, 3), (43, 2)])
def test_widest_fp32_layers(ny, nz):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="wide", NX=24, NY=ny, NZ=nz, sx=2, sy=1, overlap=1, oversampling=2, n_loc=8)
    out = []
    for kw in (dict(), dict(factor_schedule=1)):
        m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=1, **kw)
        lam = m.local_spaces(cfg.n_loc)
        out.append((lam, m.export_local(1)[0][:, -1], m.profile()["factor_flops"]))
        m.close()
    (la, pa, fa), (lb, pb, fb) = out
    assert fa != fb            # the inverse form did run
    assert (np.abs(la - lb) / np.maximum(np.abs(lb).max(axis=1, keepdims=True), 1.0)).max() <= 1e-5
    assert np.abs(pb).max() > 0 and np.linalg.norm(pa - pb) <= 1e-7 * np.linalg.norm(pb)
