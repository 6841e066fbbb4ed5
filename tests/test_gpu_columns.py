"""Counts of eigenvectors around the groups of eight columns in which the residuals and
the coarse assembly evaluate their products: the coarse solution equals, in the energy
norm, the Galerkin solution that NumPy forms from the exported local vectors with the
oracle's stiffness matrix (1e-8; both sides solve the same coarse problem in FP64, also
in mixed precision), and every subdomain reports a residual of its wanted pairs."""
import functools

import numpy as np
import pytest

from oracle.coarse import coarse_solve, gram_schmidt, run_msgfem
from parity_util import energy_rel
from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=None)
def _problem(name):
    return run_msgfem(get_config(name), n_loc=7, keep_problems=True)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_loc", [7, 8, 15, 16, 23, 24, 31])
def test_column_groups(n_loc, precision):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = get_config("t2")
    ref = _problem("t2")
    m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=precision)
    m.local_spaces(n_loc, allow_noconv=True)
    m.coarse_assemble()
    u, _ = m.solve()
    cols = []
    for j, lp in enumerate(ref.problems):
        vec, _ = m.export_local(j)
        assert m.info(j)["residual"] > 0.0, (j, m.info(j))
        keep = [lp.mu * vec[:, k] for k in list(range(n_loc)) + [vec.shape[1] - 1] if np.any(vec[:, k] != 0.0)]
        gd = (3 * lp.nodes[:, None] + np.arange(3)).ravel()
        for q in gram_schmidt(lp.A, keep):
            col = np.zeros(len(ref.b))
            col[gd] = q
            cols.append(col)
    m.close()
    V = np.stack(cols, axis=1)
    AH = V.T @ (ref.A @ V)
    want = V @ coarse_solve(0.5 * (AH + AH.T), V.T @ ref.b)
    assert energy_rel(ref.A, u, want) <= 1e-8
