"""Thresholds that no eigenvector of a subdomain passes.  A clamped subdomain without load
then contributes nothing (no rigid modes, no particular function): its basis size is 0 and
the coarse solution is the oracle's at the same threshold (1e-8, mixed 1e-5, energy norm).
With GenEO on clamped subdomains only, the whole coarse space is empty: dimension 0 and
u = 0, on a fresh handle and after a coarse space that was not empty; a later assembly is
that of a handle that never had the empty one, bit for bit."""
from dataclasses import replace

import numpy as np
import pytest

from oracle.coarse import run_msgfem
from parity_util import energy_rel
from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_subdomains_without_basis(precision):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = get_config("t2")
    m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=precision)
    lam = m.local_spaces(cfg.n_loc)
    clamped = [j for j in range(m.N) if not m.info(j)["floating"]]
    t = 2.0 / lam[clamped].min()
    ref = run_msgfem(cfg, threshold=t)
    assert m.coarse_assemble(threshold=t) == sum(ref.basis_counts)
    assert [m.info(j)["basis_size"] for j in range(m.N)] == ref.basis_counts
    assert clamped and all(ref.basis_counts[j] == 0 for j in clamped)
    u, _ = m.solve()
    assert energy_rel(ref.A, u, ref.uG) <= (1e-8 if precision == 0 else 1e-5)
    m.close()


@pytest.mark.parametrize("kw", [dict(), dict(factor_schedule=1)])
def test_empty_coarse_space(kw):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t2"), NX=6, NY=8, sx=1, sy=2, overlap=1, oversampling=1, n_loc=6)
    m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, method=1, **kw)
    lam = m.local_spaces(cfg.n_loc)
    assert lam.min() > 0.0
    none = 2.0 / lam.min()
    assert m.coarse_assemble(threshold=none) == 0          # fresh
    u, err = m.solve(u_ref=np.sin(np.arange(cfg.n_dof)))
    assert np.all(u == 0.0) and err == pytest.approx(1.0, rel=1e-12)
    nc = m.coarse_assemble()
    assert nc == cfg.n_loc * m.N
    u1, _ = m.solve()
    assert m.coarse_assemble(threshold=none) == 0          # after one that was not empty
    u, _ = m.solve()
    assert np.all(u == 0.0)
    assert m.coarse_assemble() == nc
    u2, _ = m.solve()
    assert np.any(u1 != 0.0) and np.array_equal(u1, u2)
    m.close()
