"""The inverse form of the layer-block solver (the default) against the block
Cholesky (here requested by its left-looking schedule), at the edges of its range:
one to three element layers (half chains without layers), layers of one tile and of
a ragged last tile, in-plane boxes one element wide, loads with
nodal forces, uneven boxes, several waves.  Bars: those of the oracle parity tests
(1e-8 FP64, 1e-5 mixed, relative to the largest eigenvalue / component)."""
from dataclasses import replace

import numpy as np
import pytest

from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu

CASES = {
    "nz1": dict(NX=10, NY=5, NZ=1, sx=2, sy=1, overlap=1, oversampling=2, n_loc=6),
    "nz2": dict(NX=11, NY=4, NZ=2, sx=2, sy=1, overlap=1, oversampling=2, n_loc=7),
    "nz3": dict(NX=13, NY=3, NZ=3, sx=2, sy=1, overlap=1, oversampling=2, n_loc=7),
    "narrow": dict(NX=30, NY=1, NZ=9, sx=5, sy=1, overlap=1, oversampling=2, n_loc=7),
    "one_tile_full": dict(NX=9, NY=2, NZ=6, sx=2, sy=1, overlap=1, oversampling=2, n_loc=7),
    "ragged": dict(NX=25, NY=7, NZ=8, sx=3, sy=2, overlap=2, oversampling=3, n_loc=9),
    # FP64 layers too wide for the digit products' shared memory (plain FP64 products)
    "dfma": dict(NX=18, NY=30, NZ=3, sx=2, sy=1, overlap=1, oversampling=2, n_loc=8),
    "wide": dict(NX=34, NY=16, NZ=4, sx=2, sy=1, overlap=1, oversampling=2, n_loc=8),
}


def _run(cfg, **kw):
    from paper_2211_13893_gb300 import MSGFEM
    m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, **kw)
    lam = m.local_spaces(cfg.n_loc)
    m.coarse_assemble()
    u, _ = m.solve()
    prof = m.profile()
    m.close()
    return lam, u, prof


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_inverse_form_equals_block_cholesky(name, precision):
    from paper_2211_13893_gb300 import plan
    cfg = replace(get_config("t3"), name=name, **CASES[name])
    tol = 1e-8 if precision == 0 else 1e-5
    la, ua, pa = _run(cfg, precision=precision)
    lb, ub, pb = _run(cfg, precision=precision, factor_schedule=1)
    assert pa["factor_flops"] != pb["factor_flops"]     # the two paths did run
    scale = np.maximum(np.abs(lb).max(axis=1, keepdims=True), 1.0)   # a floating row may hold rigid zeros only
    assert (np.abs(la - lb) / scale).max() <= tol
    assert np.abs(ua - ub).max() <= tol * np.abs(ub).max()
    largest = plan(cfg, precision)["largest_mb"]
    lc, uc, pc = _run(cfg, precision=precision, wave_mb=1.01 * largest)
    assert pc["waves"] >= 2
    assert (np.abs(la - lc) / scale).max() <= tol
    assert np.abs(ua - uc).max() <= tol * np.abs(ub).max()


@pytest.mark.parametrize("precision", [0, 1])
def test_nodal_loads_and_gather_signs(precision):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="ragged", **CASES["ragged"])
    rng = np.random.default_rng(5)
    load = rng.standard_normal(cfg.n_dof)
    out = []
    for kw in (dict(), dict(factor_schedule=1)):
        m = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=precision, load=load, **kw)
        m.local_spaces(cfg.n_loc)
        psi = [m.export_local(j)[0][:, -1] for j in range(m.N)]
        out.append(psi)
        m.close()
    for a, b in zip(*out):
        assert np.abs(b).max() > 0
        # the particular function's bar of the oracle parity tests, times the norms' ratio
        assert np.linalg.norm(a - b) <= (1e-9 if precision == 0 else 1e-7) * np.linalg.norm(b)


# FP32 solves: blocks of 32 rows per rank and ranks per half chain.  Layers of 45 (NY + 1)
# and 42 (NY + 1) DoFs; few half chains take clusters of 8 (NY = 4: one block each, the last
# of one row; 5: ranks without rows; 15, 21: up to 4 blocks; 22: above 1,024 DoFs, the other
# kernel), 152 half chains clusters of 2 with 5 to 8 blocks.
@pytest.mark.parametrize("ny,instances", [(4, 1), (5, 1), (15, 1), (21, 1), (22, 1), (6, 38), (7, 38), (8, 38), (10, 38)])
def test_fp32_solve_row_blocks(ny, instances):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="rows", NX=24, NY=ny, NZ=3, sx=2, sy=1, overlap=1, oversampling=2, n_loc=6)
    rng = np.random.default_rng(ny)
    ang = rng.uniform(-90.0, 90.0, instances * cfg.NX * cfg.NY * cfg.NZ)
    out = []
    for kw in (dict(), dict(factor_schedule=1)):
        m = MSGFEM.from_config(cfg, ang, seed=7, precision=1, instances=instances, **kw)
        lam = np.array(m.local_spaces(cfg.n_loc))
        out.append((lam, [m.export_local(j)[0][:, -1] for j in (0, m.N - 1)]))
        m.close()
    (la, pa), (lb, pb) = out
    scale = np.maximum(np.abs(lb).max(axis=1, keepdims=True), 1.0)
    assert (np.abs(la - lb) / scale).max() <= 1e-5
    for a, b in zip(pa, pb):
        assert np.linalg.norm(a - b) <= 1e-7 * np.linalg.norm(b)


# Clusters that are no powers of two: layers of 3 to 7 blocks (32 rows in FP32, 16 in FP64),
# and 20 half chains, for which clusters of 8 are not resident at once.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ny,instances", [(1, 1), (2, 1), (3, 1), (4, 5)])
def test_cluster_sizes(ny, instances, precision):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="ranks", NX=24, NY=ny, NZ=4, sx=2, sy=1, overlap=1, oversampling=2, n_loc=6)
    rng = np.random.default_rng(ny)
    ang = rng.uniform(-90.0, 90.0, instances * cfg.NX * cfg.NY * cfg.NZ)
    out = []
    for kw in (dict(), dict(factor_schedule=1)):
        m = MSGFEM.from_config(cfg, ang, seed=7, precision=precision, instances=instances, **kw)
        lam = np.array(m.local_spaces(cfg.n_loc))
        out.append((lam, [m.export_local(j)[0][:, -1] for j in (0, m.N - 1)]))
        m.close()
    (la, pa), (lb, pb) = out
    scale = np.maximum(np.abs(lb).max(axis=1, keepdims=True), 1.0)
    assert (np.abs(la - lb) / scale).max() <= (1e-8 if precision == 0 else 1e-5)
    for a, b in zip(pa, pb):
        assert np.linalg.norm(a - b) <= (1e-9 if precision == 0 else 1e-7) * np.linalg.norm(b)


def test_wide_layers_keep_the_block_cholesky():
    """Layers whose solve stages exceed shared memory run the block Cholesky (same results bar)."""
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="big", NX=24, NY=48, NZ=2, sx=1, sy=2, overlap=1, oversampling=2, n_loc=8)
    a = MSGFEM.from_config(cfg, element_angles(cfg), seed=7)
    la = a.local_spaces(cfg.n_loc)
    fa = a.profile()["factor_flops"]
    b = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, factor_schedule=1)
    lb = b.local_spaces(cfg.n_loc)
    assert b.profile()["factor_flops"] == fa
    assert (np.abs(la - lb) / np.abs(lb).max(axis=1, keepdims=True)).max() <= 1e-8
    a.close()
    b.close()
