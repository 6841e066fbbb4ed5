"""Device memory that the caller's allocator refuses in the middle of a call: the call
returns ENOMEM, and once memory is there again the handle works as one that never met the
refusal, bit for bit (the calls are deterministic).  Every allocation of the call is
refused once, the first, the second and so on, each on a fresh handle."""
from dataclasses import replace

import numpy as np
import pytest

from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu


class Refusing:
    """PyTorch's caching allocator; the allocation number `at` after arm(at) is refused."""

    def __init__(self):
        import torch
        self.torch, self.left, self.refused = torch, -1, False

    def arm(self, at):
        self.left, self.refused = at, False

    def alloc(self, n):
        if self.left == 0:
            self.left, self.refused = -1, True
            return None
        self.left -= self.left > 0
        return self.torch.cuda.caching_allocator_alloc(n, device=self.torch.cuda.current_device())

    def free(self, p, n):
        self.torch.cuda.caching_allocator_delete(p)

    def refuse(self, at, call):
        """call() with its allocation `at` refused (ENOMEM); False when it has no such allocation."""
        from paper_2211_13893_gb300.msgfem import MsgfemError
        self.arm(at)
        try:
            call()
        except MsgfemError as err:
            assert err.code == 2 and self.refused, err
        met, self.left = self.refused, -1
        return met


@pytest.mark.parametrize("kw", [dict(), dict(factor_schedule=1), dict(precision=1)])
def test_coarse_assembly(kw):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), n_loc=24)
    ang = element_angles(cfg)
    ref = MSGFEM.from_config(cfg, ang, seed=5, **kw)
    lam = ref.local_spaces(cfg.n_loc)
    small = 1.0 / np.median(lam)                # a threshold that keeps a smaller coarse space
    dims, sols = [], []
    for t in (0.0, small):
        dims.append(ref.coarse_assemble(threshold=t))
        sols.append(ref.solve()[0])
    ref.close()
    assert -(-dims[1] // 64) < -(-dims[0] // 64)   # another number of tiles
    mem = Refusing()
    for first in (None, small):                 # the arrays grow from nothing, from the small coarse space
        at = 0
        while True:
            m = MSGFEM.from_config(cfg, ang, seed=5, allocator=(mem.alloc, mem.free), **kw)
            m.local_spaces(cfg.n_loc)
            if first is not None:
                m.coarse_assemble(threshold=first)
            met = mem.refuse(at, m.coarse_assemble)
            for t, dim, want in ((0.0, dims[0], sols[0]), (small, dims[1], sols[1])):
                assert m.coarse_assemble(threshold=t) == dim
                assert np.array_equal(m.solve()[0], want)
            m.close()
            if not met:
                break
            at += 1
        assert at >= 4


@pytest.mark.parametrize("waves", [1, 2])
@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(solve_kernel=2)])
def test_autotuner(kw, waves):
    """The local stage after a refused autotuner is the one before it, also of waves whose
    task lists the autotuner had not reached."""
    from paper_2211_13893_gb300 import MSGFEM, plan
    cfg = get_config("t2")
    ang = element_angles(cfg)
    kw = dict(kw, wave_mb=0.0 if waves == 1 else 1.01 * plan(cfg, kw.get("precision", 0))["pool_mb"] / waves)
    mem = Refusing()
    at = 0
    while True:
        m = MSGFEM.from_config(cfg, ang, seed=5, allocator=(mem.alloc, mem.free), **kw)
        lam = m.local_spaces(cfg.n_loc).copy()
        before = m.profile()
        assert before["waves"] >= waves
        met = mem.refuse(at, lambda: m.autotune(reps=1))
        if not met:
            break
        assert m.profile()["launches"] == before["launches"]
        assert np.array_equal(m.local_spaces(cfg.n_loc), lam), at
        after = m.profile()
        assert after["factor_flops"] == before["factor_flops"]
        assert after["factor_flops_executed"] == before["factor_flops_executed"]
        m.coarse_assemble()
        u, _ = m.solve()
        assert np.all(np.isfinite(u))
        m.close()
        at = at + 1 if at < 6 else 2 * at
    m.close()
    assert at >= 6


def test_update_angles():
    """Angles that need more element matrices than the earlier ones (per element instead of
    per ply): refused, the earlier angles stay, also for the solution that is there."""
    from paper_2211_13893_gb300 import MSGFEM
    cfg = get_config("t2")
    ang = element_angles(cfg)
    other = ang + np.random.default_rng(2).standard_normal(ang.shape)
    mem = Refusing()
    ref = MSGFEM.from_config(cfg, other, seed=5)
    want = ref.local_spaces(cfg.n_loc).copy()
    ref.close()
    u_ref = np.sin(np.arange(cfg.n_dof))
    at = 0
    while True:
        m = MSGFEM.from_config(cfg, ang, seed=5, allocator=(mem.alloc, mem.free))
        lam = m.local_spaces(cfg.n_loc).copy()
        m.coarse_assemble()
        _, err = m.solve(u_ref=u_ref)
        met = mem.refuse(at, lambda: m.update_angles(other))
        if met:
            assert m.solve(u_ref=u_ref)[1] == err
            assert np.array_equal(m.local_spaces(cfg.n_loc), lam)
            m.update_angles(other)
        assert np.array_equal(m.local_spaces(cfg.n_loc), want)
        m.close()
        if not met:
            break
        at += 1
    assert at >= 2


@pytest.mark.parametrize("kw", [dict(), dict(precision=1)])
def test_schwarz_solve(kw):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = get_config("t2")
    cfg = replace(cfg, oversampling=cfg.overlap)
    ang = element_angles(cfg)
    ref = MSGFEM.from_config(cfg, ang, seed=5, **kw)
    want, _ = ref.schwarz_solve()
    ref.close()
    mem = Refusing()
    at = 0
    while True:
        m = MSGFEM.from_config(cfg, ang, seed=5, allocator=(mem.alloc, mem.free), **kw)
        met = mem.refuse(at, m.schwarz_solve)
        assert np.array_equal(m.schwarz_solve()[0], want)
        m.close()
        if not met:
            break
        at += 1
    assert at >= 2


def test_start_block():
    import torch
    from paper_2211_13893_gb300 import MSGFEM
    cfg = get_config("t2")
    ang = element_angles(cfg)
    mem = Refusing()
    at, want = 0, None
    while True:
        m = MSGFEM.from_config(cfg, ang, seed=5, allocator=(mem.alloc, mem.free))
        m.local_spaces(cfg.n_loc)
        n2, _ = m.warm_sizes(m.N - 1, cfg.n_loc)
        block = torch.zeros((n2, 8), dtype=torch.float32, device="cuda")
        met = mem.refuse(at, lambda: m.warm_targets(m.N - 1, block, 8))
        m.warm_targets(m.N - 1, block, 8)
        m.set_start_block(m.N - 1, block, 8, 8)
        got = (block.cpu().numpy(), m.local_spaces(cfg.n_loc).copy())
        m.close()
        want = got if want is None else want
        assert np.any(got[0] != 0.0) and all(np.array_equal(a, b) for a, b in zip(got, want))
        if not met:
            break
        at += 1
    assert at >= 3


def test_going_over_to_the_block_cholesky():
    """The task lists that a local stage builds when its layers are too ill-conditioned for
    the inverse form (fibres 25,000 times as stiff as the matrix, on cubes)."""
    from paper_2211_13893_gb300 import MSGFEM
    E = (1.62e5, 6.48, 6.48, 2.0, 2.0, 2.0, 0.3, 0.3, 0.3)
    cfg = replace(get_config("t2"), hx=0.25, hy=0.25, material=E, n_loc=7)
    ang = element_angles(cfg)
    mem = Refusing()
    ref = MSGFEM.from_config(cfg, ang, seed=5, precision=1)
    want = ref.local_spaces(cfg.n_loc, allow_noconv=True).copy()
    flops = ref.profile()
    assert flops["factor_flops"] != flops["factor_flops_inverse"]     # it did go over
    ref.close()
    at = 0
    while True:
        m = MSGFEM.from_config(cfg, ang, seed=5, precision=1, allocator=(mem.alloc, mem.free))
        met = mem.refuse(at, lambda: m.local_spaces(cfg.n_loc, allow_noconv=True))
        assert np.array_equal(m.local_spaces(cfg.n_loc, allow_noconv=True), want)
        m.close()
        if not met:
            break
        at += 1
    assert at >= 5
