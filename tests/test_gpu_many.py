"""More subdomains than half of a grid dimension: 33,000 in one handle, every instance of
the same beam, so every instance has the first one's eigenvalues (1e-8, mixed 1e-5: the
start blocks differ).  And the storage per subdomain besides the pool: the working blocks
of its 192 rows, 1.2 MB, with nothing of that order added per subdomain of a large batch."""
from dataclasses import replace

import numpy as np
import pytest

from workloads import element_angles, get_config

pytestmark = pytest.mark.gpu

# (48 interface DoFs and four pairs: the Krylov basis holds them before it has exhausted the interface)
TINY = dict(NX=4, NY=3, NZ=3, sx=2, sy=1, overlap=1, oversampling=1, n_loc=4)


class _Bump:
    """Blocks cut off one after the other from a single buffer."""

    def __init__(self, nbytes):
        import torch
        self.buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        self.at, self.end, self.sizes = self.buf.data_ptr(), self.buf.data_ptr() + nbytes, []
        self.at += -self.at % 256

    def alloc(self, n):
        p, self.at = self.at, self.at + n + -n % 256
        self.sizes.append(n)
        return p if self.at <= self.end else None

    def free(self, p, n):
        pass


@pytest.mark.parametrize("precision", [0, 1])
def test_more_subdomains_than_half_a_grid(precision):
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="tiny", **TINY)
    inst = 16500
    ang = np.tile(element_angles(cfg).reshape(-1), inst)
    pool = _Bump(96 << 30)
    m = MSGFEM.from_config(cfg, ang, seed=7, precision=precision, instances=inst, wave_mb=24 * 1024.0,
                           allocator=(pool.alloc, pool.free))
    assert m.N == 2 * inst
    lam = np.array(m.local_spaces(cfg.n_loc)).reshape(inst, 2, cfg.n_loc)
    m.close()
    one = MSGFEM.from_config(cfg, element_angles(cfg), seed=7, precision=precision)
    ref = one.local_spaces(cfg.n_loc)
    one.close()
    scale = np.maximum(np.abs(ref).max(axis=1, keepdims=True), 1.0)
    assert (np.abs(lam - ref[None]) / scale[None]).max() <= (1e-8 if precision == 0 else 1e-5)


def test_storage_per_subdomain():
    from paper_2211_13893_gb300 import MSGFEM
    cfg = replace(get_config("t3"), name="tiny", **TINY)
    total = []
    for inst in (700, 1400):
        pool = _Bump(10 << 30)
        ang = np.tile(element_angles(cfg).reshape(-1), inst)
        m = MSGFEM.from_config(cfg, ang, seed=7, instances=inst, allocator=(pool.alloc, pool.free))
        pool_mb = m.profile()["pool_mb"]
        total.append(sum(pool.sizes) - pool_mb * 1048576)
        m.close()
    assert (total[1] - total[0]) / 1400 <= 1.4e6
