"""The standalone solve's forms (up to 2 and 4 cells per thread in registers, or in memory)
on cell counts around their lines, by the true residual of what they return."""
import numpy as np
import pytest

from paper_2404_01931_gb300 import flip as F
from paper_2404_01931_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def apply_a(fluid, p, scale):
    """scale times the 7-point operator on fluid cells, p = 0 in air, walls dropped (FP64)."""
    cnt = np.full(p.shape, 6.0)
    for a in range(3):
        cnt = np.moveaxis(cnt, a, 0)
        cnt[0] -= 1
        cnt[-1] -= 1
        cnt = np.moveaxis(cnt, 0, a)
    out = cnt * p
    for a in range(3):
        q, o = np.moveaxis(p, a, 0), np.moveaxis(out, a, 0)
        o[:-1] -= q[1:]
        o[1:] -= q[:-1]
    return out * fluid * scale


@pytest.mark.parametrize("n,fill", [
    ((2, 2, 2), 0.6),
    ((9, 8, 17), 0.8),          # a few cells per CTA, none in most
    ((88, 64, 56), 0.97),       # two cells per thread
    ((96, 72, 88), 0.97),       # the third and fourth
    ((120, 104, 96), 0.97),     # past the line: in memory
])
def test_solve_pressure_residual(n, fill):
    mask = S.random_mask(n, fill, 5)
    rng = np.random.default_rng(3)
    b = rng.standard_normal(mask.shape).astype(np.float32)
    prm = F.default_params(*n)
    prm.cg_tol = 1e-4
    typ = torch.from_numpy(mask.astype(np.uint8).ravel()).cuda()
    p = torch.full((mask.size,), 7.0, device="cuda")
    rc, it, rel = F.flip_solve_pressure(prm, typ, torch.from_numpy(b.ravel()).cuda(), p)
    assert rc == F.FLIP_OK and rel <= prm.cg_tol
    p = p.cpu().numpy().reshape(mask.shape).astype(np.float64)
    assert not p[~mask].any()
    scale = prm.dt / (prm.rho * prm.dx ** 2)
    r = b * mask - apply_a(mask, p * mask, scale)
    bn = np.linalg.norm(b * mask)
    # the recursive residual's stop, plus the drift of `it` updates, each rounding A p by at
    # most 8 operations on values up to ||A|| ||p|| = 12 scale ||p||
    drift = it * 8 * 2.0 ** -24 * 12 * scale * np.linalg.norm(p) / bn
    assert np.linalg.norm(r) / bn <= prm.cg_tol + drift
