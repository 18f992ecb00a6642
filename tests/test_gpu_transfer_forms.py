"""The particle-grid transfers at launch widths that make a CTA take several bricks, one
brick or a part of one, against the oracle's step."""
import numpy as np
import pytest

import oracle as O
from paper_2404_01931_gb300 import flip as F
from paper_2404_01931_gb300 import scenes as S
from parity_util import face_floor, matched, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas", [1, 2, 8, 64])
@pytest.mark.parametrize("n,hi", [
    ((45, 41, 43), (1.0, 0.85, 1.0)),  # 180 bricks: rounds of bricks, one each, and parts
    ((9, 70, 8), (1.0, 0.5, 1.0)),     # a cell past a brick, walls on both sides
])
def test_transfers_match_the_oracle_at_any_launch_width(n, hi, ctas):
    sc = S.random_velocities(S.box(n, (0.0, 0.0, 0.0), hi, seed=8), 0.5, 9)
    op, fp = matched(n, cg_tol=1e-7)
    ref = O.step(op, *sc.arrays())
    with F.Simulation(fp, *sc.arrays()) as sim:
        sim.set_transfer_ctas(ctas, ctas)
        sim.step(1)
        uo = [sim.read(f) for f in (F.U_OLD, F.V_OLD, F.W_OLD)]
        got = np.stack(sim.particles()).astype(np.float64)
    for d in range(3):
        assert rel_l2(uo[d], ref.u_old[d], face_floor(n)) <= 1e-5, d
    dx = 1 / max(n)
    assert np.abs(got[:3] - np.stack([ref.x, ref.y, ref.z])).max() <= 1e-4 * dx
    vel = np.stack([ref.u, ref.v, ref.w])
    assert rel_l2(got[3:], vel, 9.81 / 240 * np.sqrt(vel.size)) <= 1e-5
