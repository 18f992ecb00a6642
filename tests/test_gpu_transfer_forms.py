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


@pytest.mark.parametrize("n", [(8, 8, 8), (24, 8, 8), (33, 8, 8), (64, 8, 9), (168, 168, 160)])
def test_binning_keeps_every_particle(n):
    """1, 3, 5, 16 and 8820 bricks: below, across and past the brick scan's vectors and chunks."""
    rng = np.random.default_rng(11)
    dx = np.float32(1 / max(n))
    pos = [(rng.uniform(0.01, n[a] - 0.01, 3001) * dx).astype(np.float32) for a in range(3)]
    vel = [rng.uniform(-0.5, 0.5, 3001).astype(np.float32) for _ in range(3)]
    op, fp = matched(n, cg_tol=1e-2)
    with F.Simulation(fp, *pos, *vel) as sim:
        rc, st = sim.step(2, stats=True)
        ids = np.asarray(sim.read(F.PID))
        typ = np.asarray(sim.read(F.CELL_TYPE)).reshape(n[2], n[1], n[0])
    assert rc == F.FLIP_OK and np.array_equal(np.sort(ids), np.arange(3001))
    assert st.n_fluid_cells == np.count_nonzero(typ)


@pytest.mark.parametrize("cell", [2, 100, 250])
def test_faces_that_only_vanishing_weights_reach(cell):
    """Two particles a few roundings of x/dx past a face: the next face's velocity is the ratio
    of FP32 weights, (f1 - f2) / (f1 + f2), within the sums' roundings."""
    n, inv = (256, 8, 8), np.float32(256)
    ulp = np.spacing(np.float32(cell)) / np.float32(256)
    x = np.float32(cell / 256) + np.array([3, 8], np.float32) * ulp
    c = np.full(2, 3.5 / 256, np.float32)
    u, o = np.array([1, -1], np.float32), np.zeros(2, np.float32)
    op, fp = matched(n)
    with F.Simulation(fp, x, c, c, u, o, o) as sim:
        sim.step(1)
        uo = np.asarray(sim.read(F.U_OLD)).reshape(8, 8, 257)[3, 3]
    f = x * inv - np.float32(cell)
    assert (f > 0).all()
    assert abs(uo[cell + 1] - (f[0] - f[1]) / (f[0] + f[1])) <= 8 * 2.0 ** -24
    assert abs(uo[cell]) <= 1e-4
