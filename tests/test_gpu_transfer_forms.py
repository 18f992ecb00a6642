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


def _axis(x, inv, n):
    """Float32: (lower node, weight of the upper) on faces and on centres, as P2G weighs a node
    (csrc/flip_internal.cuh, axis_weights; x/dx is exact in 64 bits, so its floor is the cell)."""
    cell = np.clip(np.floor(x.astype(np.float64) * inv), 0, n - 1).astype(np.int64)
    g = x * np.float32(inv)
    face = np.clip(g - cell.astype(np.float32), np.float32(0), np.float32(1))
    c = np.clip(g - np.float32(0.5), np.float32(0), np.float32(n - 1))
    base = np.minimum(np.floor(c).astype(np.int64), n - 2)
    return (cell, face), (base, c - base.astype(np.float32))


def _fma(a, b, c):  # a b is exact in 64 bits
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(np.float32)


@pytest.mark.parametrize("advect", [F.FLIP_ADVECT_PARTICLE, F.FLIP_ADVECT_GRID])
@pytest.mark.parametrize("precision", [F.FLIP_PREC_FP32, F.FLIP_PREC_MIXED_IR])
@pytest.mark.parametrize("n,hi", [
    ((45, 41, 43), (1.0, 0.85, 1.0)),  # x/dx - 1/2 rounds in every binade but the first brick's
    ((9, 70, 8), (1.0, 0.5, 1.0)),
])
def test_g2p_interpolates_with_p2gs_weights(n, hi, precision, advect):
    """Velocities and positions bit for bit: the faces that next step's P2G reaches with
    vanishing weights turn a position's last bit into any change of their velocity."""
    sc = S.random_velocities(S.box(n, (0.0, 0.0, 0.0), hi, seed=8), 0.5, 9)
    op, fp = matched(n, cg_tol=1e-7, advect_source=advect)
    fp.precision = precision
    with F.Simulation(fp, *sc.arrays()) as sim:
        sim.step(1)
        uo = [np.asarray(sim.read(f)) for f in (F.U_OLD, F.V_OLD, F.W_OLD)]
        un = [np.asarray(sim.read(f)) for f in (F.U_NEW, F.V_NEW, F.W_NEW)]
        got = sim.particles()
    pos, vel = sc.arrays()[:3], sc.arrays()[3:]
    ax = [_axis(pos[a], max(n), n[a]) for a in range(3)]
    one, r, dt = np.float32(1), np.float32(fp.flip_ratio), np.float32(fp.dt)
    for d in range(3):
        dim = [n[a] + (a == d) for a in range(3)]
        w = [ax[a][0 if a == d else 1] for a in range(3)]
        U, dU = np.zeros_like(pos[0]), np.zeros_like(pos[0])
        for q in range(8):  # x fastest
            o = [(q >> a) & 1 for a in range(3)]
            k = [w[a][1] if o[a] else one - w[a][1] for a in range(3)]
            k = k[0] * (k[1] * k[2])
            # (a node past the grid has weight 0)
            i = [np.minimum(w[a][0] + o[a], dim[a] - 1) for a in range(3)]
            i = i[0] + dim[0] * (i[1] + dim[1] * i[2])
            U, dU = _fma(k, un[d][i], U), _fma(k, un[d][i] - uo[d][i], dU)
        v = r * (vel[d] + dU) + (one - r) * U
        x = _fma(np.full_like(v, dt), U if advect == F.FLIP_ADVECT_GRID else v, pos[d])
        x = np.clip(x, np.float32(fp.skin), np.float32(n[d] * fp.dx - fp.skin))
        assert np.array_equal(got[3 + d], v), d
        assert np.array_equal(got[d], x), d


def test_reseeding_drops_by_the_order_of_a_bricks_chunks():
    """In each of 512 bricks, eight cells with two chunks of 256 particles each move half a
    cell along every axis into one cell that may keep 512: those whose chunks come first."""
    n, m = 64, 512
    rng = np.random.default_rng(5)
    b, c = np.divmod(np.repeat(np.arange((n // 8) ** 3 * 8), m), 8)
    org = [8 * (b % 8), 8 * (b // 8 % 8), 8 * (b // 64)]
    # cell 3's upper half or cell 4's lower one
    pos = [((org[a] + np.where((c >> a) & 1, 4.05, 3.55) + 0.4 * rng.random(c.size)) / n)
           .astype(np.float32) for a in range(3)]
    vel = [np.full(c.size, 0.5 / n * 240, np.float32)] * 3
    op, fp = matched(n, gravity=(0.0, 0.0, 0.0))
    fp.ppc_min, fp.ppc_max = 1, m
    with F.Simulation(fp, *pos, *vel) as sim:
        sim.step(1)
        stored = np.asarray(sim.read(F.PID)).reshape(-1, 8 * m)  # a brick a row
        sim.step(1)
        kept = np.asarray(sim.read(F.PID)).reshape(-1, m)
    assert np.array_equal(np.sort(kept, axis=1), np.sort(stored[:, :m], axis=1))


def test_reseeding_step_ends_when_waits_give_up():
    """The warps of G2P meet after every chunk with reseeding; a limit of 1 ns on its copies'
    waits makes them leave in different places, and the step returns FLIP_E_TIMEOUT."""
    sc = S.dam_break(32)
    op, fp = matched(32)
    fp.ppc_min, fp.ppc_max = 3, 12
    with F.Simulation(fp, *sc.arrays()) as sim:
        sim.set_wait_timeout(1)
        with pytest.raises(F.FlipError) as ei:
            sim.step(1, stats=True)
        assert ei.value.code == F.FLIP_E_TIMEOUT
    with F.Simulation(fp, *sc.arrays()) as sim:  # the device is as usable as before
        assert sim.step(1, stats=True)[0] == F.FLIP_OK


@pytest.mark.parametrize("limit", [1, 500, 2000, 8000])
def test_steps_after_a_timed_out_one_stay_inside_the_particle_arrays(limit):
    """Limits (ns) that some of G2P's waits meet and others do not leave keys and ranks beside
    counts that do not hold them; the next binning drops what has no slot.  With the particles
    rewritten the handle steps to the oracle's result."""
    n = 40
    sc = S.dam_break(n)
    op, fp = matched(n)
    ref = O.step(op, *sc.arrays())
    with F.Simulation(fp, *sc.arrays()) as sim:
        sim.step(1)
        sim.set_wait_timeout(limit)
        for _ in range(3):
            try:
                sim.step(1, stats=True)
            except F.FlipError as e:
                assert e.code == F.FLIP_E_TIMEOUT
        sim.set_wait_timeout(0)
        ids = np.arange(sc.n_particles, dtype=np.int32)
        F.flip_write(sim.h, F.PID, ids)
        F.flip_write_particles(sim.h, *sc.arrays())
        rc, st = sim.step(1, stats=True)
        assert rc == F.FLIP_OK and st.n_fluid_cells == ref.n_fluid
        assert rel_l2(sim.read(F.PRESSURE_F64), ref.pressure) <= 1e-5
        got = np.stack(sim.particles()[:3]).astype(np.float64)
        assert np.abs(got - np.stack([ref.x, ref.y, ref.z])).max() * n <= 1e-4


@pytest.mark.parametrize("n,hi", [((45, 41, 43), (1.0, 0.85, 1.0)), ((70, 9, 33), (0.4, 1.0, 0.5))])
def test_p2g_face_by_face_weighted_by_the_sum_of_weights(n, hi):
    """Every face, with the bound that its sum of weights allows (a face that only vanishing
    weights reach has none of its own): x/dx and x/dx - 1/2 are rounded to within 2^-23 m cells
    (m the longest extent), so each of a face's k particles' weights, products of three, moves
    by at most 3 of that, and the numerator by (k + 4) roundings of its terms; a velocity is
    at most V from the face's mean of them times 2."""
    sc = S.random_velocities(S.box(n, (0.0, 0.0, 0.0), hi, seed=4), 0.5, 6)
    op, fp = matched(n)
    with F.Simulation(fp, *sc.arrays()) as sim:
        sim.step(1)
        uo = [np.asarray(sim.read(f), np.float64) for f in (F.U_OLD, F.V_OLD, F.W_OLD)]
    m, V = max(n), 0.5
    pos = [a.astype(np.float64) * m for a in sc.arrays()[:3]]
    for d in range(3):
        dim = [n[a] + (a == d) for a in range(3)]
        base, frac = [], []
        for a in range(3):
            g = np.clip(pos[a] - (0.0 if a == d else 0.5), 0.0, dim[a] - 1.0)
            b = np.minimum(np.floor(g), dim[a] - 2).astype(np.int64)
            base.append(b)
            frac.append(g - b)
        num, den, cnt = (np.zeros(dim[0] * dim[1] * dim[2]) for _ in range(3))
        vel = sc.arrays()[3 + d].astype(np.float64)
        for q in range(8):
            o = [(q >> a) & 1 for a in range(3)]
            w = np.prod([frac[a] if o[a] else 1 - frac[a] for a in range(3)], axis=0)
            i = (base[0] + o[0]) + dim[0] * ((base[1] + o[1]) + dim[1] * (base[2] + o[2]))
            np.add.at(num, i, w * vel)
            np.add.at(den, i, w)
            np.add.at(cnt, i, 1.0)
        far = den > 1e-30  # (below, FP32 weights may be 0)
        err = np.abs(uo[d][far] - num[far] / den[far])
        bound = 2 * V * (3 * cnt[far] * 2.0 ** -23 * m / den[far] + (cnt[far] + 4) * 2.0 ** -24)
        assert (err <= np.minimum(bound, 2 * V)).all(), d
        assert not uo[d][cnt == 0].any(), d
