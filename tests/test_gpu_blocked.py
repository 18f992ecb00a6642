"""The multigrid levels that are smoothed blocked (csrc/k_mg.cu, block_pass and the levels
inside one CTA): shapes where a tile's edges, remainders or halo can go wrong, against the
oracle's V-cycle.  After one MG-PCG iteration (tolerance out of reach, cap 1 on both sides)
the pressure is a multiple of one V-cycle of the right-hand side, whose values are about
4 levels x 4 half-sweeps x 8 additions deep: 1e-5 relative allows each of those roundings
(6e-8) once.  Later iterates subtract nearly equal residuals and have no such bound."""
import numpy as np
import pytest

import oracle as O
from paper_2404_01931_gb300 import flip as F
from paper_2404_01931_gb300 import scenes as S

from parity_util import gpu_step, matched, rel_l2

pytestmark = pytest.mark.gpu


def masked_scene(n, fill, seed):
    """Random fluid cells (single cells, holes, cells at every wall) with random velocities."""
    mask = S.random_mask(n, fill, seed)
    sc = S.seed_mask(mask, 1.0 / max(n), 1, seed)
    return S.random_velocities(sc, 0.3, seed + 1)


@pytest.mark.parametrize("nu", [1, 2, 3])  # 3: deeper than the halo, pass by pass
@pytest.mark.parametrize("n,fill", [
    ((9, 17, 8), 0.5),       # one cell past a block, the smallest level above the CTA-local ones
    ((33, 7, 24), 0.9),      # an extent below a block
    ((40, 25, 31), 0.15),    # mostly isolated cells
    ((64, 48, 72), 0.97),    # several blocks a CTA group, holes in the interior
    ((16, 160, 16), 0.6),    # CTA-local levels longer than 16 cells
    ((144, 96, 80), 0.95),   # level 0 above the limit, the coarser levels blocked
])
def test_blocked_smoothing_matches_the_oracle(n, fill, nu):
    check_one_iteration(masked_scene(n, fill, 11), n, nu)


@pytest.mark.parametrize("n,fill", [
    ((16, 1040, 512), 0.02),  # more segment groups than a CTA scans by itself
    ((5, 6, 7), 0.7),         # two levels, both in one CTA but the first
    ((3, 4, 2), 0.6),         # one level
    ((130, 40, 24), 0.9),     # three segments a row, the last with two cells
    ((67, 121, 96), 0.9),     # four slots a lane with rows that end at three of four
    ((133, 90, 60), 0.6),     # ... and at one, a third segment of five cells
])
def test_level_set_up_matches_the_oracle(n, fill):
    """Level flags, segment slices and codes: a wrong one changes the V-cycle at O(1)."""
    check_one_iteration(masked_scene(n, fill, 7), n, 2)


def check_one_iteration(sc, n, nu):
    """One iteration on the step's own cell types and right-hand side, so that the solve alone
    is compared (at faces that only vanishing weights reach, P2G's FP32 and FP64 velocities,
    and with them b, differ at O(1))."""
    op, fp = matched(n, cg_tol=1e-30, cg_max_iter=1, mg_smooth=nu)
    with pytest.warns(RuntimeWarning):
        got = gpu_step(fp, sc.arrays())
    assert got["rc"] == F.FLIP_E_NOT_CONVERGED and got["stats"].cg_iterations == 1
    typ = got["type"].reshape(n[2], n[1], n[0])
    ref, _, _ = O.pcg_mg(op, typ, got["rhs"].astype(np.float64).reshape(typ.shape), tol=1e-30,
                         max_iter=1, nu=nu)
    e = rel_l2(got["p"], ref)
    assert e <= 1e-5, f"pressure after one MG-PCG iteration: rel L2 {e:.3e}"


@pytest.mark.parametrize("n", [32, 48, 64, 96, 128])
@pytest.mark.parametrize("nu", [2, 3])
def test_solver_memory_per_cell(n, nu):
    """What a multigrid scene takes beyond a Jacobi one: 26 bytes a slot of level 0 (six FP32
    vectors and the codes), the coarser levels' 11 (a seventh of it), margins, less Jacobi's
    16; not the blocked smoothing's tables, which lie in memory that is idle in a solve."""
    fp = matched(n)[1]
    fp.mg_smooth = nu
    mg = F.flip_footprint_bytes(fp, n ** 3)
    fp.preconditioner = F.FLIP_PRECOND_JACOBI
    assert 0 < mg - F.flip_footprint_bytes(fp, n ** 3) <= 16 * n ** 3
