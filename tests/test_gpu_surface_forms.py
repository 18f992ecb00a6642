"""The scalar field's kernel forms (2 x 2 x 2, 2 x 2 and 2 corners per warp) at the lines between
them and on corner counts that leave groups and tiles part empty, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2404_01931_gb300 import flip as F
from paper_2404_01931_gb300 import scenes as S

from parity_util import matched
from test_gpu_surface import _gpu_mesh, _sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,ratio", [
    ((31, 18, 7), 1 / 24, 2.0),      # R = 2 h: corners a bin apart, 2 x 2
    ((32, 17, 8), 1 / 24, 1.9),      # just past the line, pairs
    ((9, 5, 6), 1 / 8, 0.7),         # balls that do not meet, pairs
    ((60, 55, 3), 1 / 72, 6.5),      # corners far closer than a bin, 2 x 2
    ((1, 1, 1), 1 / 2, 2.0),         # eight corners
    ((30, 25, 18), 1 / 30, 2.0),     # corners on bin faces, rounded to either side: 2 x 2
    ((23, 17, 12), 1 / 23, 2.0),
    ((55, 50, 45), 1 / 55, 2.0),     # ... and 2 x 2 x 2
])
def test_sdf_forms_match_the_oracle(n, h, ratio):
    sc = S.random_velocities(S.water_drop(24, centre=(0.4, 0.45, 0.3), radius=0.25), 0.1, 3)
    sp = F.FlipSurfaceParams()
    for a in range(3):
        sp.n[a] = n[a]
        sp.origin[a] = 0.0 if round(n[0] * h, 6) == 1.0 else (-0.01, 0.003, 0.02)[a]
    sp.h, sp.search_radius = h, ratio * h
    sp.radius, sp.iso = 0.25 * sp.search_radius, 0.0
    with F.Simulation(matched(24)[1], *sc.arrays()) as sim, F.Surface(sp) as s:
        s.sdf(sim)
        phi = s.read(F.SURF_FIELD).astype(np.float64)
    ref = O.sdf(sc.x, sc.y, sc.z, tuple(sp.n), tuple(sp.origin), sp.h, sp.radius,
                sp.search_radius)
    # FP32 kernel sums: relative rounding ~1e-6 of the lengths involved (R), the bar of
    # test_gpu_surface.py
    assert np.abs(phi - ref).max() <= 2e-5 * sp.search_radius


@pytest.mark.parametrize("n", [
    (1, 1, 1024),      # rows of two corners and planes of four: many carries a step
    (1024, 1, 1),      # the longest rows, four steps and a bit
    (15, 15, 40),      # planes of 256 corners: no remainder
    (30, 33, 5),       # planes of four steps and a bit
])
def test_mesh_walks_any_grid_shape(n):
    """Dense crossings, so that the warps' lists are full; topology as the oracle's (the
    normals' rounding grows with the grid's length over a cell and is bounded elsewhere)."""
    phi = S.corner_field_random(n, 4, closed=False)
    sp = _sp(n, 0.2)
    ref = O.marching_cubes(phi.astype(np.float64), tuple(sp.origin), sp.h, 0.0)
    nv, nt, got = _gpu_mesh(sp, phi)
    assert nv > 1000 and nt > 1000
    assert np.array_equal(got["e"], ref.vertex_edge) and np.array_equal(got["t"], ref.triangles)


@pytest.mark.parametrize("n", [10, 24, 48, 101])
@pytest.mark.parametrize("ratio", [2.0, 1.9])  # 2 x 2 x 1 corners (n < 48) or 2 x 2 x 2; pairs
@pytest.mark.parametrize("dirs", [((0, 1), (0, -1)), ((1, 1), (1, -1)), ((2, 1), (2, -1)),
                                  ((0, 1), (1, 1)), ((2, -1), (1, 1)),
                                  tuple((a, s) for a in range(3) for s in (-1, 1))])
def test_particles_at_exactly_the_search_radius_do_not_count(n, ratio, dirs):
    """Corner 0 lies at (R, R, R), the particles R from it on its axes: the coordinates 0, R
    and 2 R and their differences are exact, so no particle is closer than R."""
    R = np.float32(2 / n)
    pos = np.full((3, len(dirs)), R, np.float32)
    for q, (a, s) in enumerate(dirs):
        pos[a, q] = R + np.float32(s) * R
    sp = _sp((n, n, n), float(R) / ratio, origin=(float(R),) * 3, r=0.25 * float(R), R=float(R))
    zero = np.zeros(len(dirs), np.float32)
    with F.Simulation(matched(n)[1], *pos, zero, zero, zero) as sim, F.Surface(sp) as s:
        s.sdf(sim)
        phi = s.read(F.SURF_FIELD).reshape(n + 1, n + 1, n + 1)
    assert phi[0, 0, 0] == R - np.float32(0.25) * R


@pytest.mark.parametrize("n,h,ratio", [
    ((60, 52, 57), 1 / 50, 1.9),     # corners over a bin apart, many and few groups
    ((26, 20, 23), 1 / 50, 1.6),
    ((56, 49, 51), 1 / 50, 1.02),    # just inside the line: seven bin rows each way
    ((56, 49, 51), 1 / 50, 1.0),     # past it: four corners along x
    ((14, 9, 11), 1 / 12, 0.7),      # ... with balls that do not meet, a row's rest of three
])
def test_sdf_forms_match_the_oracle_within_each_corners_conditioning(n, h, ratio):
    check_sdf(n, h, ratio)


@pytest.mark.parametrize("n,h,ratio", [
    ((47, 59, 51), 1 / 60, 3.1),     # bins wider than a cell, corners between bin faces
    ((63, 50, 55), 1 / 64, 2.7),
    ((52, 50, 53), 1 / 55, 6.5),     # corners far closer than a bin
])
def test_sdf_of_many_corners_matches_the_oracle_at_other_radii(n, h, ratio):
    """Grids of 15 thousand groups and more, which take 2 x 2 x 2 corners a warp."""
    check_sdf(n, h, ratio)


@pytest.mark.parametrize("n,h,ratio", [
    ((20, 14, 16), 1 / 8, 8.0),      # balls that meet a few rows of a thousand particles
    ((12, 9, 10), 1 / 8, 4.0),
    ((10, 11, 9), 1 / 9, 2.0),       # rows longer and shorter than the line
    ((21, 20, 19), 1 / 18, 2.0),
    ((11, 12, 9), 1 / 8, 0.9),       # four corners along x
])
def test_sdf_of_grids_coarse_against_the_particles(n, h, ratio):
    """Each lane adds up to 7 thousand / 32 terms before the tree, within the bar; corners
    beyond it are held to their conditioning, however many of so few there are."""
    check_sdf(n, h, ratio, most=1.0)


@pytest.mark.parametrize("n", [(42, 41, 40), (74, 73, 75), (92, 91, 93), (110, 109, 111)])
def test_mesh_passes_over_lists_shared_by_ctas(n):
    """37, 206, 393 and 668 tiles: eight, four, two and one CTAs a tile on 152 SMs."""
    phi = S.corner_field_random(n, 6)
    sp = _sp(n, 0.2)
    ref = O.marching_cubes(phi.astype(np.float64), tuple(sp.origin), sp.h, 0.0)
    nv, nt, got = _gpu_mesh(sp, phi)
    assert np.array_equal(got["e"], ref.vertex_edge) and np.array_equal(got["t"], ref.triangles)
    # the bar of test_gpu_surface.py
    scale = max(abs(o) for o in sp.origin) + sp.h * max(n)
    assert np.abs(got["v"] - ref.vertices).max() <= 4e-7 * scale + 1e-6 * sp.h


def check_sdf(n, h, ratio, most=1e-4):
    """The bar of the tests above, and beyond it what the roundings of t = 1 - d^2 / R^2 can
    change at a corner: phi + r = |sum k e| / sum k, k = t^3, moves by at most
    2 R sum dk / sum k (|e - mean| <= 2 R), dk = (t + eps)^3 - t^3.  eps: five roundings to
    within 2^-25 of t's terms (below 2^-22 in all), and the corner's coordinates, within 2^-23
    of their size.  Only a corner with no particle well inside its ball needs it."""
    sc = S.random_velocities(S.water_drop(24, centre=(0.4, 0.45, 0.3), radius=0.25), 0.1, 3)
    sp = F.FlipSurfaceParams()
    for a in range(3):
        sp.n[a] = n[a]
        sp.origin[a] = (-0.01, 0.003, 0.02)[a]
    sp.h, sp.search_radius = h, ratio * h
    sp.radius, sp.iso = 0.25 * sp.search_radius, 0.0
    R = sp.search_radius
    with F.Simulation(matched(24)[1], *sc.arrays()) as sim, F.Surface(sp) as s:
        s.sdf(sim)
        phi = s.read(F.SURF_FIELD).astype(np.float64).reshape(n[2] + 1, n[1] + 1, n[0] + 1)
    ref = O.sdf(sc.x, sc.y, sc.z, tuple(sp.n), tuple(sp.origin), sp.h, sp.radius, R)
    assert (ref < 0).any() and (ref == R - sp.radius).any()
    assert phi.min() >= -sp.radius * (1 + 1e-6) and phi.max() <= (R - sp.radius) * (1 + 1e-6)
    err = np.abs(phi - ref)
    far = np.argwhere(err > 2e-5 * R)
    assert len(far) <= most * err.size
    eps = 2.0 ** -22 + 2 * 2.0 ** -23 * (0.02 + max(n) * h) / R
    p = np.stack([sc.x, sc.y, sc.z]).astype(np.float64)
    for k, j, i in far:
        e = p - (np.array([i, j, k]) * h + np.array(sp.origin))[:, None]
        t = 1 - (e * e).sum(0) / R ** 2
        t = t[t > -eps].clip(0)
        dk = ((t + eps) ** 3 - t ** 3).sum() / max((t ** 3).sum(), 1e-300)
        assert err[k, j, i] <= 2e-5 * R + 2 * R * dk, (i, j, k)
