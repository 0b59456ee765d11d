"""The particle step's band tables and tile lists at the edges of its split:
one particle per CTA, several per CTA with a last CTA that is not full, boxes
of more rows than the threads that take them, slender and near-circular
ellipses.  After two steps the GPU's ownership of every cell is compared with
the oracle's raster of the GPU's own positions: owners and classes equal
(an ellipse's cell may differ where the oracle's FP64 decision lies within
1e-12 of its threshold: cos and sin of the angle come from two libraries),
fractions within 2e-7 (R + 1), the FP32 rounding of the centre relative to
the cell (about 6e-8 R per coordinate)."""
import math

import numpy as np
import pytest

from helpers import gpu_lattice
from oracle import vlbref as O
from paper_2410_23802_gb300 import workloads as W
from test_gpu_ellipse import _near_tie

pytestmark = pytest.mark.gpu


def _params(nx, ny):
    return dict(nx=nx, ny=ny, tau_f=0.8, prandtl=0.7, rho_ratio=1.5, cv_ratio=2.0, k_ratio_default=3.0,
                gravity=(0.0, -1e-5), beta=0.0, T_ref=1.0, T_fluid_init=1.0)


def _grid(n, seed, big=0.0):
    """n disks of radius 1 to 2.2 on a jittered grid of pitch 7, one of radius `big` above them."""
    rng = W.SplitMix64(seed)
    side = math.ceil(math.sqrt(n))
    xs, ys, rs = [], [], []
    for k in range(n):
        xs.append(7.0 * (k % side) + 3.5 + rng.uniform(-0.6, 0.6))
        ys.append(7.0 * (k // side) + 3.5 + rng.uniform(-0.6, 0.6))
        rs.append(rng.uniform(1.0, 2.2))
    nx, ny = 7 * side + 5, 7 * side + 3
    if big:
        nx, ny = max(nx, int(2 * big) + 9), ny + int(2 * big) + 9
        xs[n // 2], ys[n // 2], rs[n // 2] = 0.5 * nx + 0.13, ny - big - 3.7, big
    return nx, ny, xs, ys, rs


# the sizes around a change of the particles per CTA (608 CTAs), its largest
# value with a last CTA of one, and boxes of 25, 131 and 247 rows
@pytest.mark.parametrize("n,big", [(1, 10.3), (7, 121.4), (608, 0.0), (609, 0.0), (700, 62.7), (1217, 0.0), (4873, 0.0)])
def test_disk_tables_match_oracle(n, big):
    from paper_2410_23802_gb300 import vlb as V
    nx, ny, xs, ys, rs = _grid(n, 40 + n, big)
    case = W.Case("grid", _params(nx, ny), xs, ys, rs, [0.0] * n)
    rng = np.random.default_rng(n)
    p = V.vlb_params_default(precision=V.VLB_FP32, max_particles=n, **case.params)
    with V.Lattice(p) as lat:
        lat.add_particles(np.column_stack([xs, ys]), rs, case.T0, uv=rng.uniform(-0.02, 0.02, (n, 2)))
        lat.step(2)
        count, owner, flag, fsp = V.vlb_get_solid_fraction(lat.h, nx, ny)
        at = lat.particles()
    ras = O.rasterise(nx, ny, at["x"], at["y"], rs)
    np.testing.assert_array_equal(count, ras.count)
    np.testing.assert_array_equal(owner, ras.owner)
    np.testing.assert_array_equal(flag, ras.flag)
    np.testing.assert_allclose(fsp, ras.fsp, rtol=0, atol=2e-7 * (max(rs) + 1.0))


@pytest.mark.parametrize("a,b", [(40.0, 1.0), (13.0, 12.9), (60.0, 21.0), (5.0, 1.5)])
def test_ellipse_tables_match_oracle(a, b):
    from paper_2410_23802_gb300 import vlb as V
    nx, ny = 150, 290
    xs, ys, th = [74.3, 75.6], [70.2, 215.4], [0.77, -2.1]
    case = W.Case("ellipses", _params(nx, ny), xs + [20.25], ys + [143.0], [a, a, 3.0], [0.0] * 3,
                  semi_minor=[b, b, 3.0], theta0=th + [0.0])
    with gpu_lattice(case) as lat:
        lat.step(2)
        count, owner, flag, fsp = V.vlb_get_solid_fraction(lat.h, nx, ny)
        at = lat.particles()
    ras = O.rasterise_shapes(nx, ny, at["x"], at["y"], [a, a, 3.0], [b, b, 3.0], at["theta"])
    bad = np.argwhere((count != ras.count) | (owner != ras.owner).any(axis=2) | (flag != ras.flag).any(axis=2))
    for j, i in bad:
        assert any(_near_tie(i, j, at["x"][p], at["y"][p], a, b, at["theta"][p]) for p in range(2)), (i, j)
    assert len(bad) <= 2
    ok = np.ones((ny, nx), dtype=bool)
    ok[tuple(bad.T)] = False
    np.testing.assert_allclose(fsp[ok], ras.fsp[ok], rtol=0, atol=2e-7 * (a + 1.0))
