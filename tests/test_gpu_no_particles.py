"""Lattices without particles: their lattice kernels follow one another with no
particle kernel between.  A cavity heated from one side, stepped in one call and
in batched calls, equals the same run waited for after every step, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lattice(precision, side):
    from paper_2410_23802_gb300 import vlb as V
    return V.Lattice(V.vlb_params_default(
        nx=side, ny=side + 3, precision=precision, max_particles=0, gravity=(0.0, -1e-5), beta=5.0,
        T_ref=0.5, T_fluid_init=0.5, thermal_wall=(1, 1, 0, 0), wall_T=(0.0, 1.0, 0.0, 0.0)))


@pytest.mark.parametrize("precision", [0, 1, 2, 3])  # FP64, FP32, FP16, BF16 storage
@pytest.mark.parametrize("side", [33, 1501])
def test_steps_without_particles_equal_synchronised_ones(precision, side):
    from paper_2410_23802_gb300 import vlb as V
    steps = 60
    with _lattice(precision, side) as lat:
        for _ in range(steps):
            lat.step(1)
            V.vlb_synchronize(lat.h)
        want = lat.fields()
    assert float(np.abs(want["uy"]).max()) > 0.0
    with _lattice(precision, side) as lat:
        lat.step(steps)
        got = lat.fields()
    with _lattice(precision, side) as lat, _lattice(1, 65) as other:
        V.vlb_step_batch([other.h, lat.h], steps)
        batched = lat.fields()
    for k in want:
        np.testing.assert_array_equal(got[k], want[k])
        np.testing.assert_array_equal(batched[k], want[k])
