"""The warp sums of the FP32 exchange terms at terms that they could not hold: a
disk of R = 2100 cells that spins at Omega R^2 = 2205 per cell at its rim.  32
such terms of one row pass 2^31 in the sum's upper part (units of 2^-15), so
those warps have to add their lanes one by one (they do above 2^10).  The
torque after one step against the FP64 kernel's, whose lanes always add one by
one: within 1e-6 of its size Omega pi R^4 / 2 (terms of one sign, a few FP32
roundings of 6e-8 each).  That is 1.5e10, beyond the accumulators' 2^23, so both
report it modulo 2^24; a wrapped warp sum is off by 2^17, and the number of warps
that would wrap is no multiple of 2^7 here."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_terms_beyond_the_warp_sums_range():
    from paper_2410_23802_gb300 import vlb as V
    n, R, omega = 4260, 2100.0, 5e-4
    assert omega * R * R > 2048.0
    params = dict(nx=n, ny=n, tau_f=0.8, prandtl=0.7, rho_ratio=1.5, cv_ratio=2.0, k_ratio_default=3.0,
                  gravity=(0.0, -1e-5), beta=0.0, T_ref=1.0, T_fluid_init=1.0)
    torque = []
    for precision in (V.VLB_FP64, V.VLB_FP32):
        p = V.vlb_params_default(precision=precision, max_particles=1, **params)
        with V.Lattice(p) as lat:
            lat.add_particles([[n / 2 + 0.37, n / 2 - 0.61]], [R], [0.0], omega=[omega])
            lat.step(1)
            torque.append(lat.particles()["torque"][0])
    off = (torque[1] - torque[0] + 2.0 ** 23) % 2.0 ** 24 - 2.0 ** 23
    assert abs(off) < 1e-6 * omega * math.pi * R ** 4 / 2.0
    assert all(np.isfinite(torque))
