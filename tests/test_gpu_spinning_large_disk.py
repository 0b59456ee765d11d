"""A spinning disk of R = 2100 cells: its cells' classes are decided in 64 bits
(R above 1448 cells), its band table has more rows than a CTA has threads, and
near the rim its torque terms w Omega r^2 pass 2^10, where the FP32 kernel adds
its lanes' exchange terms one by one instead of summing them in the warp.  The
FP32 kernels against the FP64 ones (which take none of these paths) after one
step: classes equal, fractions within 2e-7 (R + 1), the torque, whose terms all
have one sign and carry a few FP32 roundings of 6e-8 each, within 1e-6 of its
size Omega pi R^4 / 2.  (That is 7e9, beyond the accumulators' range of 2^23,
so both sides report it modulo 2^24; their difference is not affected.)"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_spinning_large_disk_fp32_matches_fp64():
    from paper_2410_23802_gb300 import vlb as V
    n, R, omega = 4260, 2100.0, 2.35e-4
    assert omega * R * R > 1024.0  # (the bound up to which the lanes are summed in the warp)
    params = dict(nx=n, ny=n, tau_f=0.8, prandtl=0.7, rho_ratio=1.5, cv_ratio=2.0, k_ratio_default=3.0,
                  gravity=(0.0, -1e-5), beta=0.0, T_ref=1.0, T_fluid_init=1.0)
    got = []
    for precision in (V.VLB_FP64, V.VLB_FP32):
        p = V.vlb_params_default(precision=precision, max_particles=1, **params)
        with V.Lattice(p) as lat:
            lat.add_particles([[n / 2 + 0.37, n / 2 - 0.61]], [R], [0.0], omega=[omega])
            lat.step(1)
            count, _, flag, fsp = V.vlb_get_solid_fraction(lat.h, n, n)
            got.append((count, flag[:, :, 0].copy(), fsp[:, :, 0].copy(), lat.particles()["torque"][0]))
            del flag, fsp
    (c64, k64, f64, t64), (c32, k32, f32, t32) = got
    np.testing.assert_array_equal(c32, c64)
    np.testing.assert_array_equal(k32, k64)
    np.testing.assert_allclose(f32, f64, rtol=0, atol=2e-7 * (R + 1.0))
    off = (t32 - t64 + 2.0 ** 23) % 2.0 ** 24 - 2.0 ** 23
    assert abs(off) < 1e-6 * omega * math.pi * R ** 4 / 2.0
