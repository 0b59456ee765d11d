"""The audit's total mass against the sum of the populations themselves, taken
from a state image and added up exactly (fsum).  The audit adds in FP64, in
sums of at most about 700 terms one after the other (9 populations of a cell,
the cells of a thread, the threads of a block, 608 blocks), each of which rounds
within half a unit of the running sum: 700 x 1.2e-16 of the total."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_mass_is_the_sum_of_the_populations(precision):
    from paper_2410_23802_gb300 import vlb as V
    prm = dict(nx=67, ny=71, tau_f=0.8, prandtl=0.7, rho_ratio=1.5, cv_ratio=2.0, gravity=(0.0, -1e-5), beta=0.0,
               T_ref=1.0, T_fluid_init=1.0)
    p = V.vlb_params_default(precision=V.VLB_FP64 if precision == "fp64" else V.VLB_FP32, max_particles=2, **prm)
    with V.Lattice(p) as lat:
        # (fast disks, so that the populations are some 1e-2 away from those at rest)
        lat.add_particles([[20.3, 40.1], [45.7, 30.2]], [9.0, 10.0], [0.0, 0.0], uv=[0.2, 0.1, -0.15, 0.2])
        lat.step(20)
        mass = lat.audit()[0]
        img = np.frombuffer(bytes(lat.save_state()), dtype=np.uint8)
    header = int(img[12:16].view(np.uint32)[0])
    nx, ny, pitch = (int(v) for v in img[16:28].view(np.int32))
    cur = int(img[48:52].view(np.int32)[0])
    pop_bytes, s_bytes = (int(v) for v in img[72:88].view(np.uint64))
    at = header + cur * (pop_bytes + s_bytes)
    f = img[at:at + pop_bytes].view(np.float64 if precision == "fp64" else np.float32)
    f = f.reshape(18, ny, pitch)[:9, :, :nx].astype(np.float64)
    want = math.fsum([float(nx * ny), *f.ravel().tolist()])
    assert abs(mass - want) <= 700 * 1.2e-16 * want, (mass, want)
