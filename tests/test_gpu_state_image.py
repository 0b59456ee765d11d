"""State images of lattices whose planes are several MB, for every storage type
(the 2-, 4- and 8-byte forms of the split into planes), at an odd side: a run
saved and restored into a fresh handle continues bit for bit."""
import pytest

from helpers import gpu_lattice
from paper_2410_23802_gb300 import workloads as W
from test_gpu_checkpoint import _assert_same, _snapshot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,side", [("fp16", 1261), ("bf16", 1261), ("fp32", 1261), ("fp64", 1261),
                                            ("fp32", 1951)])  # (the last: planes copied one by one)
def test_large_image_resumes_bit_for_bit(precision, side):
    case = W.cavity(side=side, n=40, seed=17)
    with gpu_lattice(case, precision=precision) as a:
        a.step(9)
        img = a.save_state()
        a.step(8)
        ref = _snapshot(a)
    with gpu_lattice(case, precision=precision) as b:
        b.load_state(img)
        b.step(8)
        _assert_same(_snapshot(b), ref)


@pytest.mark.parametrize("precision", ["fp16", "fp32", "fp64"])
@pytest.mark.parametrize("before", [0, 9])
def test_saving_leaves_the_run_as_it_is(precision, before):
    """Fields and the further run are the same whether an image was taken or not
    (its scratch is a handle's own buffers)."""
    case = W.cavity(side=203, n=9, seed=18)
    with gpu_lattice(case, precision=precision) as a:
        a.step(before)
        ref = [_snapshot(a)]
        a.step(8)
        ref.append(_snapshot(a))
    with gpu_lattice(case, precision=precision) as b:
        b.step(before)
        b.save_state()
        _assert_same(_snapshot(b), ref[0])
        img = b.save_state()
        _assert_same(_snapshot(b), ref[0])
        b.step(8)
        _assert_same(_snapshot(b), ref[1])
    with gpu_lattice(case, precision=precision) as c:
        c.load_state(img)
        c.step(8)
        _assert_same(_snapshot(c), ref[1])
