"""Cases of several storage types in one batched launch, with held particles
and without: each equals the case stepped alone, bit for bit."""
import dataclasses

import pytest

from helpers import gpu_lattice
from paper_2410_23802_gb300 import workloads as W
from test_gpu_channels_batch import _same, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("held", [0, 1, 2])
def test_mixed_storage_equals_alone(held):
    from paper_2410_23802_gb300 import vlb as V
    cases = [dataclasses.replace(c, fixed_T=[held] if held else None) for c in W.channels(n=3, seed=12, w_max=120)]
    cases.append(W.cavity(side=75, n=5, seed=4))
    if held:
        cases[3].fixed_T = [held, 0, held, 0, 0]
    kinds = ["fp16", "fp32", "bf16", "fp16"]
    lats = [gpu_lattice(c, precision=p) for c, p in zip(cases, kinds)]
    try:
        for k in (7, 20):
            V.vlb_step_batch([l.h for l in lats], k)
        got = [_state(l) for l in lats]
    finally:
        for l in lats:
            l.close()
    for c, p, g in zip(cases, kinds, got):
        with gpu_lattice(c, precision=p) as lat:
            lat.step(27)
            _same(g, _state(lat))
