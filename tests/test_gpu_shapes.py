"""Launch shapes: what the tuner reports of fields that choose nothing."""
import numpy as np
import pytest

import oracle
from synth import fields
from test_gpu_parity import pkg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def test_tuner_times_only_what_has_a_choice():
    import torch
    p = pkg()
    vols = []
    for i, dims in enumerate([(40, 36, 28), (64, 48, 52), (33, 70, 21)]):
        bits, bmin, bmax = oracle.encode_volume(fields.gradient_noise(*dims, i, octaves=4, base_period=16), 8)
        vols.append(p.Volume(bits, dims, 8, bmin, bmax))
    b = p.Batch(vols)
    isos = np.asarray([0.0, 0.1, -0.2], np.float32)
    out = torch.empty((1 << 18, 3, 4), dtype=torch.float32, device="cuda")
    try:
        for _ in range(4):
            sh = b.tune(isos, out, trials=1)["shape"]
            assert (sh["count_ctas"], sh["count_tile"], sh["scan_tile"]) == (1, 32, 2048)
        b.set_shape(count_tile=64, scan_tile=1024, count_ctas=3)         # accepted and reported
        sh = b.shape
        assert (sh["count_tile"], sh["scan_tile"]) == (64, 1024)
    finally:
        b.release()
        for v in vols:
            v.release()
