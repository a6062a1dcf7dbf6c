"""Launch shapes and the sizes at which launches change: what the tuner reports
of fields that choose nothing, volumes on both sides of the size up to which a
stage is launched before the one ahead of it has finished, and the count's
tiles of one to four rounds, soup and indexed mesh."""
import numpy as np
import pytest

import oracle
from synth import fields
from test_gpu_parity import check_surface, pkg
from test_gpu_tiles import block_parity

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


# 8192 blocks is the last size whose stages are launched ahead: debug volumes
# against the oracle, then the same bytes launch by launch and as a graph
@pytest.mark.parametrize("dims", [(128, 64, 64), (125, 62, 63), (132, 64, 64), (129, 61, 64)])
def test_stages_ahead_at_their_limit(dims):
    rate, iso = 6, 0.1
    nb = int(np.prod(oracle.block_dims(dims)))
    assert (nb <= 8192) == (dims[0] <= 128) and abs(nb - 8192) <= 256
    f = fields.gradient_noise(*dims, 17, octaves=4, base_period=32)
    bits, bmin, bmax = oracle.encode_volume(f, rate)
    dbg, vol = (pkg().Volume(bits, dims, rate, bmin, bmax, debug=d) for d in (True, False))
    try:
        m = dbg.extract(iso)
        want = m.vertices.cpu().numpy().view(np.uint32).copy()
        check_surface(dbg, bits, dims, rate, bmin, bmax, iso, mesh=m)
        for k in range(12):                              # captured from the ninth on
            if k % 3 == 0:
                vol.cache_reset()
            m = vol.extract(iso)
            assert np.array_equal(m.vertices.cpu().numpy().view(np.uint32), want)
            m.release()
    finally:
        vol.release()
        dbg.release()


# candidates for one to four rounds of 256 a tile on one count CTA an SM
# (152 x 256 a round); with the default four CTAs an SM all take one
@pytest.mark.parametrize("rounds,layers", [(1, 9), (2, 16), (3, 27), (4, 38)])
def test_count_rounds_soup_and_indexed(rounds, layers):
    import torch
    blocks = (61, 60, layers)
    cand = 60 * 60 * layers
    per_round = 256 * torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-cand // per_round) == rounds and cand <= 4 * per_round
    dims, rate = tuple(4 * b for b in blocks), 2
    bits, bmin, bmax = oracle.encode_volume(block_parity(*blocks), rate)
    vol = pkg().Volume(bits, dims, rate, bmin, bmax)
    try:
        want = None
        for ctas in (0, 1):
            vol.set_shape(**({"scan_ctas": ctas} if ctas else {}))
            m = vol.extract(0.25)
            assert m.stats["n_occupied"] == m.stats["n_candidates"] == cand
            assert m.num_triangles == 60 * 2 * (dims[1] - 1) * (dims[2] - 1)
            verts, idx, st = vol.extract_indexed(0.25, guess_triangles=m.num_triangles + 1)
            got = m.vertices.cpu().numpy().view(np.uint32).copy(), verts.cpu().numpy().view(np.uint32), idx.cpu().numpy()
            m.release()
            # every corner of the soup is the vertex its index names
            assert np.array_equal(got[1][got[2].reshape(-1)], got[0].reshape(-1, 4))
            assert want is None or all(np.array_equal(a, b) for a, b in zip(got, want))
            want = got
    finally:
        vol.release()
