"""Vertex interpolation at both ends of the reciprocal's range, against the
oracle's 64-bit quotients: t = (iso - lo) / (hi - lo) from differences rounded
once each (2^-24), a reciprocal good to 2^-23 and a product rounded once
(2^-24), then p + t rounded once with p + t <= 4 (half a unit in the last
place, 2^-23): within 7 * 2^-24 altogether.  Differences outside [2^-100, 2^125)
are formed from scaled samples; the emission skips that test where a cell's
samples allow it, the dense path never does, and both write the same bytes."""
import numpy as np
import pytest

import oracle
from synth import fields
from test_gpu_parity import pkg, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


# samples of about 2^e: differences on both sides of 2^-100 and of 2^125 (the
# emission's own limit on a sample's distance is 2^124), and well inside
@pytest.mark.parametrize("e", [-122, -101, -99, -60, 0, 60, 121, 123, 125])
def test_positions_against_64_bit_quotients(e):
    p = pkg()
    dims, rate = (29, 26, 22), 32
    f = np.ldexp(np.clip(fields.gradient_noise(*dims, 31, octaves=5, base_period=16), -3.5, 3.5), e).astype(np.float32)
    assert np.isfinite(f).all()
    bits, bmin, bmax = oracle.encode_volume(f, rate)
    d = oracle.decode_volume(bits, dims, rate)
    assert np.isfinite(d).all()
    iso = float(np.float32(np.ldexp(0.1, e)))
    ref = oracle.extract(bits, dims, rate, bmin, bmax, iso)
    vol = p.Volume(bits, dims, rate, bmin, bmax, debug=True)
    try:
        m = vol.extract(iso)
        v = m.vertices.cpu().numpy().reshape(-1, 3, 4)
        m.release()
        edges = vol.debug("edge_ids").reshape(-1, 3)
    finally:
        vol.release()
    assert len(v) == ref["num_triangles"] > 1000
    assert np.abs(v[:, :, :3].astype(np.float64) - ref["local_pos"].reshape(-1, 3, 3)).max() <= 7 * 2.0 ** -24
    dv, st, dedges = p.mc_dense(to_dev(d), iso, edge_ids=True)
    assert st["num_triangles"] == len(v)
    dv, dedges = dv.cpu().numpy(), dedges.cpu().numpy().view(np.uint64)
    a, b = np.lexsort(edges.T), np.lexsort(dedges.T)
    assert np.array_equal(edges[a], dedges[b])
    assert np.array_equal(v[a].view(np.uint32), dv[b].view(np.uint32))
