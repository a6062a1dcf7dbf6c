"""Sizes at which the tiled kernels change their split of the work, against the
CPU oracle: the count and scan's tiles (256 to 1024 candidates, by how many
there are for the CTAs), decode chunks and warps that end inside a volume, the
ray caster's path for rays whose reciprocal direction overflows, and the
rasteriser with and without its counts.  Everything here is compared bit for
bit but vertex positions, which test_gpu_parity bounds.
"""
import numpy as np
import pytest

import oracle
from synth import cameras, fields
from test_gpu_parity import check_surface, pkg, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def block_parity(nbx, nby, nbz):
    """a field whose blocks alternate along x: every block with a neighbour on +x is a candidate"""
    x = np.arange(4 * nbx) // 4 % 2
    f = np.where(x == 0, -1.0, 1.0).astype(np.float32)
    return np.ascontiguousarray(np.broadcast_to(f, (4 * nbz, 4 * nby, 4 * nbx)))


# candidates: one tile and its edges, then past one and three rounds of 152 x 256
@pytest.mark.parametrize("blocks", [(2, 1, 1), (257, 1, 1), (258, 1, 1), (1026, 1, 1), (61, 60, 12), (61, 60, 34)])
def test_count_tiles(blocks):
    dims, rate = tuple(4 * b for b in blocks), 2
    f = block_parity(*blocks)
    bits, bmin, bmax = oracle.encode_volume(f, rate)
    vol = pkg().Volume(bits, dims, rate, bmin, bmax, debug=blocks[2] < 20)
    n = (blocks[0] - 1) * blocks[1] * blocks[2]
    try:
        per_sheet = 2 * (dims[1] - 1) * (dims[2] - 1)
        want = None
        for ctas in (0, 1):                              # the default, then one CTA an SM
            vol.set_shape(**({"scan_ctas": ctas} if ctas else {}))
            m = vol.extract(0.25)
            assert m.stats["n_occupied"] == n and m.num_triangles == (blocks[0] - 1) * per_sheet
            got = m.vertices.cpu().numpy().view(np.uint32)
            assert want is None or np.array_equal(got, want)
            want = got
            if blocks[2] < 20:
                check_surface(vol, bits, dims, rate, bmin, bmax, 0.25, mesh=m)
            else:
                m.release()
    finally:
        vol.release()


# blocks of a decode: a warp's and a chunk's edges, with blocks repeated and out of order
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129])
@pytest.mark.parametrize("rate", [1, 3, 17, 32])
def test_decode_chunk_edges(n, rate):
    rng = np.random.default_rng(100 * rate + n)
    bits = rng.integers(0, 1 << 63, (200, rate), dtype=np.uint64)
    bits[:, 0] |= np.uint64(1)
    bits[::5, 0] &= ~np.uint64(1)                        # zero blocks among them
    bits[::7, rate - 1] = 0                              # codes that end in zeros
    ids = rng.integers(0, 200, n).astype(np.uint32)
    want = oracle.decode_blocks(bits, rate, ids)
    got = pkg().decode_blocks(to_dev(bits), rate, to_dev(ids)).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


# direction components so small that their reciprocals are infinite
@pytest.mark.parametrize("tiny", [1e-39, -1e-42])
def test_raycast_reciprocal_overflow(tiny):
    dims, rate = (33, 26, 19), 12
    f = fields.gradient_noise(*dims, 4, octaves=4, base_period=16)
    bits, bmin, bmax = oracle.encode_volume(f, rate)
    d = oracle.decode_volume(bits, dims, rate)
    iso = float(np.median(d))
    vol = pkg().Volume(bits, dims, rate, bmin, bmax)
    eye = np.asarray([-3.0, 12.3, 9.1], np.float32)
    fwd, right, up = (np.asarray(v, np.float32) for v in ([1.0, tiny, tiny], [0.0, tiny, 0.0], [0.0, 0.0, 0.4]))
    try:
        for w, h in ((33, 17), (8, 9)):
            hits, rgba, st = vol.raycast(iso, eye, fwd, right, up, (0.2, 0.3, 0.9), w, h)
            want_h, want_c = oracle.raycast(d, iso, eye, fwd, right, up, (0.2, 0.3, 0.9), w, h)
            assert np.array_equal(hits.cpu().numpy().view(np.uint64), want_h)
            assert np.array_equal(rgba.cpu().numpy().view(np.uint32), want_c)
    finally:
        vol.release()


@pytest.mark.parametrize("size", [(1, 1), (31, 17), (640, 360)])
def test_render_counts_change_nothing(size):
    dims, rate = (40, 33, 29), 8
    f = fields.gradient_noise(*dims, 9, octaves=4, base_period=16)
    bits, bmin, bmax = oracle.encode_volume(f, rate)
    vol = pkg().Volume(bits, dims, rate, bmin, bmax)
    try:
        m = vol.extract(0.0)
        cam = cameras.orbit(dims, 30.0, 25.0, aspect=size[0] / size[1])
        a = pkg().render(m.vertices, m.num_triangles, dims, cam, (0, 0, 1), *size)
        b = pkg().render(m.vertices, m.num_triangles, dims, cam, (0, 0, 1), *size, stats=True)
        assert np.array_equal(a[0].cpu().numpy(), b[0].cpu().numpy())
        assert np.array_equal(a[1].cpu().numpy(), b[1].cpu().numpy())
        assert a[2] is None and b[2] is not None
        m.release()
    finally:
        vol.release()
