"""Device memory the calls hold: bytes a cache slot of a server's request
lists, and that the lists which two ticks share never mix their requests.
PyTorch's caching allocator serves the library here, so its own count of
requested bytes is the measure."""
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


@pytest.fixture
def held():
    """held(): bytes asked of PyTorch's allocator and not given back (with the
    library's among them); held(peak=True): the most since the last reset"""
    import torch
    torch.cuda.synchronize()
    pkg().use_torch_allocator()

    def count(peak=False):
        torch.cuda.synchronize()
        return torch.cuda.memory_stats()["requested_bytes.all." + ("peak" if peak else "current")]
    try:
        yield count
    finally:
        pkg().use_pool_allocator()


def noise(dims, rate, seed=11):
    f = fields.gradient_noise(*dims, seed, octaves=4, base_period=32)
    return oracle.encode_volume(f, rate)


@pytest.mark.parametrize("max_batch", [1, 8])
def test_server_bytes_a_slot(held, max_batch):
    dims, rate = (96, 88, 80), 4
    bits, bmin, bmax = noise(dims, rate)
    vol = pkg().Volume(bits, dims, rate, bmin, bmax)
    nb = int(np.prod(oracle.block_dims(dims)))           # as many cache slots
    try:
        before = held()
        srv = pkg().Server(vol, max_batch=max_batch)
        grown = held() - before
        srv.release()
        # 32 bytes a request's slot; descriptors and control blocks beside it
        # are 8 bytes a tile of at least 256 (candidates) or 2048 blocks
        assert grown <= 40 * max_batch * nb
    finally:
        vol.release()


# ticks of two or three under a backlog (each front overlaps the emission
# before it) and a vertex budget of about one mesh and a half (so a tick emits
# in rounds while the next one's front has already run)
@pytest.mark.parametrize("max_batch", [2, 3])
@pytest.mark.parametrize("budget", [0.0, 1.5])
def test_ticks_that_share_lists_keep_apart(max_batch, budget):
    p = pkg()
    dims, rate = (72, 60, 52), 8
    bits, bmin, bmax = noise(dims, rate)
    vol, alone = (p.Volume(bits, dims, rate, bmin, bmax) for _ in range(2))
    isos = [float(x) for x in np.random.default_rng(8).uniform(-0.8, 0.8, 14)]
    want = []
    for x in isos:
        m = alone.extract(x)
        want.append(m.vertices.cpu().numpy().copy())
        m.release()
    largest = max(w.nbytes for w in want)
    srv = p.Server(vol, max_batch=max_batch, vertex_budget_bytes=int(budget * largest))
    try:
        tickets = dict(zip([srv.submit(x) for x in isos], want))
        while tickets:
            srv.step()
            for t in list(tickets):
                status, m = srv.take(t)
                if status == p.ISO_PENDING:
                    continue
                assert status == p.ISO_OK
                assert np.array_equal(m.vertices.cpu().numpy().view(np.uint32), tickets.pop(t).view(np.uint32))
                m.release()
    finally:
        srv.release()
        vol.release()
        alone.release()


def test_volume_bytes_a_block(held):
    import torch
    dims, rate = (160, 160, 240), 2
    nb = int(np.prod(oracle.block_dims(dims)))
    bits = torch.zeros((nb, rate), dtype=torch.int64, device="cuda")
    rng = torch.zeros(nb, dtype=torch.float32, device="cuda")
    before = held()
    vol = pkg().Volume(bits, dims, rate, rng, rng)
    try:
        # bitstream, two hulls, slot map, samples, then nine lists of 4 bytes
        # a slot and three of 8; a byte for what is kept by the tile
        assert held() - before <= (8 * rate + 16 + 4 + 256 + 9 * 4 + 3 * 8 + 1) * nb
    finally:
        vol.release()


def by_candidate(vol, ref, vertices=None):
    cand = vol.debug("candidates")
    at = np.searchsorted(ref["ids"], cand)
    assert np.array_equal(ref["ids"][at], cand)
    tris = vol.debug("block_tris")
    assert np.array_equal(tris & 0xFFFF, ref["block_tri"][at])
    assert (tris >> 16).sum() == (vertices or 0) and not (tris >> 16)[ref["block_tri"][at] == 0].any()
    assert np.array_equal(vol.debug("block_offsets"), ref["block_off"][at])


# the triangles and offsets of every candidate, which no extraction writes:
# after soups, indexed meshes and a cache reset, and none after a ray cast
def test_candidates_counts_on_request():
    p = pkg()
    dims, rate = (41, 34, 27), 8
    bits, bmin, bmax = noise(dims, rate)
    vol = p.Volume(bits, dims, rate, bmin, bmax)
    try:
        for iso in (0.1, -0.4):
            ref = oracle.extract(bits, dims, rate, bmin, bmax, iso)
            vol.extract(iso).release()
            by_candidate(vol, ref)
            vol.cache_reset()
            by_candidate(vol, ref)
            verts, idx, st = vol.extract_indexed(iso)
            by_candidate(vol, ref, st["num_vertices"])
        vol.extract(float(bmax.max()) + 1.0).release()
        assert len(vol.debug("block_tris")) == 0
        vol.raycast(0.1, (-9, 15, 12), (1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 0, 1), 16, 16)
        assert len(vol.debug("block_tris")) == len(vol.debug("candidates")) > 0
        assert not vol.debug("block_tris").any()
    finally:
        vol.release()


# a cast's own memory is a bit a block, and what it leaves in the volume's
# lists does not reach the extractions after it
def test_raycast_bytes_a_block(held):
    import torch
    p = pkg()
    dims, rate = (120, 96, 100), 8
    nb = int(np.prod(oracle.block_dims(dims)))
    bits, bmin, bmax = noise(dims, rate)
    vol = p.Volume(bits, dims, rate, bmin, bmax)
    cam = ((-40, 48, 50), (1, 0, 0), (0, 0.8, 0), (0, 0, 0.8), (0, 0, 1), 64, 48)
    hits, rgba = (torch.empty((48, 64), dtype=d, device="cuda") for d in (torch.int64, torch.int32))
    try:
        m = vol.extract(0.2)
        want = m.vertices.cpu().numpy().view(np.uint32).copy()
        m.release()
        before = held()
        torch.cuda.reset_peak_memory_stats()
        vol.raycast(-0.3, *cam, hits=hits, rgba=rgba)
        assert held(peak=True) - before <= nb // 8 + 2048
        assert int((hits != -1).sum()) > 0
        m = vol.extract(0.2)
        assert np.array_equal(m.vertices.cpu().numpy().view(np.uint32), want)
        m.release()
    finally:
        vol.release()
