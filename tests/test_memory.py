"""Device memory the calls hold: bytes a cache slot of a server's request
lists, and that the lists which two ticks share never mix their requests.
PyTorch's caching allocator serves the library here, so its own count of
allocated bytes is the measure (rounded up to 512 bytes an allocation)."""
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
    """held(): bytes the library holds, through PyTorch's allocator"""
    import torch
    torch.cuda.synchronize()
    pkg().use_torch_allocator()

    def count():
        torch.cuda.synchronize()
        return torch.cuda.memory_allocated()
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
