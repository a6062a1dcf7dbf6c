"""Caller buffers that are not aligned to 16 bytes.  The codec calls move 16
bytes a lane where a buffer allows it; a float buffer may start at any float
(a contiguous view of a larger tensor does), and then gives the same bits.  A
pointer that its element type cannot use is refused before any device work."""
import ctypes

import numpy as np
import pytest

import oracle
from synth import fields


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2009_03254_gb300 import build
    build.build()


def pkg():
    import paper_2009_03254_gb300 as p
    return p


def test_pointers_no_element_fits_are_refused():
    # host arithmetic: addresses that are never dereferenced
    p = pkg()
    L, bad = p.lib(), p.ISO_ERR_INVALID_ARG
    at = ctypes.c_void_p
    ok = 4096
    for bits, field in ((ok + 4, ok), (ok, ok + 2)):
        assert L.iso_decode_volume(at(bits), 8, 8, 8, 4, at(field), None) == bad
    for bits, ids, out in ((ok + 4, ok, ok), (ok, ok + 1, ok), (ok, ok, ok + 2)):
        assert L.iso_decode_blocks(at(bits), 4, at(ids), 5, at(out), None) == bad
    for args in ((ok + 1, ok, ok, ok), (ok, ok + 4, ok, ok), (ok, ok, ok + 2, ok), (ok, ok, ok, ok + 3)):
        field, bits, lo, hi = map(at, args)
        assert L.iso_encode_field(field, 8, 8, 8, 4, bits, lo, hi, None) == bad
    opt = p._Options()
    opt.flags = p.ISO_INPUT_ON_DEVICE
    for lo, hi in ((ok + 2, ok), (ok, ok + 1)):
        h = ctypes.c_void_p()
        assert L.iso_load_volume(ctypes.byref(h), at(ok), 8 * 4 * 8, 8, 8, 8, 4, at(lo), at(hi),
                                 ctypes.byref(opt)) == bad


def offset(shape, floats, src=None):
    """a contiguous float32 CUDA tensor that starts `floats` past a 16-byte boundary"""
    import torch
    n = int(np.prod(shape))
    t = torch.zeros(n + 4, dtype=torch.float32, device="cuda")
    assert t.data_ptr() % 16 == 0
    t = t[floats:floats + n].view(*shape)
    return t if src is None else t.copy_(torch.from_numpy(src))


# rows of a multiple of four floats (moved whole where the buffer allows) and others
@pytest.mark.gpu
@pytest.mark.parametrize("floats", [0, 1, 2, 3])
@pytest.mark.parametrize("dims", [(40, 21, 18), (35, 22, 9)])
def test_offset_buffers_give_the_same_bits(dims, floats):
    import torch
    p, rate = pkg(), 6
    f = fields.gradient_noise(*dims, 5, octaves=4, base_period=16)
    bits, lo, hi = oracle.encode_volume(f, rate)
    nb = int(np.prod(oracle.block_dims(dims)))
    words = torch.empty((nb, rate), dtype=torch.int64, device="cuda")
    r = p.encode_field(offset(f.shape, floats, f), rate, out=(words, offset((nb,), floats), offset((nb,), floats)))
    assert np.array_equal(r[0].cpu().numpy().view(np.uint64), bits)
    assert np.array_equal(r[1].cpu().numpy(), lo) and np.array_equal(r[2].cpu().numpy(), hi)
    out = p.decode_volume(words, dims, rate, out=offset(f.shape, floats))
    assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.decode_volume(bits, dims, rate).view(np.uint32))
    ids = torch.arange(nb - 1, -1, -1, dtype=torch.int32, device="cuda")
    blocks = offset((nb, 64), floats)
    rc = p.lib().iso_decode_blocks(p._ptr(words), rate, p._ptr(ids), nb, p._ptr(blocks), p._current_stream())
    assert rc == p.ISO_OK
    want = oracle.decode_blocks(bits, rate, np.arange(nb - 1, -1, -1, dtype=np.uint32))
    assert np.array_equal(blocks.cpu().numpy().view(np.uint32), want.view(np.uint32))
