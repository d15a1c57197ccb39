"""Warps whose lanes take different ways through the 3-D codec kernels: zero
blocks (a single bit, decoded without a plane), dense ones, blocks with a few
values (their planes end early) and blocks partial in x, which pass through
shared memory on their way in and out.  Bit for bit against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import codec as oc
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def lane_per_block():
    for encode in (0, 1):
        for rate in (8, 16):
            z.zfpx_set_units_per_warp(encode, rate, 1)
    yield
    for encode in (0, 1):
        for rate in (8, 16):
            z.zfpx_set_units_per_warp(encode, rate, 0)


def mixed_field(nz, ny, nx, seed):
    """Every 4 x 4 x 4 block zero, dense, of one value or of one tiny exponent, at random."""
    r = np.random.default_rng(seed)
    kind = r.integers(0, 4, (-(-nz // 4), -(-ny // 4), -(-nx // 4)))
    kind = np.kron(kind, np.ones((4, 4, 4), int))[:nz, :ny, :nx]
    x = r.standard_normal((nz, ny, nx))
    return np.select([kind == 0, kind == 1, kind == 2], [0.0 * x, x, x * (r.random(x.shape) < 0.03)],
                     np.ldexp(x, -110)).astype(np.float32)


# rows of two to eight blocks with one, two or three values in the last; pitches
# for 16-byte rows (also the partial blocks' neighbours then move 16 bytes at a
# time), 8-byte rows, rows that start differently; extents partial in y and z too
@pytest.mark.parametrize("rate", [8, 16])
@pytest.mark.parametrize("nx,pitch", [(5, 8), (7, 7), (14, 16), (14, 14), (31, 32), (30, 31)])
def test_lanes_with_and_without_partial_blocks(nx, pitch, rate):
    nz, ny = 10, 70
    x = mixed_field(nz, ny, nx, nx * rate + pitch)
    src, dst = (torch.full((nz, ny, pitch), 7.0, device="cuda")[:, :, :nx] for _ in range(2))
    src.copy_(torch.from_numpy(x))
    n = (nx, ny, nz)
    s = torch.zeros(z.zfpx_stream_bytes(3, rate, n), dtype=torch.uint8, device="cuda")
    ref = oc.encode_array(3, rate, x)
    rd = np.empty_like(x)
    oc.decode_array(3, rate, ref, rd)
    for _ in range(3):
        s.zero_()
        dst.fill_(float("nan"))
        z.zfpx_encode(3, rate, src, s)
        z.zfpx_decode(3, rate, s, dst)
        assert s.cpu().numpy().tobytes() == bytes(ref)
        assert np.array_equal(dst.cpu().numpy().view(np.uint32), rd.view(np.uint32))


@pytest.mark.parametrize("nx,pitch", [(5, 8), (14, 14), (30, 31)])
def test_variable_rate_with_partial_blocks(nx, pitch):
    nz, ny = 10, 70
    x = mixed_field(nz, ny, nx, nx)
    src, dst = (torch.full((nz, ny, pitch), 7.0, device="cuda")[:, :, :nx] for _ in range(2))
    src.copy_(torch.from_numpy(x))
    n = (nx, ny, nz)
    lens = torch.zeros(z.zfpx_stream_bytes(3, 8, n) // 64, dtype=torch.int16, device="cuda")
    pay = torch.zeros(z.zfpx_accuracy_max_payload_bytes(n), dtype=torch.uint8, device="cuda")
    total = torch.zeros(1, dtype=torch.int64, device="cuda")
    work = torch.zeros(z.zfpx_accuracy_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    z.zfpx_encode_accuracy(src, 1e-4, lens, pay, total, work)
    z.zfpx_decode_accuracy(lens, pay, dst, work)
    rl, rp, rt = oc.encode_accuracy(x, 1e-4)
    rd = np.empty_like(x)
    oc.decode_accuracy(rl, rp, rd)
    assert int(total) == rt and np.array_equal(lens.cpu().numpy().view(np.uint16), rl)
    assert np.array_equal(pay.cpu().numpy()[:len(rp)], rp)
    assert np.array_equal(dst.cpu().numpy().view(np.uint32), rd.view(np.uint32))
