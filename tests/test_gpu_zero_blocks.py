"""Fields with large zero parts (precipitation, cloud, masked areas): warps of
zero blocks alone, which skip the coder, beside warps of mixed and of dense
blocks and after them in the same warp.  Bit for bit against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import codec as oc
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


def patchy(shape, seed, run):
    """Normal values with runs of `run` zero blocks (4 values along x) and of dense ones."""
    r = np.random.default_rng(seed)
    nz, ny, nx = shape
    rows = -(-ny // 4) * -(-nz // 4)
    bx = -(-nx // 4)
    keep = np.repeat(r.random(-(-rows * bx // run)) < 0.5, run)[:rows * bx].reshape(-(-nz // 4), -(-ny // 4), bx)
    keep = np.kron(keep, np.ones((4, 4, 4), bool))[:nz, :ny, :nx]
    return np.where(keep, r.standard_normal(shape), r.choice([0.0, -0.0], shape))


# runs shorter than a warp's 32 blocks, of just as many, and longer; nothing but zeros
@pytest.mark.parametrize("run", [1, 7, 32, 96, 10 ** 6])
@pytest.mark.parametrize("dims,rate", [(1, 8), (2, 8), (2, 16), (3, 8), (3, 16)])
def test_zero_runs(dims, rate, run):
    x = patchy((6, 40, 500), run, run).astype(np.float32)
    if run == 10 ** 6:
        x *= 0
    n = tuple(reversed(x.shape))
    xd = torch.from_numpy(x).cuda()
    s = torch.full((z.zfpx_stream_bytes(dims, rate, n),), 255, dtype=torch.uint8, device="cuda")
    d = torch.full(x.shape, float("nan"), device="cuda")
    ref = oc.encode_array(dims, rate, x)
    rd = np.empty_like(x)
    oc.decode_array(dims, rate, ref, rd)
    z.zfpx_encode(dims, rate, xd, s)
    z.zfpx_decode(dims, rate, s, d)
    assert s.cpu().numpy().tobytes() == bytes(ref)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), rd.view(np.uint32))


# odd and even rates, streams on 16 and on 8 bytes; enough blocks that a warp
# takes several units, zero ones after dense ones
@pytest.mark.parametrize("rate,offset", [(1, 0), (8, 0), (8, 8), (15, 8), (16, 0), (32, 0)])
@pytest.mark.parametrize("shape,run", [((3, 9, 41), 5), ((6, 40, 500), 32), ((24, 256, 512), 500), ((4, 4, 300), 10 ** 6)])
def test_zero_runs_float64(rate, offset, shape, run):
    x = patchy(shape, run, run) * (0.0 if run == 10 ** 6 else 1.0)
    n = tuple(reversed(shape))
    nb = z.zfpx_stream_bytes_f64(rate, n)
    s = torch.full((nb + 16,), 255, dtype=torch.uint8, device="cuda")[offset:offset + nb]
    xd, d = torch.from_numpy(x).cuda(), torch.full(shape, float("nan"), dtype=torch.float64, device="cuda")
    ref = oc.encode_array_f64(rate, x)
    z.zfpx_encode_f64(rate, xd, s)
    assert np.array_equal(s.cpu().numpy(), ref)
    z.zfpx_decode_f64(rate, s, d)
    rd = np.empty(shape)
    oc.decode_array_f64(rate, ref, rd)
    assert np.array_equal(d.cpu().numpy().view(np.uint64), rd.view(np.uint64))
