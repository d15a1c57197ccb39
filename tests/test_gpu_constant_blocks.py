"""Constant blocks (masked areas of surface fields): warps of nothing else, which the
2-D encoder writes in one go, and warps that hold them beside zero and varying
blocks.  Bit for bit against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import codec as oc
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


def fields():
    r = np.random.default_rng(5)
    shape = (2, 32, 4 * 128)

    def blocks(v):                                     # a value per 4 x 4 block of each level
        return np.kron(v, np.ones((1, 4, 4)))
    n = (2, 8, 128)
    sign = r.choice([-1.0, 1.0], n)
    yield "one value", np.full(shape, 273.15)
    yield "every number of leading empty planes", blocks(sign * np.ldexp(r.uniform(0.5, 1.0, n), r.integers(-3, 4, n)))
    yield "single bits", blocks(sign * np.ldexp(1.0, r.integers(-126, 128, n)))
    yield "all significant bits", blocks(sign * np.ldexp(np.nextafter(np.float32(1), np.float32(0)), r.integers(-125, 128, n)))
    yield "subnormal, zero, infinite, largest", blocks(r.choice([1e-40, -3e-39, 0.0, -0.0, np.inf, 3.4028235e38, -1.5], n))
    mixed = blocks(sign * r.uniform(1, 2, n))
    mixed[:, :, 200:300] += r.standard_normal((2, 32, 100))          # warps with varying blocks among them
    mixed[1, 16:, :] = 0.0
    yield "mixed", mixed
    yield "one odd value", np.where(np.arange(shape[2]) == 77, 1.0 + 2.0 ** -23, 1.0) * np.ones(shape)


@pytest.mark.parametrize("dims,rate", [(2, 8), (2, 16), (1, 8), (3, 8)])
def test_constant_blocks(dims, rate):
    for name, x in fields():
        x = x.astype(np.float32)
        n = tuple(reversed(x.shape))
        s = torch.full((z.zfpx_stream_bytes(dims, rate, n),), 255, dtype=torch.uint8, device="cuda")
        d = torch.full(x.shape, float("nan"), device="cuda")
        ref = oc.encode_array(dims, rate, x)
        rd = np.empty_like(x)
        oc.decode_array(dims, rate, ref, rd)
        z.zfpx_encode(dims, rate, torch.from_numpy(x).cuda(), s)
        z.zfpx_decode(dims, rate, s, d)
        assert s.cpu().numpy().tobytes() == bytes(ref), name
        assert np.array_equal(d.cpu().numpy().view(np.uint32), rd.view(np.uint32)), name
