"""The codec's paths at the sizes and bit patterns where they can go wrong, bit
for bit against the CPU oracle (paper Sec. II-C; tolerance 0 throughout)."""
import numpy as np
import pytest
import torch

from oracle import codec as oc
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


def round_trip(x, dims, rate):
    """Stream bytes and decoded values of x ([lev][lat][lon]) equal the oracle's."""
    n = tuple(reversed(x.shape))
    xd = torch.from_numpy(x).cuda()
    s = torch.zeros(z.zfpx_stream_bytes(dims, rate, n), dtype=torch.uint8, device="cuda")
    d = torch.full(x.shape, float("nan"), device="cuda")
    z.zfpx_encode(dims, rate, xd, s)
    z.zfpx_decode(dims, rate, s, d)
    ref = oc.encode_array(dims, rate, x)
    assert s.cpu().numpy().tobytes() == bytes(ref)
    rd = np.empty_like(x)
    oc.decode_array(dims, rate, ref, rd)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), rd.view(np.uint32))


# values whose exponents are spread over all 32 planes, so that coefficients
# become significant one at a time, several at once and in the last planes, with
# runs of every length between
@pytest.mark.parametrize("dims", [1, 3])
@pytest.mark.parametrize("rate", [8, 16])
def test_significance_spread_over_the_planes(dims, rate):
    r = np.random.default_rng(100 * dims + rate)
    shape = (4, 64, 4 * 48)
    e = r.integers(0, 33, shape) * r.integers(0, 2, shape)
    x = np.ldexp(r.choice([-1.0, 1.0], shape) * r.choice([1.0, 1.0, 1.5, 1.999], shape), -e)
    x *= r.integers(0, 4, shape) != 0
    round_trip(x.astype(np.float32), dims, rate)


# launches of one unit, of a last unit with one block, and on both sides of the
# number of units from which a warp takes two
@pytest.mark.parametrize("blocks", [1, 31, 33, 1056])
@pytest.mark.parametrize("rate", [8, 16])
def test_units_at_the_edges(blocks, rate):
    x = np.random.default_rng(blocks).standard_normal((4, 4, 4 * blocks)).astype(np.float32)
    round_trip(x, 3, rate)


@pytest.mark.parametrize("rate", [8, 16])
def test_default_units_per_warp_either_side_of_the_rule(rate):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for per_sm in (8 * 15, 8 * 21):                    # fewer and more than eight units per resident warp
        y = (sms * per_sm * 32 + 63) // 64             # 64 blocks a row of blocks
        x = torch.randn((4, 4 * y, 256), device="cuda", generator=torch.Generator("cuda").manual_seed(per_sm))
        outs = []
        for upw in (0, 1, 2):
            z.zfpx_set_units_per_warp(1, rate, upw)
            z.zfpx_set_units_per_warp(0, rate, upw)
            try:
                s = torch.zeros(z.zfpx_stream_bytes(3, rate, (256, 4 * y, 4)), dtype=torch.uint8, device="cuda")
                d = torch.zeros_like(x)
                z.zfpx_encode(3, rate, x, s)
                z.zfpx_decode(3, rate, s, d)
                outs.append((s, d))
            finally:
                z.zfpx_set_units_per_warp(1, rate, 0)
                z.zfpx_set_units_per_warp(0, rate, 0)
        for s, d in outs[1:]:
            assert torch.equal(s, outs[0][0]) and torch.equal(d, outs[0][1])
