"""The longitude FFT of rows of 64 r values in two register passes, for every
first radix it is built for, against the float64 oracle (paper Sec. II-A)."""
import numpy as np
import pytest
import torch

from oracle import fourier as of
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


# The bound per row is that of the other lengths' tests: a radix-p pass is
# sqrt(p) times a unitary map and adds a few u of its input's norm, 16 log2(N) u
# ||x|| / sqrt(N) in all.  Row counts below, at and above a CTA's four rows.
@pytest.mark.parametrize("r1", [4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20])
@pytest.mark.parametrize("rows", [(1, 1), (3, 5)])
def test_rows_of_64_r(r1, rows):
    N, u = 64 * r1, 2.0 ** -24
    nlev, nlat = rows
    x = np.random.default_rng(r1).standard_normal((nlev, nlat, N)).astype(np.float32)
    x[0, 0] = np.cos(2 * np.pi * (N // 2 - 1) * np.arange(N) / N)
    for K in (1, N // 2 - 1, N // 2 + 1):
        # padded rows and outputs: rows that start on 8 bytes only
        src = torch.zeros((nlev, nlat, N + 2), device="cuda")
        src[:, :, :N] = torch.from_numpy(x).cuda()
        re = torch.full((nlev, nlat, K + 3), float("nan"), device="cuda")
        im = torch.full_like(re, float("nan"))
        z.zfpx_rfft_lon(src[:, :, :N], re[:, :, :K], im[:, :, :K])
        rre, rim = of.rfft_lon(x, K)
        err = np.sqrt((re[:, :, :K].cpu().numpy() - rre) ** 2 + (im[:, :, :K].cpu().numpy() - rim) ** 2)
        bound = 16 * np.log2(N) * u * np.linalg.norm(x.astype(np.float64), axis=2) / np.sqrt(N)
        assert np.all(np.linalg.norm(err, axis=2) <= bound)
        assert torch.isnan(re[:, :, K:]).all() and torch.isnan(im[:, :, K:]).all()


# the fused decompression runs the same transform: bit for bit the separate calls
@pytest.mark.parametrize("N", [256, 576, 960, 1280])
def test_fused_rows_equal_the_separate_calls(N):
    x = torch.randn((5, 6, N), device="cuda", generator=torch.Generator("cuda").manual_seed(N))
    plan = z.Plan.for_fields(x, 2, 3, 0, 3)
    recv = torch.zeros(plan.buffer_bytes(16), dtype=torch.uint8, device="cuda")
    z.zfpx_pack_compress(plan, 16, x, recv, layout=z.LAYOUT_RECV)
    d = torch.empty_like(x)
    z.zfpx_decompress_unpack(plan, 16, recv, d)
    out = [torch.full((5, 6, N // 2 + 1), float("nan"), device="cuda") for _ in range(4)]
    z.zfpx_rfft_lon(d, out[0], out[1])
    z.zfpx_decompress_rfft(plan, 16, recv, out[2], out[3])
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])
