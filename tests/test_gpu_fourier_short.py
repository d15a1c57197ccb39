"""The longitude FFT of the lengths whose stages are fixed when the kernels are
compiled, against the float64 oracle and, fused with the decoder, against the
separate calls (paper Sec. II-A)."""
import numpy as np
import pytest
import torch

from oracle import fourier as of
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


# The bound per row is that of the other lengths' tests (16 log2(N) u ||x|| /
# sqrt(N)).  Row counts below, at and above a CTA's eight rows; every number of
# wavenumbers around half and all of them and around a warp's 32; rows on 16 and on
# 8 bytes.
@pytest.mark.parametrize("N", [32, 64, 96, 128, 160, 192])
@pytest.mark.parametrize("rows,pad", [((1, 1), 0), ((2, 4), 2), ((3, 11), 4)])
def test_short_rows(N, rows, pad):
    u = 2.0 ** -24
    nlev, nlat = rows
    x = np.random.default_rng(N).standard_normal((nlev, nlat, N)).astype(np.float32)
    x[0, 0] = np.cos(2 * np.pi * (N // 2 - 1) * np.arange(N) / N)
    src = torch.zeros((nlev, nlat, N + pad), device="cuda")
    src[:, :, :N] = torch.from_numpy(x).cuda()
    bound = 16 * np.log2(N) * u * np.linalg.norm(x.astype(np.float64), axis=2) / np.sqrt(N)
    for K in sorted({1, N // 4, N // 4 + 1, min(33, N // 2), N // 2 - 1, N // 2, N // 2 + 1}):
        re = torch.full((nlev, nlat, K + 3), float("nan"), device="cuda")
        im = torch.full_like(re, float("nan"))
        z.zfpx_rfft_lon(src[:, :, :N], re[:, :, :K], im[:, :, :K])
        rre, rim = of.rfft_lon(x, K)
        err = np.sqrt((re[:, :, :K].cpu().numpy() - rre) ** 2 + (im[:, :, :K].cpu().numpy() - rim) ** 2)
        assert np.all(np.linalg.norm(err, axis=2) <= bound)
        assert torch.isnan(re[:, :, K:]).all() and torch.isnan(im[:, :, K:]).all()


@pytest.mark.parametrize("rate", [8, 16])
@pytest.mark.parametrize("N", [32, 64, 96, 128, 160, 192])
def test_fused_short_rows_equal_the_separate_calls(N, rate):
    x = torch.randn((5, 9, N), device="cuda", generator=torch.Generator("cuda").manual_seed(N))
    plan = z.Plan.for_fields(x, 2, 3, 0, 3)
    recv = torch.zeros(plan.buffer_bytes(rate), dtype=torch.uint8, device="cuda")
    z.zfpx_pack_compress(plan, rate, x, recv, layout=z.LAYOUT_RECV)
    d = torch.empty_like(x)
    z.zfpx_decompress_unpack(plan, rate, recv, d)
    out = [torch.full((5, 9, N // 2 + 1), float("nan"), device="cuda") for _ in range(4)]
    z.zfpx_rfft_lon(d, out[0], out[1])
    z.zfpx_decompress_rfft(plan, rate, recv, out[2], out[3])
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])
