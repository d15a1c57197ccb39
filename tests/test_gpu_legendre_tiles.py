"""The Legendre contraction's tiles at the edges of their sizes: columns (twice
the levels) around 192, the widest tile, and around a multiple of 256, where a
workspace block is narrower than the tiles over it; rows around 128; depths
around a slice of 32.  Bound: twice the float32 dot-product bound (nlat / 2 + 2) u
sum |w Pbar| |F| that the transform is held to everywhere."""
import numpy as np
import pytest
import torch

from oracle import legendre as ol
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.mark.parametrize("nlat,T,nlev", [(8, 5, 8), (8, 5, 95), (8, 5, 96), (8, 5, 97), (8, 5, 128), (8, 5, 129),
                                         (8, 5, 200), (8, 5, 289), (64, 63, 1), (66, 65, 9), (258, 253, 2),
                                         (258, 254, 7), (260, 257, 2)])
def test_tile_edges(nlat, T, nlev):
    r = np.random.default_rng(nlat + T + nlev)
    re, im = (r.standard_normal((nlev, nlat, T + 1)).astype(np.float32) for _ in range(2))
    p = z.Legendre(nlat, T)
    out = [torch.full((nlev, p.ncoeffs), float("nan"), device="cuda") for _ in range(2)]
    p.forward(torch.from_numpy(re).cuda(), torch.from_numpy(im).cuda(), *out)
    torch.cuda.synchronize()
    p.status()
    rre, rim, mag = ol.legendre_forward(re, im, T)
    bound = 2 * (nlat // 2 + 2) * U * mag + 1e-30
    for g, want in zip(out, (rre, rim)):
        assert np.all(np.abs(g.cpu().numpy().astype(np.float64) - want) <= bound)
    p.close()
