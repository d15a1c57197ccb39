"""What the framework's performance is measured on: the work a spectral model's
transposition path hands to it, through the public entry points, from the
smallest field to the benchmark's.

Fields are seeded random fields with a power-law spectrum of slope -1.5 in
total wavenumber, unit RMS per level, correlated from level to level, plus
white noise of 0.01 (the shape of the repository's benchmark field), in three
flavours: "wind" (as is), "temperature" (250 + 20 f) and "humidity"
(exp(-8 + 2 f)).  They are made on the device from the seed alone.
"""
import numpy as np
import torch

from paper_2609_24294_gb300 import zfpx as z

KINDS = ("transposition", "raw", "pair", "batch", "accuracy", "f64", "rfft", "legendre")


def listed():
    return [
        # the smallest whole call: a T21 test field over 2 x 2 ranks, where launches and latency count
        {"name": "t21_transposition_r16", "kind": "transposition", "nlon": 64, "nlat": 32, "nlev": 8, "pr": 2,
         "pc": 2, "which": 0, "dims": 3, "rate": 16, "pad": 0, "flavour": "wind"},
        # one rank's pencil of the 2560 x 1280 x 137 grid on 121 ranks: what each GPU codes at scale; odd extents
        {"name": "rank_pencil_r8", "kind": "raw", "nlon": 233, "nlat": 117, "nlev": 137, "dims": 3, "rate": 8,
         "pad": 3, "flavour": "temperature"},
        # the benchmark's transposition: compress, all-to-all, decompress of a full field over 8 x 8 ranks
        {"name": "field_transposition_r8", "kind": "transposition", "nlon": 1280, "nlat": 640, "nlev": 137, "pr": 8,
         "pc": 8, "which": 0, "dims": 3, "rate": 8, "pad": 0, "flavour": "wind"},
        # both transpositions of a step as one CUDA graph, at the accurate rate
        {"name": "field_pair_graph_r16", "kind": "pair", "nlon": 1280, "nlat": 640, "nlev": 137, "pr": 8, "pc": 8,
         "rate": 16, "fold": False, "flavour": "wind"},
        # an uneven split (3 x 3 ranks) of a field whose rows are padded for an in-place FFT: nothing on 16 bytes
        {"name": "ragged_transposition_r8", "kind": "transposition", "nlon": 1000, "nlat": 501, "nlev": 91, "pr": 3,
         "pc": 3, "which": 1, "dims": 3, "rate": 8, "pad": 2, "flavour": "temperature"},
        # single-level fields (surface variables) in 2-D blocks
        {"name": "surface_2d_r16", "kind": "transposition", "nlon": 1280, "nlat": 640, "nlev": 37, "pr": 4, "pc": 4,
         "which": 0, "dims": 2, "rate": 16, "pad": 0, "flavour": "temperature"},
        # rows on their own in 1-D blocks, the smallest blocks of the codec
        {"name": "rows_1d_r8", "kind": "raw", "nlon": 1280, "nlat": 640, "nlev": 37, "dims": 1, "rate": 8, "pad": 0,
         "flavour": "humidity"},
        # fields on the octahedral reduced grid, 3-D and single-level ones at both rates, batched in one launch
        {"name": "octahedral_batch", "kind": "batch", "N": 640, "nlev": 60, "nsingle": 6},
        # the variable-rate mode over ranks: compress to a tolerance, all-to-all-v, decompress
        {"name": "accuracy_transposition", "kind": "accuracy", "nlon": 640, "nlat": 320, "nlev": 137, "pr": 4,
         "pc": 4, "which": 0, "tolerance": 1e-3, "precision": 0, "flavour": "wind"},
        # float64 model fields coded as they are
        {"name": "f64_r16", "kind": "f64", "nlon": 640, "nlat": 320, "nlev": 91, "rate": 16, "pad": 0,
         "flavour": "temperature"},
        # the longitude FFT of the decoded lambda-pencils
        {"name": "fft_1280", "kind": "rfft", "nlon": 1280, "nlat": 640, "nlev": 137, "K": 640, "fused": False,
         "rate": 8, "pr": 8, "pc": 8, "flavour": "wind"},
        # the Legendre transform of the theta-pencils
        {"name": "legendre_t639", "kind": "legendre", "T": 639, "nlat": 640, "nlev": 137},
    ]


def _logint(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _smooth_even(rng, lo, hi):
    """An even length of 2, 3 and 5 only, log-uniform over [lo, hi]."""
    target = lo * (hi / lo) ** rng.random()
    best = 2
    a = 2
    while a <= hi:
        b = a
        while b <= hi:
            c = b
            while c <= hi:
                if lo <= c and abs(c - target) < abs(best - target):
                    best = c
                c *= 5
            b *= 3
        a *= 2
    return best


def draw(rng):
    kind = rng.choice(KINDS)
    c = {"kind": kind}
    flavour = rng.choice(("wind", "temperature", "humidity"))
    if kind in ("transposition", "raw", "pair", "accuracy"):
        c.update(nlon=_logint(rng, 64, 1280), nlat=_logint(rng, 32, 640), nlev=_logint(rng, 4, 137), flavour=flavour)
    if kind in ("transposition", "pair", "accuracy"):
        c.update(pr=rng.randint(1, 8), pc=rng.randint(1, 8))
    if kind in ("transposition", "accuracy"):
        c.update(which=rng.randint(0, 1))
    if kind in ("transposition", "raw"):
        dims = rng.choice((3, 3, 2, 1))
        if dims != 3:                                   # what the listed single-level cases hold at most
            c.update(nlev=min(c["nlev"], 37))
        c.update(dims=dims, rate=rng.choice((8, 16)), pad=rng.choice((0, 0, 2, 3)))
    elif kind == "pair":
        c.update(rate=rng.choice((8, 16)), fold=rng.random() < 0.5)
    elif kind == "batch":
        c.update(N=_logint(rng, 32, 640), nlev=_logint(rng, 4, 60), nsingle=rng.randint(1, 6))
    elif kind == "accuracy":
        c.update(nlon=min(c["nlon"], 640), nlat=min(c["nlat"], 320), flavour=rng.choice(("wind", "temperature")),
                 tolerance=float(10.0 ** -rng.uniform(1, 4)), precision=rng.choice((0, 0, rng.randint(8, 24))))
    elif kind == "f64":
        c.update(nlon=_logint(rng, 64, 640), nlat=_logint(rng, 32, 320), nlev=_logint(rng, 4, 91),
                 rate=rng.choice((8, 11, 16, 24, 32)), pad=rng.choice((0, 0, 1, 2)), flavour=flavour)
    elif kind == "rfft":
        n = _smooth_even(rng, 64, 1280)
        c.update(nlon=n, nlat=_logint(rng, 32, 640), nlev=_logint(rng, 4, 137), K=rng.choice((n // 2, n // 2 + 1, n // 3)),
                 fused=rng.random() < 0.4, rate=rng.choice((8, 16)), pr=rng.randint(1, 8), pc=rng.randint(1, 8),
                 flavour=rng.choice(("wind", "temperature")))
    elif kind == "legendre":
        nlat = 2 * _logint(rng, 16, 320)
        c.update(nlat=nlat, T=max(15, int((nlat - 1) * rng.choice((1.0, 0.667)))), nlev=_logint(rng, 4, 137))
    return c


# ---------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _field(nlev, nlat, nlon, flavour, gen, rho=0.9):
    """float32 [nlev][nlat][nlon] on the device."""
    ky = torch.fft.fftfreq(nlat, 1.0 / nlat, device="cuda")
    kx = torch.fft.rfftfreq(nlon, 1.0 / nlon, device="cuda")
    amp = (torch.sqrt(ky[:, None] ** 2 + kx[None, :] ** 2) + 1.0) ** -1.5
    out = torch.empty((nlev, nlat, nlon), dtype=torch.float32, device="cuda")
    s = float(np.sqrt(1.0 - rho * rho))
    prev = None
    for k in range(nlev):
        w = torch.randn((2, nlat, nlon // 2 + 1), device="cuda", generator=gen)
        w = torch.complex(w[0], w[1]) * amp
        prev = w if prev is None else rho * prev + s * w
        f = torch.fft.irfft2(prev, s=(nlat, nlon))
        out[k] = f / f.square().mean().sqrt()
    out += 0.01 * torch.randn(out.shape, device="cuda", generator=gen)
    if flavour == "temperature":
        out.mul_(20.0).add_(250.0)
    elif flavour == "humidity":
        out.mul_(2.0).sub_(8.0).exp_()
    return out


def _wavenumbers(nlev, nlat, T, gen):
    """Real and imaginary parts [nlev][nlat][T + 1], falling off with the order as the spectrum does."""
    amp = (torch.arange(T + 1, device="cuda") + 1.0) ** -1.5
    re, im = (torch.randn((nlev, nlat, T + 1), device="cuda", generator=gen) * amp for _ in range(2))
    im[:, :, 0] = 0.0
    return re, im


def _padded(f, pad):
    """The same field inside rows `pad` values longer, as a model's work array holds it."""
    if not pad:
        return f
    a = torch.zeros(f.shape[:2] + (f.shape[2] + pad,), dtype=f.dtype, device=f.device)
    v = a[:, :, :f.shape[2]]
    v.copy_(f)
    return v


def _bytes(n):
    return torch.zeros(int(n), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    c, kind, gen = case, case["kind"], _gen(seed)
    s = {"case": dict(case)}
    if kind in ("transposition", "raw"):
        s["src"] = _padded(_field(c["nlev"], c["nlat"], c["nlon"], c["flavour"], gen), c["pad"])
        s["dst"] = _padded(torch.zeros((c["nlev"], c["nlat"], c["nlon"]), device="cuda"), c["pad"])
        if kind == "raw":
            s["send"] = _bytes(z.zfpx_stream_bytes(c["dims"], c["rate"], (c["nlon"], c["nlat"], c["nlev"])))
        else:
            s["plan"] = z.Plan.for_fields(s["src"], c["pr"], c["pc"], c["which"], c["dims"], dst=s["dst"])
            s["plan"].prepare(c["rate"])
            s["send"] = _bytes(s["plan"].buffer_bytes(c["rate"]))
            s["recv"] = torch.zeros_like(s["send"])
    elif kind == "pair":
        s["src"] = _field(c["nlev"], c["nlat"], c["nlon"], c["flavour"], gen)
        s["mid"], s["dst"] = torch.zeros_like(s["src"]), torch.zeros_like(s["src"])
        first = z.Plan.for_fields(s["src"], c["pr"], c["pc"], 0, 3)
        second = z.Plan.for_fields(s["src"], c["pr"], c["pc"], 1, 3)
        n = max(first.buffer_bytes(c["rate"]), second.buffer_bytes(c["rate"]))
        s["send"], s["recv"] = _bytes(n), _bytes(n)
        s["graph"] = z.PairGraph(first, second, c["rate"], s["src"], s["mid"], s["dst"], s["send"], s["recv"],
                                 fold_permute=c["fold"])
    elif kind == "batch":
        north = 20 + 4 * np.arange(c["N"], dtype=np.int64)
        lens = np.concatenate([north, north[::-1]])
        longest = int(lens.max())
        at = torch.from_numpy(np.concatenate([r * longest + np.arange(n) for r, n in enumerate(lens)])).to("cuda")
        mix = [(c["nlev"], "temperature", 3, 8), (c["nlev"], "wind", 3, 16), (max(1, c["nlev"] // 2), "humidity", 3, 8)]
        mix += [(1, ("temperature", "humidity")[k % 2], 1, (8, 16)[k % 2]) for k in range(c["nsingle"])]
        fields = []
        for nlev, flavour, dims, rate in mix:
            f = _field(nlev, len(lens), longest, flavour, gen).reshape(nlev, -1)[:, at].contiguous()
            fields.append((f, torch.zeros_like(f), dims, rate))
        s["fields"] = fields
        s["batch"] = z.Batch(lens.tolist(), fields)
        s["send"] = _bytes(s["batch"].nbytes())
    elif kind == "accuracy":
        s["src"] = _field(c["nlev"], c["nlat"], c["nlon"], c["flavour"], gen)
        s["dst"] = torch.zeros_like(s["src"])
        s["acc"] = z.AccuracyTransposition(z.Plan.for_fields(s["src"], c["pr"], c["pc"], c["which"], 3))
        s["acc"].plan.prepare(16)
    elif kind == "f64":
        f = _field(c["nlev"], c["nlat"], c["nlon"], c["flavour"], gen).double()
        f *= 1.0 + 1e-8 * torch.randn(f.shape, device="cuda", generator=gen, dtype=torch.float64)
        s["src"] = _padded(f, c["pad"])
        s["dst"] = _padded(torch.zeros_like(f), c["pad"])
        s["send"] = _bytes(z.zfpx_stream_bytes_f64(c["rate"], (c["nlon"], c["nlat"], c["nlev"])))
    elif kind == "rfft":
        s["src"] = _field(c["nlev"], c["nlat"], c["nlon"], c["flavour"], gen)
        s["re"] = torch.zeros((c["nlev"], c["nlat"], c["K"]), device="cuda")
        s["im"] = torch.zeros_like(s["re"])
        if c["fused"]:
            s["plan"] = z.Plan.for_fields(s["src"], c["pr"], c["pc"], 0, 3)
            s["recv"] = _bytes(s["plan"].buffer_bytes(c["rate"]))
            z.zfpx_pack_compress(s["plan"], c["rate"], s["src"], s["recv"], layout=z.LAYOUT_RECV)
            s["work"] = z.zfpx_decompress_rfft(s["plan"], c["rate"], s["recv"], s["re"], s["im"])
    elif kind == "legendre":
        s["re"], s["im"] = _wavenumbers(c["nlev"], c["nlat"], c["T"], gen)
        s["plan"] = z.Legendre(c["nlat"], c["T"])
        s["are"], s["aim"] = (torch.zeros((c["nlev"], s["plan"].ncoeffs), device="cuda") for _ in range(2))
    else:
        raise ValueError(kind)
    return s


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "transposition":
        z.zfpx_pack_compress(s["plan"], c["rate"], s["src"], s["send"])
        z.zfpx_permute(s["plan"], c["rate"], s["send"], s["recv"])
        z.zfpx_decompress_unpack(s["plan"], c["rate"], s["recv"], s["dst"])
        return {"send": s["send"], "recv": s["recv"], "dst": s["dst"]}
    if kind == "raw":
        z.zfpx_encode(c["dims"], c["rate"], s["src"], s["send"])
        z.zfpx_decode(c["dims"], c["rate"], s["send"], s["dst"])
        return {"stream": s["send"], "dst": s["dst"]}
    if kind == "pair":
        s["graph"].launch()
        return {"mid": s["mid"], "dst": s["dst"], "recv": s["recv"]}
    if kind == "batch":
        s["batch"].encode(s["send"])
        s["batch"].decode(s["send"])
        return {"stream": s["send"], "dst": [f[1] for f in s["fields"]]}
    if kind == "accuracy":
        a = s["acc"]
        if c["precision"]:
            a.compress_precision(s["src"], c["precision"])
        else:
            a.compress(s["src"], c["tolerance"])
        a.exchange()
        a.decompress(s["dst"])
        return {"lengths": a.len_send, "words": a.words, "sent": a.pay_send, "received": a.pay_recv,
                "received_lengths": a.len_recv, "dst": s["dst"]}
    if kind == "f64":
        z.zfpx_encode_f64(c["rate"], s["src"], s["send"])
        z.zfpx_decode_f64(c["rate"], s["send"], s["dst"])
        return {"stream": s["send"], "dst": s["dst"]}
    if kind == "rfft":
        if c["fused"]:
            z.zfpx_decompress_rfft(s["plan"], c["rate"], s["recv"], s["re"], s["im"], work=s["work"])
        else:
            z.zfpx_rfft_lon(s["src"], s["re"], s["im"])
        return {"re": s["re"], "im": s["im"]}
    s["plan"].forward(s["re"], s["im"], s["are"], s["aim"])
    return {"are": s["are"], "aim": s["aim"]}


# ---------------------------------------------------------------------------- what a pass cannot do without
def _part(n, parts):
    return [n // parts + (1 if i < n % parts else 0) for i in range(parts)]


def _coded(c, which, dims, rate):
    """Stream bytes of a plan's messages (every call reads or writes them once)."""
    xs = _part(c["nlon"], c["pc"] if which == 0 else c["pr"])
    ys, zs = _part(c["nlat"], c["pr"]), _part(c["nlev"], c["pc"])
    bx = sum(-(-v // 4) for v in xs)
    by = sum(-(-v // 4) if dims > 1 else v for v in ys)
    bz = sum(-(-v // 4) if dims == 3 else v for v in zs)
    return bx * by * bz * 4 ** dims * rate // 8


def work(case):
    c, kind = case, case["kind"]
    flops = 0
    if kind == "legendre":
        T, nlev = c["T"], c["nlev"]
        coeffs = (T + 1) * (T + 2) // 2
        # the wavenumber fields, w Pbar on half the latitudes, the coefficients; a multiply and an add per product
        return {"bytes": 4 * (2 * nlev * c["nlat"] * (T + 1) + coeffs * (c["nlat"] // 2) + 2 * nlev * coeffs),
                "flops": 2 * coeffs * (c["nlat"] // 2) * 2 * nlev}
    if kind == "batch":
        north = [20 + 4 * i for i in range(c["N"])]
        lens = north + north[::-1]
        quads = sum(-(-max(lens[q:q + 4]) // 4) for q in range(0, len(lens), 4))
        per = sum(lens)
        half = max(1, c["nlev"] // 2)
        levels = 2 * c["nlev"] + half + c["nsingle"]
        stream = quads * (-(-c["nlev"] // 4) * 64 * 3 + -(-half // 4) * 64)
        stream += sum(per * (8, 16)[k % 2] // 8 for k in range(c["nsingle"]))
        return {"bytes": 2 * (4 * per * levels + stream), "flops": 0}
    n = c["nlon"] * c["nlat"] * c["nlev"]
    if kind == "transposition":
        b = 8 * n + 4 * _coded(c, c["which"], c["dims"], c["rate"])
    elif kind == "raw":
        b = 8 * n + 2 * z.zfpx_stream_bytes(c["dims"], c["rate"], (c["nlon"], c["nlat"], c["nlev"]))
    elif kind == "pair":
        k = 2 if c["fold"] else 4
        b = 16 * n + k * (_coded(c, 0, 3, c["rate"]) + _coded(c, 1, 3, c["rate"]))
    elif kind == "accuracy":
        # at most 16 bits a value, about 14 at the tolerances used; the encoder also clears its whole buffer
        blocks = _coded(c, c["which"], 3, 8) // 64
        b = 8 * n + 4 * blocks * (112 + 2)
    elif kind == "f64":
        b = 16 * n + 2 * z.zfpx_stream_bytes_f64(c["rate"], (c["nlon"], c["nlat"], c["nlev"]))
    else:
        b = (_coded(c, 0, 3, c["rate"]) if c["fused"] else 4 * n) + 8 * c["K"] * c["nlat"] * c["nlev"]
        flops = int(2.5 * n * np.log2(c["nlon"]))
    return {"bytes": int(b), "flops": flops}


# ---------------------------------------------------------------------------- in 64 bits
def _legendre64(re, im, nlat, T):
    mu, w = np.polynomial.legendre.leggauss(nlat)
    mu = torch.from_numpy(mu[::-1].copy()).to("cuda")
    w = torch.from_numpy(w[::-1].copy()).to("cuda")
    F = torch.complex(re.double(), im.double()) * w[None, :, None]
    nlev, M = re.shape[0], T + 1
    m = torch.arange(M, dtype=torch.float64, device="cuda")
    s = torch.sqrt(1.0 - mu * mu)
    log = 0.5 * torch.log((2.0 * m + 1.0) / (2.0 * m.clamp(min=1.0)))
    log[0] = 0.0
    sign = torch.where(m.long() % 2 == 1, -1.0, 1.0).double()
    diag = sign * torch.exp(0.5 * np.log(0.5) + torch.cumsum(log, 0) + m * torch.log(s)[:, None])
    out = torch.zeros((nlev, M * (M + 1) // 2), dtype=torch.complex128, device="cuda")
    start = (m.long() * M - m.long() * (m.long() - 1) // 2)
    cur = torch.zeros((nlat, M), dtype=torch.float64, device="cuda")
    old = torch.zeros_like(cur)
    for l in range(M):
        new = torch.zeros_like(cur)
        if l:
            k = m[:l]
            a = torch.sqrt((4.0 * l * l - 1.0) / (l * l - k * k))
            b = torch.sqrt(((l - 1.0) ** 2 - k * k).clamp(min=0.0) / (4.0 * (l - 1.0) ** 2 - 1.0))
            new[:, :l] = a * (mu[:, None] * cur[:, :l] - b * old[:, :l])
        new[:, l] = diag[:, l]
        old, cur = cur, new
        out[:, start[:l + 1] + l - m[:l + 1].long()] = (F[:, :, :l + 1] * cur[None, :, :l + 1]).sum(1)
    return out.real.contiguous(), out.imag.contiguous()


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "legendre":
        are, aim = _legendre64(*_wavenumbers(c["nlev"], c["nlat"], c["T"], _gen(seed)), c["nlat"], c["T"])
        return {"are": are, "aim": aim}
    if kind == "rfft" and not c["fused"]:
        f = torch.fft.rfft(_field(c["nlev"], c["nlat"], c["nlon"], c["flavour"], _gen(seed)).double(), dim=2)
        f = f[:, :, :c["K"]] / c["nlon"]
        return {"re": f.real.contiguous(), "im": f.imag.contiguous()}
    return None                              # a lossy code: its bytes and values are the method's own, bit for bit
