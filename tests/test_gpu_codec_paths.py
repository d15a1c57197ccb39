"""The codec's paths at the sizes and bit patterns where they can go wrong, bit
for bit against the CPU oracle (paper Sec. II-C; tolerance 0 throughout)."""
import numpy as np
import pytest
import torch

from oracle import codec as oc
from oracle import packs as op
from oracle import plan as opl
from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


# the 3-D codec by the library's choice (in small launches a warp per block) and
# always with a lane per block
@pytest.fixture(autouse=True, params=["chosen", "lane"])
def path(request):
    for encode in (0, 1):
        for rate in (8, 16):
            z.zfpx_set_units_per_warp(encode, rate, 1 if request.param == "lane" else 0)
    yield request.param
    for encode in (0, 1):
        for rate in (8, 16):
            z.zfpx_set_units_per_warp(encode, rate, 0)


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
    for per_sm in (6 * 15, 6 * 21):                    # fewer and more than six units per resident warp
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


# payloads whose words hold many blocks (1 and 9 bits each), end inside a word
# and in the middle of a warp's 32 blocks, blocks cut at 1024 bits beside zero
# blocks, and messages of one block: the payload written word by word against the
# oracle's bit string, and the tail zeroed
@pytest.mark.parametrize("blocks", [1, 31, 32, 33, 130, 1025])
@pytest.mark.parametrize("kind", ["tiny", "mixed", "full"])
def test_variable_rate_payload_words(blocks, kind):
    r = np.random.default_rng(blocks)
    x = r.standard_normal((4, 4, 4 * blocks)).astype(np.float32)
    keep = {"tiny": r.random(blocks) < 0.02, "mixed": r.random(blocks) < 0.5, "full": np.ones(blocks, bool)}[kind]
    x *= np.repeat(np.where(keep, 1.0, np.where(r.random(blocks) < 0.5, 0.0, 1e-6)), 4).astype(np.float32)
    tol = 1e-9 if kind == "full" else 1e-2
    n = (4 * blocks, 4, 4)
    xd = torch.from_numpy(x).cuda()
    lens = torch.zeros(blocks, dtype=torch.int16, device="cuda")
    pay = torch.full((z.zfpx_accuracy_max_payload_bytes(n),), 255, dtype=torch.uint8, device="cuda")
    total = torch.zeros(1, dtype=torch.int64, device="cuda")
    work = torch.zeros(z.zfpx_accuracy_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    z.zfpx_encode_accuracy(xd, tol, lens, pay, total, work)
    rl, rp, rt = oc.encode_accuracy(x, tol)
    assert np.array_equal(lens.cpu().numpy().view(np.uint16), rl) and int(total) == rt
    got = pay.cpu().numpy()                            # the oracle's payload ends with its last byte
    assert np.array_equal(got[:len(rp)], rp) and not got[len(rp):].any()
    d = torch.full(x.shape, float("nan"), device="cuda")
    z.zfpx_decode_accuracy(lens, pay, d, work)
    rd = np.empty_like(x)
    oc.decode_accuracy(rl, rp, rd)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), rd.view(np.uint32))


@pytest.mark.parametrize("shape,pr,pc", [((13, 9, 7), 3, 2), ((40, 24, 16), 10, 4), ((9, 5, 2), 2, 3)])
def test_variable_rate_messages_of_few_blocks(shape, pr, pc):
    x = np.random.default_rng(7).standard_normal(shape[::-1]).astype(np.float32)
    x[:, :, : shape[0] // 2] = 0.0
    xd = torch.from_numpy(x).cuda()
    plan = z.Plan.for_fields(xd, pr, pc, 0, 3)
    acc = z.AccuracyTransposition(plan)
    acc.pay_send.fill_(255)
    out = torch.full_like(xd, float("nan"))
    acc.compress(xd, 1e-3)
    acc.exchange()
    acc.decompress(out)
    for i, (ranks, (x0, nx, y0, ny, z0, nz)) in enumerate(plan.messages()):
        box = x[z0:z0 + nz, y0:y0 + ny, x0:x0 + nx]
        bits = 0
        if box.size:
            rl, rp, bits = oc.encode_accuracy(np.ascontiguousarray(box), 1e-3)
            rd = np.empty(box.shape, dtype=np.float32)
            oc.decode_accuracy(rl, rp, rd)
            got = out[z0:z0 + nz, y0:y0 + ny, x0:x0 + nx].cpu().numpy()
            assert np.array_equal(got.view(np.uint32), rd.view(np.uint32))
        assert int(acc.words[i]) == (bits + 63) // 64
    assert not acc.pay_send[8 * int(acc.words.sum()):].any()


# message counts around the powers of the 32-way message search, messages of one
# block each, and empty ones (more ranks than values)
@pytest.mark.parametrize("pr,pc", [(1, 1), (1, 5), (2, 4), (1, 6), (11, 3), (8, 12), (31, 6)])
@pytest.mark.parametrize("dims", [1, 2, 3])
def test_message_search(pr, pc, dims):
    x = np.random.default_rng(pr * pc).standard_normal((5, 33, 44)).astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    plan = z.Plan.for_fields(xd, pr, pc, 0, dims)
    s = torch.zeros(max(1, plan.buffer_bytes(8)), dtype=torch.uint8, device="cuda")
    d = torch.full_like(xd, float("nan"))
    z.zfpx_pack_compress(plan, 8, xd, s)
    z.zfpx_decompress_unpack(plan, 8, s, d, layout=z.LAYOUT_SEND)
    got, vals = s.cpu().numpy(), d.cpu().numpy()
    for (src, dst, _, _), (x0, nx, y0, ny, z0, nz) in plan.messages():
        box = np.ascontiguousarray(x[z0:z0 + nz, y0:y0 + ny, x0:x0 + nx])
        if not box.size:
            continue
        ref = oc.encode_array(dims, 8, box)
        off = plan.message_offset(8, z.LAYOUT_SEND, src, dst)
        assert np.array_equal(got[off:off + len(ref)], ref)
        rd = np.empty_like(box)
        oc.decode_array(dims, 8, ref, rd)
        assert np.array_equal(vals[z0:z0 + nz, y0:y0 + ny, x0:x0 + nx].view(np.uint32), rd.view(np.uint32))


# parts that close in the first, second and third 32-bit window, run through a
# whole window, end in its last bit or at the implied coefficient: streams of long
# runs of ones and zeros
@pytest.mark.parametrize("rate", [8, 16])
def test_streams_of_long_runs(rate):
    r = np.random.default_rng(rate)
    n = (4 * 512, 4, 4)
    bits = []
    for _ in range(512):
        b = np.zeros(64 * rate, np.uint8)
        p, v = 9, 1
        while p < len(b):
            q = p + int(r.choice([1, 2, 3, 7, 31, 32, 33, 63, 64, 65]))
            b[p:q] = v
            p, v = q, 1 - v
        b[:9] = 1, *r.integers(0, 2, 8)
        bits.append(b)
    s = np.packbits(np.concatenate(bits), bitorder="little")
    d = torch.full((4, 4, n[0]), float("nan"), device="cuda")
    z.zfpx_decode(3, rate, torch.from_numpy(s).cuda(), d)
    rd = np.empty((4, 4, n[0]), dtype=np.float32)
    oc.decode_array(3, rate, s, rd)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), rd.view(np.uint32))


# 2-D blocks: extents around a block and a unit, padded rows (element loads),
# planes in both halves of a word, blocks cut inside the verbatim, group-tested
# and all-significant planes at both budgets
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 7), (2, 4, 128), (1, 33, 132), (5, 64, 260)])
@pytest.mark.parametrize("rate", [8, 16])
def test_blocks_2d(shape, rate):
    r = np.random.default_rng(sum(shape))
    for x in (r.standard_normal(shape), np.ldexp(r.choice([-1.0, 1.0], shape), -r.integers(0, 33, shape)),
              np.cumsum(r.standard_normal(shape), 2) + 250.0, np.ldexp(r.standard_normal(shape), -120 - r.integers(0, 8, shape))):
        round_trip(x.astype(np.float32), 2, rate)


@pytest.mark.parametrize("rate", [8, 16])
def test_random_streams_2d(rate):
    r = np.random.default_rng(rate)
    n = (4 * 256, 8, 2)
    s = r.integers(0, 256, z.zfpx_stream_bytes(2, rate, n), dtype=np.uint8)
    s[:: 2 * rate] |= 1                                # every block non-zero
    half = len(s) // 2                                 # half of them with long runs
    s[:half] = np.where(r.random(half) < 0.7, 0, s[:half]) | (np.arange(half) % (2 * rate) == 0)
    d = torch.full((2, 8, n[0]), float("nan"), device="cuda")
    z.zfpx_decode(2, rate, torch.from_numpy(s).cuda(), d)
    rd = np.empty((2, 8, n[0]), dtype=np.float32)
    oc.decode_array(2, rate, s, rd)
    assert np.array_equal(d.cpu().numpy().view(np.uint32), rd.view(np.uint32))


# float64: coefficients that become significant in every one of the 64 planes, so
# that the low 32 planes are reached in phase A (sparse blocks, any rate), in the
# verbatim planes (rates from about 24 on) or not at all; odd rates and streams on
# 8 bytes; a unit with one block
@pytest.mark.parametrize("rate", [1, 3, 8, 15, 16, 24, 31, 32])
@pytest.mark.parametrize("shape,offset", [((4, 4, 4), 0), ((5, 9, 132), 8)])
def test_float64_planes(rate, shape, offset):
    r = np.random.default_rng(rate)
    n = tuple(reversed(shape))
    nb = z.zfpx_stream_bytes_f64(rate, n)
    for x in (np.ldexp(r.choice([-1.0, 1.0], shape) * r.choice([1.0, 1.25, 1.999], shape), -r.integers(0, 65, shape)),
              np.full(shape, 3.0) + np.ldexp(r.standard_normal(shape), -r.integers(30, 60)),
              np.cumsum(r.standard_normal(shape), 2) + 250.0,
              np.ldexp(r.standard_normal(shape), -1010 - r.integers(0, 20, shape)),
              np.where(r.random(shape) < 0.02, np.inf, r.standard_normal(shape))):
        s = torch.zeros(nb + 16, dtype=torch.uint8, device="cuda")[offset:offset + nb]
        xd, d = torch.from_numpy(x).cuda(), torch.full(shape, float("nan"), dtype=torch.float64, device="cuda")
        z.zfpx_encode_f64(rate, xd, s)
        ref = oc.encode_array_f64(rate, x)
        assert np.array_equal(s.cpu().numpy(), ref)
        z.zfpx_decode_f64(rate, s, d)
        rd = np.empty(shape)
        oc.decode_array_f64(rate, ref, rd)
        assert np.array_equal(d.cpu().numpy().view(np.uint64), rd.view(np.uint64))


# rows of every kind -- on 16, 8 and 4 bytes, rows that start alike and rows that
# don't (odd row pitch), values apart -- with every remainder of the x extent, one
# and several messages, both directions, nothing written outside the view
@pytest.mark.parametrize("rate", [8, 16])
@pytest.mark.parametrize("start,pitch,step", [(0, 0, 1), (0, 2, 1), (1, 2, 1), (2, 2, 1), (3, 1, 1), (1, 3, 1), (1, 2, 2)])
@pytest.mark.parametrize("nx", [4, 37, 42, 131])
def test_row_kinds(nx, start, pitch, step, rate):
    r = np.random.default_rng(nx)
    ny, nz = 9, 6
    width = start + step * nx + pitch
    width += width & 1 if pitch == 2 else 0            # even row pitch: rows start alike
    a = torch.from_numpy(r.standard_normal((nz, ny, width)).astype(np.float32)).cuda()
    o = torch.full((nz, ny, width), 7.0, device="cuda")
    src, dst = (t[:, :, start:start + step * nx:step] for t in (a, o))
    x = np.ascontiguousarray(src.cpu().numpy())
    for pr, pc in ((1, 1), (2, 3)):
        plan = z.Plan.for_fields(src, pr, pc, 0, 3, dst=dst)
        s = torch.zeros(plan.buffer_bytes(rate), dtype=torch.uint8, device="cuda")
        o.fill_(7.0)
        z.zfpx_pack_compress(plan, rate, src, s)
        z.zfpx_decompress_unpack(plan, rate, s, dst, layout=z.LAYOUT_SEND)
        got, full = s.cpu().numpy(), o.cpu().numpy()
        vals = full[:, :, start:start + step * nx:step]
        for (sr, ds, _, _), (x0, mx, y0, my, z0, mz) in plan.messages():
            box = np.ascontiguousarray(x[z0:z0 + mz, y0:y0 + my, x0:x0 + mx])
            ref = oc.encode_array(3, rate, box)
            off = plan.message_offset(rate, z.LAYOUT_SEND, sr, ds)
            assert np.array_equal(got[off:off + len(ref)], ref)
            rd = np.empty_like(box)
            oc.decode_array(3, rate, ref, rd)
            assert np.array_equal(vals[z0:z0 + mz, y0:y0 + my, x0:x0 + mx].view(np.uint32), rd.view(np.uint32))
        full[:, :, start:start + step * nx:step] = 7.0
        assert (full == 7.0).all()


# batches on both sides of the claim path (fewer and more units than the grid has
# warps) and of the library's own launch shape, unit size and claims: every choice
# gives the bytes and values of the one-warp-per-unit settings
@pytest.mark.parametrize("N,nlev,nsingle", [(8, 1, 1), (24, 5, 3), (160, 9, 2), (320, 8, 4)])
def test_batch_defaults(N, nlev, nsingle):
    north = 20 + 4 * np.arange(N)
    lens = np.concatenate([north, north[::-1]]).tolist()
    g = torch.Generator("cuda").manual_seed(N)
    fields = []
    for k, (lev, dims) in enumerate([(nlev, 3)] * 2 + [(1, 1)] * nsingle):
        f = 250.0 + torch.cumsum(torch.randn((lev, sum(lens)), device="cuda", generator=g), 1) * 0.1
        fields.append((f, torch.zeros_like(f), dims, (8, 16)[k % 2]))
    ref = None
    for settings in (None, (3, 16, 1), (2, 5, 64), (8, 1, 3)):
        b = z.Batch(lens, fields)
        if settings:
            b.set_launch(settings[0])
            b.set_unit_blocks(settings[1])
            b.set_claim_units(settings[2])
        s = torch.zeros(b.nbytes(), dtype=torch.uint8, device="cuda")
        for f in fields:
            f[1].zero_()
        b.encode(s)
        b.decode(s)
        got = [s] + [f[1].clone() for f in fields]
        ref = ref or got
        assert all(torch.equal(a, c) for a, c in zip(got, ref))
        b.close()


# the variable-rate chain's launches overlap their predecessors; a replayed
# capture of two encodes and a decode over one scratch gives the eager results
@pytest.mark.parametrize("shape", [(3, 2, 5), (17, 75, 161)])
def test_captured_accuracy_chain(shape):
    n = tuple(reversed(shape))
    r = np.random.default_rng(sum(shape))
    xs = [torch.from_numpy(r.standard_normal(shape).astype(np.float32)).cuda() for _ in range(2)]
    nb = int(np.prod([(k + 3) // 4 for k in n]))
    work = torch.zeros(z.zfpx_accuracy_workspace_bytes(n), dtype=torch.uint8, device="cuda")

    def outputs():
        return [(torch.zeros(nb, dtype=torch.uint16, device="cuda"),
                 torch.full((z.zfpx_accuracy_max_payload_bytes(n),), 255, dtype=torch.uint8, device="cuda"),
                 torch.zeros(1, dtype=torch.int64, device="cuda")) for _ in xs], torch.zeros(shape, device="cuda")

    def chain(outs, d):
        for x, o in zip(xs, outs):
            z.zfpx_encode_accuracy(x, 1e-3, *o, work)
        z.zfpx_decode_accuracy(outs[1][0], outs[1][1], d, work)

    want, dw = outputs()
    got, dg = outputs()
    chain(want, dw)
    chain(got, dg)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    graph = z.capture(lambda: chain(got, dg), st)
    for o in got:
        o[0].zero_(), o[1].fill_(255), o[2].zero_()
    dg.zero_()
    torch.cuda.synchronize()
    graph.launch(st)
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert all(torch.equal(i.view(torch.uint8), j.view(torch.uint8)) for i, j in zip(a, b))
    assert torch.equal(dw.view(torch.int32), dg.view(torch.int32))


# special blocks, partial along every axis, in views with any strides; one more
# unit than a warp per block takes
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 2, 5), (9, 7, 13), (5, 6, 66)])
@pytest.mark.parametrize("rate", [8, 16])
def test_small_arrays_of_any_layout(shape, rate):
    r = np.random.default_rng(rate + sum(shape))
    x = (r.standard_normal(shape) * 10.0 ** r.integers(-44, 38, shape)).astype(np.float32)
    x[r.random(shape) < 0.1] = 0.0
    x[r.random(shape) < 0.01] = np.inf
    x[r.random(shape) < 0.01] = np.nan
    x[r.random(shape) < 0.05] = np.float32(3.4e38)
    n = tuple(reversed(shape))
    ref = oc.encode_array(3, rate, x)
    rd = np.empty_like(x)
    oc.decode_array(3, rate, ref, rd)
    for order, step in (((0, 1, 2), 1), ((2, 1, 0), 1), ((1, 2, 0), 1), ((0, 1, 2), 3)):
        def view(a):                                   # the values in another memory order, `step` apart
            big = torch.full([shape[i] * (step if k == 2 else 1) for k, i in enumerate(order)], 7.0, device="cuda")
            v = big[..., ::step].permute(*[order.index(i) for i in range(3)])
            v.copy_(torch.from_numpy(a))
            return big, v
        _, src = view(x)
        big, dst = view(np.zeros_like(x))
        s = torch.zeros(z.zfpx_stream_bytes(3, rate, n), dtype=torch.uint8, device="cuda")
        z.zfpx_encode(3, rate, src, s)
        z.zfpx_decode(3, rate, s, dst)
        assert s.cpu().numpy().tobytes() == bytes(ref)
        assert np.array_equal(dst.cpu().numpy().view(np.uint32), rd.view(np.uint32))
        if step > 1:
            assert bool((big.view(-1, step)[:, 1:] == 7.0).all())


@pytest.mark.parametrize("rate", [8, 16])
def test_either_side_of_a_warp_per_block(rate):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for units in (14 * sms // 32, 14 * sms // 32 + 1):
        x = np.random.default_rng(units).standard_normal((4, 4 * units, 4 * 32)).astype(np.float32)
        round_trip(x, 3, rate)


# messages shorter than the 2 KB a warp moves at a time, longer, ending inside
# it and inside 16 bytes, and empty ones (more ranks than values)
@pytest.mark.parametrize("n,pr,pc", [((64, 32, 8), 2, 2), ((33, 17, 5), 3, 2), ((130, 67, 21), 2, 3), ((7, 3, 2), 4, 5)])
@pytest.mark.parametrize("rate", [8, 16, z.RATE_F32, z.RATE_F16])
def test_permute_of_any_message_size(n, pr, pc, rate):
    for dims in (1, 3):
        plan = z.Plan(n, pr, pc, 0, dims)
        r = np.random.default_rng(sum(n))
        s = r.integers(0, 256, plan.buffer_bytes(rate), dtype=np.uint8)
        recv = torch.zeros(plan.buffer_bytes(rate), dtype=torch.uint8, device="cuda")
        z.zfpx_permute(plan, rate, torch.from_numpy(s).cuda(), recv)
        want = np.frombuffer(op.permute(opl.Plan(*n, pr, pc, 0, dims), rate, s), np.uint8)
        assert np.array_equal(recv.cpu().numpy(), want)
        plan.close()
