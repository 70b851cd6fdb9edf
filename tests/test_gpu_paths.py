"""Where a call changes kernels, and where code lengths change routes, against the oracle: the edges of the launches that
place their tiles themselves, of the one-cluster relative bound, of the width classes of the decoder and the hop, and of
streams that fill their buffers to the last byte."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_18554_b200 import fields

pytestmark = pytest.mark.gpu
T = 4096


@pytest.fixture(scope="module")
def z():
    from paper_2502_18554_b200 import build, zccl
    build.build()
    return zccl


@pytest.fixture(scope="module")
def ctx(z):
    c = z.Context(1000 * T, 0)
    yield c
    c.close()


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def steps_with_lengths(n, lengths, step, seed):
    """Values on the grid of `step` whose blocks of 32 take the code lengths of `lengths` in turn."""
    rng = np.random.default_rng(seed)
    d = np.zeros(n, np.int64)
    for b in range(0, n, 32):
        top = lengths[(b // 32) % len(lengths)]
        m = min(32, n - b)
        if top:
            mag = rng.integers(0, 1 << top, m)
            mag[rng.integers(0, m)] = (1 << top) - 1
            d[b:b + m] = mag * np.where(np.arange(m) % 2 == 0, 1, -1)   # alternating: the codes stay small
    return (np.cumsum(d) * step).astype(np.float32)


def check(z, ctx, x, mode, eb, local=None, flags=0):
    want, wrc = oracle.compress(x, mode, eb)
    got, rc = z.compress_to_bytes(ctx, dev(x), mode, eb)
    assert rc == wrc and np.array_equal(got.cpu().numpy(), want)
    exact = got.clone()                      # a buffer that ends with the stream
    y, rc = z.decompress_from_bytes(ctx, exact, x.size)
    assert rc == z.OK and np.array_equal(y.cpu().numpy().view(np.uint32), oracle.decompress(want).view(np.uint32))
    if local is None:
        return
    want2, wrc2 = oracle.drc(want, local=local, flags=flags)
    for raw in (None, torch.full((x.size + 8,), 7.0, device="cuda")):
        out = torch.full((z.compress_bound(x.size) + 64,), 0xEE, dtype=torch.uint8, device="cuda")
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        ctx.decompress_reduce_compress(exact, x.size, out[:-64], nb, local=dev(local), raw_out=None if raw is None else raw[: x.size], flags=flags)
        assert ctx.status() == wrc2
        assert np.array_equal(out[: int(nb.item())].cpu().numpy(), want2)
        assert bool((out[-64:] == 0xEE).all()) and (raw is None or bool((raw[x.size:] == 7.0).all()))


@pytest.mark.parametrize("n", [1, 31, 33, T - 1, T, T + 1, 8 * T - 1, 8 * T, 8 * T + 1])
def test_relative_bound_in_one_cluster_and_beyond(z, ctx, n):
    x = fields.smooth_1d(n + 1, seed=n)[:n]
    if n == 1:
        x = np.concatenate([x, -x])
    check(z, ctx, x, oracle.EB_REL, 1e-3)
    out = torch.empty(z.compress_bound(x.size), dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    ctx.compress(dev(x), z.EB_RESOLVED, 0.0, out, nb)      # the bound it left behind
    assert ctx.status() >= 0 and np.array_equal(out[: int(nb.item())].cpu().numpy(), oracle.compress(x, oracle.EB_REL, 1e-3)[0])


def test_relative_bound_without_extent_in_one_cluster(z, ctx):
    x = torch.full((3 * T,), 2.5, device="cuda")
    out = torch.empty(z.compress_bound(x.numel()), dtype=torch.uint8, device="cuda")
    nb = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    ctx.compress(x, z.EB_REL, 1e-3, out, nb)
    assert ctx.status() == z.E_DEGENERATE and int(nb.item()) == 0
    check(z, ctx, fields.smooth_1d(3 * T, seed=4), oracle.EB_REL, 1e-3)


@pytest.mark.parametrize("tiles_per_sm,extra", [(4, 0), (4, 1), (6, 0), (6, 5)])
def test_where_a_launch_stops_placing_its_tiles_itself(z, ctx, tiles_per_sm, extra):
    n = tiles_per_sm * sms() * T + extra
    x, loc = fields.smooth_1d(n, seed=21), fields.smooth_1d(n, seed=22)
    check(z, ctx, x, oracle.EB_ABS, 2e-3, loc)


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("mode", [oracle.EB_ABS, oracle.EB_REL])
def test_where_compressions_change_from_a_tile_per_block_to_many(z, extra, mode):
    """Seven tiles per SM, and one more: of one array, and of four in a launch (there the last tile has one element)."""
    tiles = 7 * sms()
    c = z.Context((tiles + 4) * T, 4)
    x = fields.smooth_1d((tiles + extra) * T, seed=23)
    check(z, c, x, mode, 1e-3)
    n = tiles * T // 4 + extra
    send = [fields.smooth_1d(n, seed=24 + r) for r in range(4)]
    want, wrc, sizes = oracle.sim_allgather(send, mode, 1e-3)
    recv = [torch.full((4 * n + 3,), 7.0, device="cuda") for _ in range(4)]
    for _ in range(2):
        c.sim_allgather([dev(a) for a in send], [r[: 4 * n] for r in recv], mode, 1e-3)
        assert c.status() == wrc and np.array_equal(np.array(c.sim_sizes()), sizes)
        for r in range(4):
            got = recv[r].cpu().numpy()
            assert np.array_equal(got[: 4 * n].view(np.uint32), want[r].view(np.uint32)) and np.all(got[4 * n:] == 7.0)
    c.close()


@pytest.mark.parametrize("lengths", [(0, 7), (7, 8), (8, 9, 0), (15, 3), (15, 16), (16, 17, 1), (20, 0, 5), (4, 5), (12, 13)])
@pytest.mark.parametrize("n", [2 * T, 3 * T - 45])
def test_code_lengths_at_the_edges_of_the_width_classes(z, ctx, lengths, n):
    eb, step = 1e-3, None
    _, s, _ = oracle.resolve(oracle.EB_ABS, eb)
    step = float(s)
    x = steps_with_lengths(n, lengths, step, seed=sum(lengths))
    loc = steps_with_lengths(n, lengths[::-1], step, seed=1 + sum(lengths))
    for flags in (z.OP_SUM, z.OP_MAX, z.OP_MIN):
        check(z, ctx, x, oracle.EB_ABS, eb, loc, flags)


def test_hop_of_a_damaged_stream_writes_inside_its_buffers_and_leaves_the_context_usable(z, ctx):
    n = 5 * T + 7
    x, loc = fields.smooth_1d(n, seed=5), fields.smooth_1d(n, seed=6)
    want, _ = oracle.compress(x, oracle.EB_ABS, 2e-3)
    bad = want.copy()
    bad[32 + 4 * 2: 32 + 4 * 3] = 0xFF                     # one index entry
    out = torch.full((z.compress_bound(n) + 64,), 0xEE, dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    ctx.decompress_reduce_compress(dev(bad), n, out[:-64], nb, local=dev(loc))
    assert ctx.status() == z.E_BAD_STREAM and bool((out[-64:] == 0xEE).all())
    check(z, ctx, x, oracle.EB_ABS, 2e-3, loc)


@pytest.mark.parametrize("N,n,lengths", [(2, 2 * T, (3, 8)), (5, 5 * 2 * T + 3, (8, 9, 0)), (8, 8 * 3 * T, (15, 16, 2)), (16, 16 * T + 32, (7, 6)), (17, 17 * T, (5, 0)),
                                         (3, 3 * 1024 - 7, (20, 1)), (4, 4 * T, (13, 12))])
@pytest.mark.parametrize("op", [0, 2, 4])
def test_ring_steps_of_one_launch_and_of_several(z, N, n, lengths, op):
    eb = 1e-3
    _, s, _ = oracle.resolve(oracle.EB_ABS, eb)
    send = [steps_with_lengths(n, lengths, float(s), seed=7 * r + sum(lengths)) for r in range(N)]
    want, wrc, whop = oracle.sim_allreduce(send, oracle.EB_ABS, eb, flags=op, want_hop_bytes=True)
    c = z.Context(max(n, 2 * T), N)
    base = [torch.full((n + 9,), 7.0, device="cuda") for _ in range(N)]
    recv = [b[1: n + 1] if r % 2 else b[:n] for r, b in enumerate(base)]      # every other rank's buffers off the 16-byte boundary
    ins = [torch.empty(n + 1, device="cuda")[1:].copy_(dev(a)) if r % 3 == 2 else dev(a) for r, a in enumerate(send)]
    for _ in range(2):
        c.sim_allreduce(ins, recv, z.EB_ABS, eb, op)
        assert c.status() == wrc
        for r in range(N):
            assert np.array_equal(recv[r].cpu().numpy().view(np.uint32), want[r].view(np.uint32)), r
            assert bool((base[r][n + 1:] == 7.0).all())
        assert np.array_equal(np.array(c.sim_sizes()).reshape(N, N), whop)
    c.close()


@pytest.mark.parametrize("N,n,lengths", [(2, 2 * T, (3, 8)), (3, 3 * 1024 - 7, (20, 1)), (5, 5 * 2 * T + 3, (8, 9, 0)), (8, 8 * 35 * T + 77, (15, 16, 2)),
                                         (16, 16 * T + 32, (7, 6))])
@pytest.mark.parametrize("op", [0, 2, 4])
def test_ring_steps_of_one_launch_leave_the_streams_of_every_step(z, N, n, lengths, op):
    """The launch decodes none of the streams it writes, so they are compared themselves: header, index, every tile's place."""
    eb = 1e-3
    _, s, _ = oracle.resolve(oracle.EB_ABS, eb)
    send = [steps_with_lengths(n, lengths, float(s), seed=11 * r + sum(lengths)) for r in range(N)]
    m = -(-n // N)
    part = lambda r, ch: send[r][ch * m: min(n, (ch + 1) * m)]
    want = [[oracle.compress(part(r, (r - 1) % N), oracle.EB_ABS, eb)[0] for r in range(N)]]
    for k in range(1, N):
        steps = [oracle.drc(want[k - 1][(r - 1) % N], local=part(r, (r - k - 1) % N), flags=op, want_raw=True) for r in range(N)]
        want.append([st[0] for st in steps])
    c = z.Context(max(n, 2 * T), N)
    slot = z.compress_bound(m)
    recv = [torch.full((m + 3,), 7.0, device="cuda") for _ in range(N)]
    for _ in range(2):
        streams = torch.full((N * N * slot,), 0xEE, dtype=torch.uint8, device="cuda")
        sizes = torch.zeros(N * N, dtype=torch.int64, device="cuda")
        c.debug_ring_streams([dev(a) for a in send], recv, z.EB_ABS, eb, op, streams, slot, sizes)
        assert c.status() >= 0
        got, lengths_got = streams.cpu().numpy().reshape(N, N, slot), sizes.cpu().numpy().reshape(N, N)
        for k in range(N):
            for r in range(N):
                assert lengths_got[k, r] == want[k][r].size and np.array_equal(got[k, r, : want[k][r].size], want[k][r]), (k, r)
                assert bool((got[k, r, want[k][r].size:] == 0xEE).all()), (k, r)
        for r in range(N):
            sums = steps[r][2]
            assert np.array_equal(recv[r][: sums.size].cpu().numpy().view(np.uint32), sums.view(np.uint32)) and bool((recv[r][sums.size:] == 7.0).all())
    c.close()


@pytest.mark.parametrize("N", [3, 4])
def test_where_the_ring_stops_being_one_launch(z, N):
    """On both sides of as many tiles as CTAs of the ring's launch are resident together (four per SM)."""
    most = 4 * sms()
    whole = most // N * N * T                              # every chunk a whole number of tiles
    launches = []
    c = z.Context(whole + N * T, N)
    for n in (whole, whole + 1):                           # one more element: a tile more per chunk
        send = [fields.smooth_1d(n, seed=r) for r in range(N)]
        want, wrc, whop = oracle.sim_allreduce(send, oracle.EB_ABS, 2e-3, want_hop_bytes=True)
        recv = [torch.zeros(n, device="cuda") for _ in range(N)]
        before = z.launch_count()
        c.sim_allreduce([dev(a) for a in send], recv, z.EB_ABS, 2e-3)
        launches.append(z.launch_count() - before)
        assert c.status() == wrc and np.array_equal(np.array(c.sim_sizes()).reshape(N, N), whop)
        for r in range(N):
            assert np.array_equal(recv[r].cpu().numpy().view(np.uint32), want[r].view(np.uint32)), r
    assert launches[0] == 2 and launches[1] > N            # the ring and the decoding; a launch per step and more
    c.close()


@pytest.mark.parametrize("bits", [(3, 9, 17, 28), (29, 2, 14, 15), (16, 16, 16, 16), (0, 0, 15, 0), (15, 15, 15, 14), (7, 8, 7, 8)])
@pytest.mark.parametrize("n", [4096, 3 * 4096 + 1025, 8191])
@pytest.mark.parametrize("shift", [0, 1])
def test_binary64_rounds_of_mixed_widths(z, ctx, bits, n, shift):
    """Code lengths that change from round to round of a tile: width classes, general rounds beside short ones, blobs on
    both sides of what the decoder's buffer holds; with and without a 16-byte boundary."""
    rng = np.random.default_rng(sum(bits) + n)
    amp = np.array([2.0 ** b for b in bits])[(np.arange(n) // 1024) % 4]
    x = rng.uniform(-0.5, 0.5, n) * amp
    want = oracle.compress_f64(x, 0, 0.5)
    dx = torch.zeros(n + 1, dtype=torch.float64, device="cuda")[shift : shift + n]
    dx.copy_(torch.from_numpy(x))
    out = torch.empty(z.compress_bound(n), dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    ctx.compress_f64(dx, 0, 0.5, out, nb)
    assert ctx.status() == z.OK
    got = out[: int(nb.item())]
    assert np.array_equal(got.cpu().numpy(), want)
    y = torch.zeros(n + 1, dtype=torch.float64, device="cuda")[shift : shift + n]
    ctx.decompress_f64(got, y)
    assert ctx.status() == z.OK
    assert np.array_equal(y.cpu().numpy().view(np.uint64), oracle.decompress_f64(want).view(np.uint64))


@pytest.mark.parametrize("lengths", [(1,), (10, 11), (11, 12), (13, 14), (16, 17, 0), (15, 3)])
def test_placement_of_payloads_on_both_sides_of_what_is_staged(z, ctx, lengths):
    """Two launches, hops of more tiles than four per SM and compressions of binary64: the placement brings 1536 payload words of
    a tile by bulk copies and the rest by loads."""
    n = (4 * sms() + 33) * T + 1029
    eb = 1e-3
    # (pieces of a tile: the codes of a long walk in such steps would leave their range; a tile's first step is what it has to be)
    def walk(count, step):
        pieces = [steps_with_lengths(T, lengths, 1.0, seed=sum(lengths) + k).astype(np.float64) * step for k in range(12)]
        return np.concatenate([pieces[k] for k in np.random.default_rng(1).integers(0, 12, count // T + 1)])[:count]
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    x = walk(n, float(oracle.resolve(oracle.EB_ABS, eb)[1])).astype(np.float32)
    src, _ = oracle.compress(np.zeros(n, np.float32), oracle.EB_ABS, eb)      # the sum is x, and so are its code lengths
    want, wrc = oracle.drc(src, local=x)
    dx, ds, out = dev(x), dev(src), torch.empty(z.compress_bound(n), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        ctx.decompress_reduce_compress(ds, n, out, nb, local=dx)
        assert ctx.status() == wrc
        assert np.array_equal(out[: int(nb.item())].cpu().numpy(), want)
    n = 167 * T + 1029                                                       # six groups of 32 tiles
    x = walk(n, oracle.resolve_f64(0, eb)[1])
    want, dx = oracle.compress_f64(x, 0, eb), dev(x)
    for _ in range(2):
        ctx.compress_f64(dx, 0, eb, out, nb)
        assert ctx.status() == z.OK
        assert np.array_equal(out[: int(nb.item())].cpu().numpy(), want)


@pytest.mark.parametrize("tiles", [2, 9, 33, 500])
def test_tiles_are_taken_in_the_order_in_which_blocks_start(z, tiles):
    """A launch that places its tiles itself: every block takes its tile from its array's counter when it starts, whichever tile
    comes first, and the counter is back at 0 when all have one, launch behind launch."""
    n = tiles * T - 100
    N = 2
    c = z.Context(N * n, N)
    x, loc = fields.smooth_1d(n, seed=tiles), fields.smooth_1d(n, seed=tiles + 1)
    want, _ = oracle.compress(x, oracle.EB_ABS, 2e-3)
    want2, _ = oracle.drc(want, local=loc)
    sums, _ = oracle.sim_allreduce([x, loc], oracle.EB_ABS, 2e-3)
    dx, dl = dev(x), dev(loc)
    out, out2 = (torch.zeros(z.compress_bound(n), dtype=torch.uint8, device="cuda") for _ in range(2))
    nb = torch.zeros(2, dtype=torch.int64, device="cuda")
    recv = [torch.zeros(n, device="cuda") for _ in range(N)]
    for first in (0, 1, tiles // 2, tiles - 1):
        in_chunk = first % (tiles // N)
        c.debug_first_tile(first)
        c.compress(dx, z.EB_ABS, 2e-3, out, nb[:1])
        c.decompress_reduce_compress(out, n, out2, nb[1:], local=dl)
        assert c.status() == z.OK and c.debug_tile_counters(1) == [0]
        c.debug_first_tile(in_chunk)
        c.sim_allreduce([dx, dl], recv, z.EB_ABS, 2e-3)
        assert c.status() == z.OK and c.debug_tile_counters(N) == [0] * N
        assert np.array_equal(out[: int(nb[0].item())].cpu().numpy(), want)
        assert np.array_equal(out2[: int(nb[1].item())].cpu().numpy(), want2)
        for r in range(N):
            assert np.array_equal(recv[r].cpu().numpy().view(np.uint32), sums[r].view(np.uint32))
    c.close()


@pytest.mark.parametrize("extra", [-1, 0, 7])
def test_tiles_of_large_decompressions_dealt_out_by_a_counter(z, extra):
    """From 16 tiles per CTA (five per SM) on: every tile is decoded once, launch after launch, the counter being back where it
    was; the same where several streams of a launch are forwarded, and behind a damaged stream."""
    tiles = 16 * 5 * sms() + extra
    n = tiles * T - 99
    eb = 1e-3
    _, s, _ = oracle.resolve(oracle.EB_ABS, eb)
    rng = np.random.default_rng(extra + 2)
    kinds = [steps_with_lengths(T, (k, max(k - 1, 0)), float(s), seed=k) for k in (0, 3, 9, 15, 16)]
    x = np.concatenate([kinds[k] for k in rng.choice(5, tiles, p=(0.2, 0.5, 0.2, 0.08, 0.02))])[:n]
    want, _ = oracle.compress(x, oracle.EB_ABS, eb)
    ref = oracle.decompress(want).view(np.uint32)
    c = z.Context(n, 2)
    stream = dev(want)
    y = torch.full((n + 9,), 7.0, device="cuda")
    for shift in (0, 1, 0):
        y.fill_(7.0)
        c.decompress(stream, y[shift: n + shift])
        assert c.status() == z.OK and bool((y[n + shift:] == 7.0).all())
        assert np.array_equal(y[shift: n + shift].cpu().numpy().view(np.uint32), ref)
    bad = want.copy()
    bad[32 + 4 * 100: 32 + 4 * 101] = 0xFF                     # one index entry: two tiles without a blob
    c.decompress(dev(bad), y[:n])
    assert c.status() == z.E_BAD_STREAM
    half = n // 2
    parts = [dev(x[:half]), dev(x[n - half:])]
    recv = [torch.zeros(2 * half, device="cuda") for _ in range(2)]
    refs = [oracle.decompress(oracle.compress(p, oracle.EB_ABS, eb)[0]).view(np.uint32) for p in (x[:half], x[n - half:])]
    for _ in range(2):
        c.sim_allgather(parts, recv, z.EB_ABS, eb)
        assert c.status() >= 0
        for r in range(2):
            assert np.array_equal(recv[r][(1 - r) * half: (2 - r) * half].cpu().numpy().view(np.uint32), refs[1 - r])
    c.close()


@pytest.mark.parametrize("lengths", [(0,), (1,), (7, 8), (9, 10, 11), (15, 16), (16, 17, 0), (22, 3), (24,)])
@pytest.mark.parametrize("shift", [0, 1])
def test_large_compressions_in_one_launch(z, lengths, shift):
    """Beyond seven tiles per SM a CTA takes tile after tile: payloads wait in the warps' rings (code lengths up to 16) or in the
    stage they came in (beyond); with and without the copy engine; launch behind launch; a buffer that is too small."""
    n = (7 * sms() + 700) * T + 1029
    eb = 1e-3
    _, s, _ = oracle.resolve(oracle.EB_ABS, eb)
    # (pieces of a tile: the codes of a long walk in such steps would leave their range)
    pieces = [steps_with_lengths(T, lengths[k % len(lengths):] + lengths[:k % len(lengths)], float(s), seed=k + shift) for k in range(12)]
    x = np.concatenate([pieces[k] for k in np.random.default_rng(shift).integers(0, 12, n // T + 1)])[:n]
    want, wrc = oracle.compress(x, oracle.EB_ABS, eb)
    c = z.Context(n, 0)
    dx = torch.zeros(n + 1, device="cuda")[shift: n + shift]
    dx.copy_(torch.from_numpy(x))
    cap = z.compress_bound(n)
    out = torch.full((cap + 64,), 0xEE, dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    for _ in range(2):
        out.fill_(0xEE)
        c.compress(dx, z.EB_ABS, eb, out[:cap], nb)
        assert c.status() == wrc and int(nb.item()) == want.size
        assert np.array_equal(out[: want.size].cpu().numpy(), want) and bool((out[want.size:] == 0xEE).all())
    short = (want.size * 3 // 4) & ~3
    if short >= 32 + 4 * (n // T + 1):
        out.fill_(0xEE)
        c.compress(dx, z.EB_ABS, eb, out[:short], nb)
        assert c.status() == z.E_CAPACITY and bool((out[short:] == 0xEE).all())
    c.close()


@pytest.mark.parametrize("N,tiles", [(1, 1100), (3, 500), (8, 150)])
def test_large_allgathers_compress_in_one_launch(z, N, tiles):
    """Several arrays of different streams in such a launch, each with the copy of a rank's own contribution."""
    n = tiles * T - 77
    send = [fields.smooth_1d(n, seed=50 + r) for r in range(N)]
    c = z.Context(N * n, max(N, 2))
    recv = [torch.full((N * n,), 7.0, device="cuda") for _ in range(N)]
    for _ in range(2):
        c.sim_allgather([dev(a) for a in send], recv, z.EB_REL, 1e-3)
        assert c.status() >= 0
    want, _, _ = oracle.sim_allgather(send, oracle.EB_REL, 1e-3)
    for r in range(N):
        assert np.array_equal(recv[r].cpu().numpy().view(np.uint32), want[r].view(np.uint32)), r
    c.close()


@pytest.mark.parametrize("value", [3.25, float("inf")])
@pytest.mark.parametrize("N,n", [(1, 1), (2, 1029), (3, 300 * T + 7), (1, 1100 * T), (3, 500 * T - 77), (8, 150 * T + 1030), (33, 33 * T + 5)])
def test_allgathers_without_a_range_keep_their_own_contributions(z, N, n, value):
    """A relative bound on constant arrays is reported; every rank's own contribution arrives all the same, whichever launch it
    goes along with, and nothing beyond the buffers is touched.  The next call is in order."""
    c = z.Context(N * n, max(N, 2))
    send = [torch.full((n,), value, device="cuda") for _ in range(N)]
    recv = [torch.full((N * n + 3,), 7.0, device="cuda") for _ in range(N)]
    for _ in range(2):
        c.sim_allgather(send, [r[:N * n] for r in recv], z.EB_REL, 1e-3)
        assert c.status() == z.E_DEGENERATE
        for r in range(N):
            assert bool((recv[r][r * n: (r + 1) * n] == value).all()) and bool((recv[r][N * n:] == 7.0).all())
    send = [dev(fields.smooth_1d(n, seed=r)) for r in range(N)]
    c.sim_allgather(send, [r[:N * n] for r in recv], z.EB_ABS, 1e-3)
    assert c.status() >= 0
    for r in range(N):
        assert torch.equal(recv[r][r * n: (r + 1) * n], send[r]) and bool((recv[r][N * n:] == 7.0).all())
        for k in range(N):
            assert float((recv[r][k * n: (k + 1) * n] - send[k]).abs().max()) <= 1e-3
    c.close()


def test_large_compressions_wait_with_a_limit_and_their_launch_counter_wraps(z):
    n = (7 * sms() + 300) * T - 5
    x = fields.smooth_1d(n, seed=4)
    want, _ = oracle.compress(x, oracle.EB_REL, 1e-3)
    c = z.Context(n, 0)
    dx, cap = dev(x), z.compress_bound(n)
    out = torch.full((cap + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    c.debug_skip_publish(n // T // 2)
    c.compress(dx, z.EB_REL, 1e-3, out[:cap], nb)
    assert c.status() == z.E_TIMEOUT and bool((out[cap:] == 0x5A).all())
    c.debug_skip_publish(-1)
    c.debug_set_launch_counter(0x7FFFFFFF - 1)
    for _ in range(4):
        out.fill_(0)
        c.compress(dx, z.EB_REL, 1e-3, out[:cap], nb)
        assert c.status() >= 0 and np.array_equal(out[: int(nb.item())].cpu().numpy(), want)
    c.close()


@pytest.mark.parametrize("tiles", [-300, 150, 900])
def test_headers_of_large_compressions_stored_late(z, tiles):
    """Storing warps that come to their first tile only when every tile of the launch has been placed, and the range keys have
    gone back to their start: the header still has the launch's bound.  (Below seven tiles per SM nothing rests.)"""
    n = (7 * sms() + tiles) * T + 9
    x = fields.smooth_1d(n, seed=18)
    want, _ = oracle.compress(x, oracle.EB_REL, 1e-3)
    c = z.Context(n, 2)
    dx, out = dev(x), torch.zeros(z.compress_bound(n), dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    c.debug_store_pause(1000)
    for _ in range(2):
        out.zero_()
        c.compress(dx, z.EB_REL, 1e-3, out, nb)
        assert c.status() >= 0 and np.array_equal(out[: int(nb.item())].cpu().numpy(), want)
    half = n // 2
    parts = [x[:half], x[n - half:]]
    recv = [torch.zeros(2 * half, device="cuda") for _ in range(2)]
    c.sim_allgather([dev(p) for p in parts], recv, z.EB_REL, 1e-3)
    assert c.status() >= 0
    ref, _, _ = oracle.sim_allgather(parts, oracle.EB_REL, 1e-3)
    for r in range(2):
        assert np.array_equal(recv[r].cpu().numpy().view(np.uint32), ref[r].view(np.uint32))
    c.compress(torch.full((n,), 3.25, device="cuda"), z.EB_REL, 1e-3, out, nb)
    assert c.status() == z.E_DEGENERATE and int(nb.item()) == 0
    c.debug_store_pause(0)
    c.compress(dx, z.EB_REL, 1e-3, out, nb)
    assert c.status() >= 0 and np.array_equal(out[: int(nb.item())].cpu().numpy(), want)
    c.close()


def test_large_compressions_one_behind_the_other(z):
    """Enqueued without a wait on the host: with absolute bounds the blocks of the launch behind take the places of those that
    have left, and their first tiles' numbers; other launches stand in between and behind."""
    sizes = [(7 * sms() + 1) * T, 2600 * T - 3, (7 * sms() + 600) * T + 5, 900 * T, 1700 * T]
    xs = [fields.smooth_1d(n, seed=60 + k) for k, n in enumerate(sizes)]
    c = z.Context(max(sizes), 0)
    dx = [dev(x) for x in xs]
    calls = [(0, "abs"), (1, "abs"), (2, "abs"), (2, "rel"), (1, "abs"), (3, "abs"), (4, "abs"), (0, "abs"), (1, "hop"), (4, "abs"), (2, "rel"), (2, "abs"), (1, "abs")]
    want = {("abs", k): oracle.compress(x, oracle.EB_ABS, 1e-3)[0] for k, x in enumerate(xs)}
    want["rel", 2] = oracle.compress(xs[2], oracle.EB_REL, 1e-3)[0]
    want["hop", 1] = oracle.drc(want["abs", 1], local=xs[1])[0]
    src = dev(want["abs", 1])
    res = []
    for rep in range(2):
        torch.cuda.synchronize()
        for k, what in calls:
            out, nb = torch.zeros(z.compress_bound(sizes[k]) // 2, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
            y = torch.zeros(sizes[k], device="cuda")
            res.append((k, what, out, nb, y))
        torch.cuda.synchronize()
        for i, (k, what, out, nb, y) in enumerate(res[rep * len(calls):]):
            if what == "hop":
                c.decompress_reduce_compress(src, sizes[k], out, nb, local=dx[k])
            else:
                c.compress(dx[k], z.EB_ABS if what == "abs" else z.EB_REL, 1e-3, out, nb)
            if rep and i % 3 == 1:
                c.decompress(out, y)
        assert c.status() >= 0
    for i, (k, what, out, nb, y) in enumerate(res):
        assert np.array_equal(out[: int(nb.item())].cpu().numpy(), want[what, k]), (i, k, what)
        if i >= len(calls) and (i - len(calls)) % 3 == 1:
            assert np.array_equal(y.cpu().numpy().view(np.uint32), oracle.decompress(want[what, k]).view(np.uint32)), (i, k, what)
    c.close()


def test_two_contexts_on_two_streams_run_large_compressions_side_by_side(z):
    """Two large compressions do not fit the device together, their blocks wait for sizes of their own launch, and each launch's
    numbers and places are its context's: whichever share of the device each gets, both give the oracle's streams."""
    sizes = [(7 * sms() + 900) * T + 77, 3000 * T]
    ctxs, streams = [z.Context(n, 0) for n in sizes], [torch.cuda.Stream(), torch.cuda.Stream()]
    xs = [fields.smooth_1d(n, seed=80 + k) for k, n in enumerate(sizes)]
    modes = [oracle.EB_ABS, oracle.EB_REL]
    want = [[oracle.compress(x, m, 1e-3)[0] for m in modes] for x in xs]
    dx = [dev(x) for x in xs]
    out = [[torch.zeros(z.compress_bound(n) // 2, dtype=torch.uint8, device="cuda") for _ in range(8)] for n in sizes]
    nb = [[torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(8)] for _ in sizes]
    torch.cuda.synchronize()
    for rep in range(8):
        for k in range(2):
            with torch.cuda.stream(streams[k]):
                ctxs[k].compress(dx[k], modes[(rep >> 1) & 1], 1e-3, out[k][rep], nb[k][rep], stream=streams[k])
    torch.cuda.synchronize()
    for k in range(2):
        assert ctxs[k].status() >= 0
        for rep in range(8):
            assert np.array_equal(out[k][rep][: int(nb[k][rep].item())].cpu().numpy(), want[k][(rep >> 1) & 1]), (k, rep)
        ctxs[k].close()


@pytest.mark.parametrize("N,n", [(5, 16), (8, 5), (8, 11), (33, 64), (40, 70)])
@pytest.mark.parametrize("late", [0, 1000])
def test_chunks_without_elements_whose_blocks_come_late(z, N, n, late):
    """Collectives whose last chunks have no elements: their blocks need the launch's bound too (it goes into their headers), also
    when all others are through by then.  In a reduce-scatter the first rank's is such a chunk."""
    c = z.Context(max(n, 64), N)
    send = [fields.smooth_1d(n, seed=90 + r) for r in range(N)]
    ds = [dev(a) for a in send]
    want, wrc, whop = oracle.sim_allreduce(send, oracle.EB_REL, 1e-3, want_hop_bytes=True)
    want_rs, wrc_rs, whop_rs = oracle.sim_reduce_scatter(send, oracle.EB_REL, 1e-3)
    c.debug_store_pause(late)
    for counter in (0, 0x7FFFFFFF - 1, 0):
        if counter:
            c.debug_set_launch_counter(counter)
        recv = [torch.full((n + 8,), 7.0, device="cuda") for _ in range(N)]
        c.sim_allreduce(ds, [r[:n] for r in recv], z.EB_REL, 1e-3)
        assert c.status() == wrc
        assert np.array_equal(np.array(c.sim_sizes()).reshape(N, N), whop)
        for r in range(N):
            got = recv[r].cpu().numpy()
            assert np.array_equal(got[:n].view(np.uint32), want[r].view(np.uint32)) and np.all(got[n:] == 7.0), r
        recv = [torch.full((want_rs[r].size + 8,), 7.0, device="cuda") for r in range(N)]
        c.sim_reduce_scatter(ds, recv, z.EB_REL, 1e-3)
        assert c.status() == wrc_rs
        assert np.array_equal(np.array(c.sim_sizes()).reshape(N - 1, N), whop_rs)
        for r in range(N):
            got = recv[r].cpu().numpy()
            assert np.array_equal(got[:want_rs[r].size].view(np.uint32), want_rs[r].view(np.uint32)) and np.all(got[want_rs[r].size:] == 7.0), r
    c.close()


@pytest.mark.parametrize("leave,skip,counter", [(0, 0, 0), (0, 3000, 0), (0, 3000, 0x7FFFFFFF), (1, None, 0), (2, None, 0), (3, None, 0x7FFFFFFF), (9, None, 0), (9, 100, 0), (12, None, 0)])
def test_large_compressions_whose_waits_run_out_leave_the_next_in_order(z, leave, skip, counter):
    """More tiles per block than its queue of eight holds: places that never come, and warps that leave in the middle of a block's
    tiles.  Nothing is written beyond the buffers, and the next launches are in order without anything put back by hand."""
    n = 50 * sms() * T + 77                     # (over twelve tiles per block)
    x = fields.smooth_1d(n, seed=21)
    want, _ = oracle.compress(x, oracle.EB_REL, 1e-3)
    c = z.Context(n, 3)
    dx, cap = dev(x), z.compress_bound(n)
    out = torch.full((cap + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    m = n // 3
    send = [dx[k * m: (k + 1) * m] for k in range(3)]
    recv = [torch.full((3 * m,), 7.0, device="cuda") for _ in range(3)]
    for several in (False, True, False):
        if counter:
            c.debug_set_launch_counter(counter)
        c.debug_leave_before(leave)
        c.debug_skip_publish(-1 if skip is None else skip)
        if several:                             # three arrays in one launch (the streams that are missing are refused behind it)
            c.sim_allgather(send, recv, z.EB_REL, 1e-3)
        else:
            c.compress(dx, z.EB_REL, 1e-3, out[:cap], nb)
        assert c.status() == z.E_TIMEOUT and bool((out[cap:] == 0x5A).all())
        c.debug_leave_before(0)
        c.debug_skip_publish(-1)
        for _ in range(2):
            out[:cap].fill_(0)
            c.compress(dx, z.EB_REL, 1e-3, out[:cap], nb)
            assert c.status() >= 0 and int(nb.item()) == want.size
            assert np.array_equal(out[: want.size].cpu().numpy(), want) and bool((out[cap:] == 0x5A).all())
    c.close()


def test_large_compressions_without_a_range(z):
    """A constant array has no range: an empty result, reported, and the next call is in order."""
    n = (7 * sms() + 150) * T + 9
    x = fields.smooth_1d(n, seed=8)
    want, _ = oracle.compress(x, oracle.EB_REL, 1e-3)
    c = z.Context(n, 0)
    out, nb = torch.zeros(z.compress_bound(n), dtype=torch.uint8, device="cuda"), torch.full((1,), 5, dtype=torch.int64, device="cuda")
    for _ in range(2):
        c.compress(torch.full((n,), 3.25, device="cuda"), z.EB_REL, 1e-3, out, nb)
        assert c.status() == z.E_DEGENERATE and int(nb.item()) == 0
        c.compress(dev(x), z.EB_REL, 1e-3, out, nb)
        assert c.status() >= 0 and np.array_equal(out[: int(nb.item())].cpu().numpy(), want)
    c.close()


def test_large_allocation_free_compressions(z):
    """The allocation-free entry point beyond seven tiles per SM, which has no slots."""
    n = (7 * sms() + 200) * T + 33
    _, s, _ = oracle.resolve(oracle.EB_ABS, 1e-3)
    x = steps_with_lengths(n, (3, 16, 19, 0), float(s), seed=1)
    want, _ = oracle.compress(x, oracle.EB_ABS, 1e-3)
    dx, out = dev(x), torch.zeros(z.compress_bound(n), dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    for _ in range(2):
        z.compress_noalloc(dx, 1e-3, out, nb)
        assert np.array_equal(out[: int(nb.item())].cpu().numpy(), want)
