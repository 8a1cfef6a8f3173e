"""GPU parity of the one-pass compression (near rows exactly, far rows by interpolation) at the edges of its tiles, against
the fp64 CPU oracle.  Its own error beside the roundings, in 64 bits over ratios of 1 to 30, is at most 3.5e-4 of a row and
1.5e-4 of the matrix with 4 nodes a tile, 1.3e-4 and 6e-5 with 6, 1e-4 and 3e-5 with 8.  So the bounds of the other bf16 paths
hold unchanged: 1e-2 a matrix, 3e-2 a row."""
import math

import pytest
import torch

from paper_2505_00570_b200 import binding as fk
from paper_2505_00570_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = fk.Context(0)
    yield c
    c.close()


def workload(cap, sink, B=1, Ly=1, H=2, rho=0.9):
    return synth.Workload("t", B, Ly, H, 128, cap, torch.bfloat16, sink, rho, 2, synth.BASE_SEED + 11)


# kept rows: two tiles and a row, three whole tiles; 16 and 17 tiles (8 and 6 nodes each), 21 and 22 (6 and 4), 33 (two blocks
# of far rows); nearly all rows kept (a tile then writes rows the next one reads); a wide window (one row in 30)
@pytest.mark.parametrize("n_in,kept,sink", [(514, 257, 4), (1001, 384, 0), (2731, 2048, 4), (3000, 2049, 1), (5376, 2688, 4),
                                            (3001, 2689, 0), (4500, 4097, 4), (300, 299, 2), (1500, 1409, 4), (8000, 267, 4)])
def test_edges_of_the_tiles(ctx, n_in, kept, sink):
    parity.check_compress(ctx, workload(n_in + sink + 3, sink), n_in + sink, kept, sink, fk.GEMM)
    parity.check_compress(ctx, workload(n_in + sink + 3, sink, rho=0.0), n_in + sink, kept, sink, fk.GEMM, row_pad=8, sample=2)


@pytest.mark.parametrize("n_in,kept", [(1028, 514), (700, 650), (3001, 749)])
def test_many_groups_repeat_bit_for_bit(ctx, n_in, kept):
    """More groups of channels than the ring of far sums has places; the tiles of all CTAs overwrite each other's input in
    place, and the result is the same every time, and that of each matrix pair alone."""
    w = workload(n_in + 4, 4, B=2, Ly=9, H=13)
    k0, v0 = synth.make_cache(w, "cuda")
    ctx.set_variant(fk.AUTO)
    first = None
    for _ in range(6):
        k, v = k0.clone(), v0.clone()
        ctx.compress(k, v, n_in + 4, kept, 4)
        if first is None:
            first = (k, v)
        assert torch.equal(k, first[0]) and torch.equal(v, first[1])
    assert ctx.last_device_status() == fk.OK
    for b, layer, h in ((0, 0, 0), (1, 8, 12), (1, 3, 7)):
        k, v = k0[b:b + 1, layer:layer + 1, h:h + 1].clone(), v0[b:b + 1, layer:layer + 1, h:h + 1].clone()
        ctx.compress(k, v, n_in + 4, kept, 4)
        assert torch.equal(k[0, 0, 0], first[0][b, layer, h]) and torch.equal(v[0, 0, 0], first[1][b, layer, h])


def test_ragged_batch_of_different_ranks(ctx):
    """Sequences of 8, 6 and 4 nodes a tile in one launch, each as on its own, bit for bit."""
    lens, kept = [1300, 4500, 5200, 700], [640, 2500, 2900, 690]
    w = workload(5200, 4, B=4, Ly=2, H=3)
    k0, v0 = synth.make_cache(w, "cuda")
    ctx.set_variant(fk.AUTO)
    k, v = k0.clone(), v0.clone()
    ctx.compress_ragged(k, v, lens, kept, 4)
    assert ctx.last_device_status() == fk.OK
    for b, (n, m) in enumerate(zip(lens, kept)):
        one_k, one_v = k0[b:b + 1].clone(), v0[b:b + 1].clone()
        ctx.compress(one_k, one_v, n, m, 4)
        assert torch.equal(one_k[0], k[b]) and torch.equal(one_v[0], v[b]), b


def test_a_long_sequence_among_short_ones():
    """Sixteen blocks of far rows beside sequences of one: the work area is hardly larger than that of the long sequence alone, and
    every sequence comes out as on its own, bit for bit."""
    lens, kept = [600] * 32, [300] * 32
    lens[5], kept[5] = 131072, 65536
    k0 = torch.zeros(32, 1, 1, 131072, 128, device="cuda", dtype=torch.bfloat16)
    for b, n in enumerate(lens):
        k0[b, :, :, :n].normal_()
    k, v = k0.clone(), k0.clone()
    one_k, one_v = k0[5:6].clone(), k0[5:6].clone()
    spare = torch.zeros(4, 1, 1, 600, 128, device="cuda", dtype=torch.bfloat16)
    c = fk.Context(0)
    c.compress_ragged(spare, spare.clone(), [600, 560, 580, 600], [300, 270, 290, 300], 0)    # loads the kernels
    c.close()
    used = []
    for _ in range(2):
        c = fk.Context(0)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        if not used:
            c.compress(one_k, one_v, 131072, 65536, 0)
        else:
            c.compress_ragged(k, v, lens, kept, 0)
        assert c.last_device_status() == fk.OK
        used.append(before - torch.cuda.mem_get_info()[0])
        c.close()
    assert torch.equal(one_k[0], k[5]) and torch.equal(one_v[0], v[5])
    c = fk.Context(0)
    try:
        for b in (0, 4, 6, 31):
            one_k, one_v = k0[b:b + 1].clone(), k0[b:b + 1].clone()
            c.compress(one_k, one_v, 600, 300, 0)
            assert torch.equal(one_k[0], k[b]) and torch.equal(one_v[0], v[b]), b
    finally:
        c.close()
    print(used)
    assert used[1] < used[0] + (800 << 20)     # four places of 180 MB instead of one


def test_ragged_calls_in_turn(ctx):
    """Ragged calls of other lengths, sinks, layouts and caches one after the other, with nothing waited for in between: the tables
    of each call lie where those of the call before lay.  Every sequence as on its own, bit for bit."""
    ctx.set_variant(fk.AUTO)
    calls = []
    for i, (cap, sink, lens) in enumerate([(2100, 4, [2100, 700, 1300]), (1500, 0, [601, 1500]), (2100, 1, [999, 2048, 2100]),
                                           (1600, 4, [1600, 1200, 900, 1500, 600, 1001])] * 2):
        w = workload(cap, sink, B=len(lens), Ly=2, H=2 + i % 3)
        k, v = synth.make_cache(w, "cuda")
        if i % 2:  # rows 8 elements apart from the next
            k, v = (torch.nn.functional.pad(t, (0, 8))[..., :128] for t in (k, v))
        calls.append((k, v, k.clone(), v.clone(), lens, [(n - sink) // 2 for n in lens], sink))
        for n, m in zip(lens, calls[-1][5]):
            ctx.plan(n - sink, m, fk.BF16, fk.GEMM)
    torch.cuda.synchronize()
    for k, v, _, _, lens, kept, sink in calls:
        ctx.compress_ragged(k, v, lens, kept, sink)
    assert ctx.last_device_status() == fk.OK
    for k, v, k0, v0, lens, kept, sink in calls:
        for b, (n, m) in enumerate(zip(lens, kept)):
            one_k, one_v = k0[b:b + 1].clone(), v0[b:b + 1].clone()
            ctx.compress(one_k, one_v, n, m, sink)
            assert torch.equal(one_k[0], k[b]) and torch.equal(one_v[0], v[b]), (lens, b)


# heads of 64: an odd number of triples leaves the last group half empty; the fewest calls of the one-pass kernel on 148 SMs
# are 10 triples with heads of 64 and 3 with heads of 256
@pytest.mark.parametrize("hd,B,Ly,H,n_in,kept", [(64, 1, 1, 11, 990, 495), (64, 1, 1, 19, 2046, 1023), (64, 3, 1, 7, 1024, 512),
                                                 (64, 1, 2, 5, 2044, 1533), (256, 1, 3, 1, 3000, 1500), (256, 1, 2, 5, 1024, 512)])
def test_other_head_sizes(ctx, hd, B, Ly, H, n_in, kept):
    """Heads of 64 channels (two matrix pairs a group) and of 256 (one matrix a group), in calls large enough for the one-pass
    kernel: against the oracle, and more accurate than the fast transform."""
    w = synth.Workload("t", B, Ly, H, hd, n_in + 7, torch.bfloat16, 4, 0.9, 2, synth.BASE_SEED + 12)
    lay = fk.layout_contiguous(fk.BF16, B, Ly, H, n_in + 7, hd)[1]
    ctx.set_variant(fk.AUTO)
    assert ctx.resolve_variant(lay, n_in, kept) == fk.FDCT
    err = parity.check_compress(ctx, w, n_in + 4, kept, 4, fk.AUTO, sample=8)
    before = ctx.get_timing()[2]
    parity.check_compress(ctx, w, n_in + 4, kept, 4, fk.AUTO, row_pad=8, sample=4)
    assert ctx.get_timing()[2] - before == 2          # the kernel and the one that clears its counters
    assert err < parity.check_compress(ctx, w, n_in + 4, kept, 4, fk.FDCT, sample=8)
    ctx.set_variant(fk.AUTO)


@pytest.mark.parametrize("hd,triples", [(64, 9), (64, 10), (256, 2), (256, 3)])
def test_smallest_calls_of_other_head_sizes(ctx, hd, triples):
    """Either side of the rule: as many slabs of 8 channels as SMs for the fast transform, more for the one-pass kernel."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the sizes are those of 148 SMs")
    w = synth.Workload("t", 1, 1, triples, hd, 1024, torch.bfloat16, 0, 0.9, 2, synth.BASE_SEED + 17)
    parity.check_compress(ctx, w, 1024, 512, 0, fk.AUTO, sample=2)
    before = ctx.get_timing()[2]
    parity.check_compress(ctx, w, 1024, 512, 0, fk.AUTO, sample=2)
    assert ctx.get_timing()[2] - before == (1 if triples in (9, 2) else 2)


def test_three_blocks_of_far_rows(ctx):
    """More than 8192 kept rows: the far rows of the tiles fill more than two blocks of 128, alone and beside short sequences."""
    parity.check_compress(ctx, workload(16510, 4, H=1), 16504, 8300, 4, fk.GEMM, sample=1)
    w = workload(16504, 4, B=3, H=1)
    k, v = synth.make_cache(w, "cuda")
    k0, v0 = k.clone(), v.clone()
    lens, kept = [700, 16504, 1300], [348, 8300, 600]
    ctx.set_variant(fk.AUTO)
    ctx.compress_ragged(k, v, lens, kept, 4)
    assert ctx.last_device_status() == fk.OK
    for b, (n, m) in enumerate(zip(lens, kept)):
        one_k, one_v = k0[b:b + 1].clone(), v0[b:b + 1].clone()
        ctx.compress(one_k, one_v, n, m, 4)
        assert torch.equal(one_k[0], k[b]) and torch.equal(one_v[0], v[b]), b


@pytest.mark.parametrize("n_in,kept", [(5376, 2689), (8194, 4097), (5400, 2700), (8188, 4094), (4092, 2046)])
def test_every_row_of_the_basis(ctx, n_in, kept):
    """Impulses as input give the basis itself.  An entry near the diagonal is rounded to bf16 once, 2^-9 of itself at most; the
    entries taken by interpolation, rounded three times and up to 3.5e-4 of the row off, hold a few hundredths of a row's energy:
    every row is within 2.5e-3 of its norm.  A short last tile (2689, 4097: one row) leaves the tile before it no far rows on one
    side."""
    heads = (n_in + 127) // 128
    x = torch.zeros(heads * 128, n_in, device="cuda")
    x[:n_in] = torch.eye(n_in, device="cuda")
    k = x.view(1, 1, heads, 128, n_in).transpose(3, 4).to(torch.bfloat16).contiguous()
    v = torch.zeros_like(k)
    ctx.set_variant(fk.AUTO)
    ctx.compress(k, v, n_in, kept, 0)
    got = k[0, 0, :, :kept].permute(1, 0, 2).reshape(kept, -1)[:, :n_in].double()
    t = torch.arange(kept, device="cuda")

    def rows(n):  # the first rows of the orthonormal DCT-II of n points
        i = torch.arange(n, device="cuda")
        c = torch.cos(((2 * i[None, :] + 1) * t[:, None] % (4 * n)).double() * (math.pi / (2 * n))) * math.sqrt(2 / n)
        c[0] *= math.sqrt(0.5)
        return c
    want = math.sqrt(kept / n_in) * rows(kept).T @ rows(n_in)
    error = (got - want).norm(dim=1) / want.norm(dim=1)
    assert error.max().item() < 2.5e-3, f"row {error.argmax().item()}: {error.max().item():.2e}"
    assert v.abs().max().item() == 0


def test_heads_of_64_captured_after_a_plan():
    """A compression of 64-channel heads, large enough for the one-pass kernel, captured as the context's first call after
    freqkv_plan: the capture allocates nothing and the replays give what the fast transform gives, also after a larger call of
    the context."""
    w = synth.Workload("t", 1, 3, 13, 64, 1024, torch.bfloat16, 0, 0.9, 2, synth.BASE_SEED + 13)
    k0, v0 = synth.make_cache(w, "cuda")
    c, stream = fk.Context(0), torch.cuda.Stream()
    try:
        c.set_variant(fk.FDCT)
        want_k, want_v = k0.clone(), v0.clone()
        c.compress(want_k, want_v, 1024, 512, 0)
        torch.cuda.synchronize()
    finally:
        c.close()
    c = fk.Context(0)
    try:
        lay = fk.layout_of(k0)
        with torch.cuda.stream(stream):
            c.plan(1024, 512, fk.BF16, c.resolve_variant(lay, 1024, 512))
        torch.cuda.synchronize()
        k, v = k0.clone(), v0.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            c.compress(k, v, 1024, 512, 0)
        for _ in range(2):
            with torch.cuda.stream(stream):
                k.copy_(k0)
                v.copy_(v0)
                graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(k, want_k) and torch.equal(v, want_v)
            with torch.cuda.stream(stream):
                big = torch.zeros(1, 8, 64, 4092, 64, device="cuda", dtype=torch.bfloat16)
                c.compress(big, big.clone(), 4092, 2046, 0)
        del graph
    finally:
        c.close()


def test_heads_of_64_without_memory_for_a_work_area():
    """A call large enough for the one-pass kernel on a device with a few MB free: it runs the fast transform, which needs none."""
    w = synth.Workload("t", 1, 4, 36, 64, 4092, torch.bfloat16, 0, 0.9, 2, synth.BASE_SEED + 14)
    k0, v0 = synth.make_cache(w, "cuda")
    small = torch.zeros(1, 1, 40, 1024, 64, device="cuda", dtype=torch.bfloat16)
    c, filler = fk.Context(0), []
    try:
        c.compress(small, small.clone(), 1024, 512, 0)          # loads the kernels
        c.set_variant(fk.FDCT)
        want_k, want_v = k0.clone(), v0.clone()
        c.compress(want_k, want_v, 4092, 2046, 0)
        c.set_variant(fk.AUTO)
        k, v = k0.clone(), v0.clone()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        size = torch.cuda.mem_get_info()[0] >> 20 << 20
        while size >= 2 << 20:
            try:
                filler.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.cuda.OutOfMemoryError:
                size //= 2
        assert torch.cuda.mem_get_info()[0] < 8 << 20           # its far sums alone take 10 MB
        c.plan(4092, 2046, fk.BF16, fk.FDCT)
        c.compress(k, v, 4092, 2046, 0)
        assert c.last_device_status() == fk.OK
        filler.clear()
        assert torch.equal(k, want_k) and torch.equal(v, want_v)
    finally:
        filler.clear()
        torch.cuda.empty_cache()
        c.close()


@pytest.mark.parametrize("hd,B,H,n_in,kept", [(64, 2, 72, 4092, 2046), (64, 1, 41, 1024, 512), (256, 1, 300, 3000, 1500)])
def test_calls_after_a_plan_allocate_nothing(hd, B, H, n_in, kept):
    w = synth.Workload("t", B, 2, H, hd, n_in, torch.bfloat16, 0, 0.9, 2, synth.BASE_SEED + 15)
    free = []
    for _ in range(2):      # the first also loads the kernels, which takes memory of its own
        k, v = synth.make_cache(w, "cuda")
        c = fk.Context(0)
        c.plan(n_in, kept, fk.BF16, c.resolve_variant(fk.layout_of(k), n_in, kept))
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        before = c.get_timing()[2]
        c.compress(k, v, n_in, kept, 0)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        assert c.get_timing()[2] - before == 2                  # the one-pass kernel and the one that clears its counters
        c.close()
    assert free[2] == free[3], free


@pytest.mark.parametrize("hd,H,n_in,kept", [(128, 3, 1028, 514), (128, 2, 5376, 2689), (64, 41, 1024, 512)])
def test_infinities_and_nan_stay_in_their_channel(ctx, hd, H, n_in, kept):
    """An infinity near the first row, one under a middle tile, a NaN: nothing of their channels is claimed but that a NaN is in
    every row; all other channels keep their bits.  A channel of values just below a third of the range stays finite."""
    w = synth.Workload("t", 1, 1, H, hd, n_in + 4, torch.bfloat16, 4, 0.9, 2, synth.BASE_SEED + 16)
    k0, v0 = synth.make_cache(w, "cuda")
    ctx.set_variant(fk.AUTO)
    clean_k, clean_v = k0.clone(), v0.clone()
    ctx.compress(clean_k, clean_v, n_in + 4, kept, 4)
    top = torch.finfo(torch.bfloat16).max
    k, v = k0.clone(), v0.clone()
    k[0, 0, 1, 4 + 7, 9] = float("inf")
    k[0, 0, 0, 4 + n_in // 2, 0] = float("-inf")
    v[0, 0, 1, 4 + n_in - 1, hd - 1] = float("nan")
    v[0, 0, 0, 4:, 17] = top / 3.1
    ctx.compress(k, v, n_in + 4, kept, 4)
    assert ctx.last_device_status() == fk.OK
    assert not torch.isfinite(k[0, 0, 1, 4:4 + kept, 9]).all() and not torch.isfinite(k[0, 0, 0, 4:4 + kept, 0]).all()
    assert torch.isnan(v[0, 0, 1, 4:4 + kept, hd - 1]).all()
    steady = v[0, 0, 0, 4:4 + kept, 17].double() / (top / 3.1) - 1
    assert steady.abs().max().item() < 3e-2
    for got, want, touched in ((k, clean_k, ((1, 9), (0, 0))), (v, clean_v, ((1, hd - 1), (0, 17)))):
        for head, channel in touched:
            got[0, 0, head, :, channel] = want[0, 0, head, :, channel] = 0
        assert torch.equal(got, want)


@pytest.mark.parametrize("hd,B,Ly,H", [(64, 2, 9, 3), (64, 1, 8, 1), (256, 1, 8, 1)])
def test_host_buffers_come_out_as_on_the_device(ctx, hd, B, Ly, H):
    """The host-buffer form works through a call a few layers at a time: heads of 64 and 256 channels take the kernel that the whole
    call would take, and come out bit for bit as on the device."""
    w = synth.Workload("t", B, Ly, H, hd, 1028, torch.bfloat16, 4, 0.9, 2, synth.BASE_SEED + 18)
    k, v = synth.make_cache(w, "cuda")
    host_k, host_v = k.cpu().pin_memory(), v.cpu().pin_memory()
    ctx.set_variant(fk.AUTO)
    ctx.compress_host(host_k, host_v, 1028, 512, 4)
    torch.cuda.synchronize()
    ctx.compress(k, v, 1028, 512, 4)
    torch.cuda.synchronize()
    assert torch.equal(host_k, k.cpu()) and torch.equal(host_v, v.cpu())
