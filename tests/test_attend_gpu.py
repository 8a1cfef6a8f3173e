"""GPU parity of freqkv_attend_decode (decode attention over the bounded cache, RoPE at in-cache
positions) against the fp64 oracle of oracle/attention.py on the same seeded inputs.

Tolerances, per query head, relative L2 of the 128 output channels: bf16 caches 1e-2 (the output
is rounded once to bf16: 2^-9); fp32 caches 2e-4 -- the scores carry the error of an fp32 rotation
whose cos/sin are stepped row to row for up to 32 rows (about 3e-6 relative per score term, times
scores of magnitude 10-20 in these inputs), which the softmax turns into the same relative error
of the weights."""
import numpy as np
import pytest
import torch

from oracle import attention as oa
from paper_2505_00570_b200 import binding as fk
from paper_2505_00570_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 2e-4, torch.bfloat16: 1e-2}


@pytest.fixture(scope="module")
def ctx():
    c = fk.Context(0)
    yield c
    c.close()


def workload(B, Ly, H, cap, dtype, seed=11):
    return synth.Workload("attn", B, Ly, H, 128, cap, dtype, 4, 0.9, 2, synth.BASE_SEED + seed)


def queries(B, heads, dtype, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(B, heads, 128, generator=gen, device="cuda").to(dtype)


def check(ctx, k, v, layer, q, lens, base, heads=None, scale=0.0):
    out = ctx.attend_decode(k, v, layer, q, lens, rope_base=base, scale=scale)
    assert ctx.last_device_status() == fk.OK
    B, Hq = q.shape[0], q.shape[1]
    G = Hq // k.shape[2]
    worst = 0.0
    pick = heads if heads is not None else [(b, h) for b in range(B) for h in range(k.shape[2])]
    for b, h in pick:
        want = oa.attend_decode(parity.to_f64(q[b, h * G:(h + 1) * G]), parity.to_f64(k[b, layer, h]),
                                parity.to_f64(v[b, layer, h]), lens[b], base, None if scale <= 0 else scale)
        got = parity.to_f64(out[b, h * G:(h + 1) * G])
        for g in range(G):
            worst = max(worst, parity.rel_l2(got[g], want[g]))
    assert worst <= TOL[q.dtype], f"relative L2 {worst:.3e}"
    return worst


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("G", [1, 2, 4, 8])
def test_attend_small_all_heads(ctx, dtype, G):
    w = workload(3, 3, 2, 300, dtype)
    k, v = synth.make_cache(w, "cuda")
    k0, v0 = k.clone(), v.clone()
    q = queries(3, 2 * G, dtype, 5 + G)
    check(ctx, k, v, 1, q, [300, 37, 1], 10000.0)
    assert torch.equal(k, k0) and torch.equal(v, v0)  # the cache is only read


@pytest.mark.parametrize("base,scale", [(0.0, 0.0), (500000.0, 0.05), (10000.0, 0.2)])
def test_attend_rope_off_other_base_and_scale(ctx, base, scale):
    w = workload(2, 2, 3, 200, torch.bfloat16, seed=12)
    k, v = synth.make_cache(w, "cuda")
    check(ctx, k, v, 0, queries(2, 6, torch.bfloat16, 3), [199, 64], base, scale=scale)
    check(ctx, k, v, 1, queries(2, 6, torch.bfloat16, 4), [2, 200], base, scale=scale)


def test_attend_row_padding_and_lengths_around_the_split_sizes(ctx):
    w = workload(1, 1, 2, 1100, torch.bfloat16, seed=13)
    (_, k), (_, v) = parity.guarded_cache(w, torch.device("cuda"), fill_len=1100, row_pad=8)
    q = queries(1, 4, torch.bfloat16, 6)
    for n in (15, 16, 17, 63, 64, 65, 255, 256, 257, 1023, 1024, 1025, 1100):
        check(ctx, k, v, 0, q, [n], 10000.0)


def test_attend_dominant_key_and_uniform_keys(ctx):
    """Special cases with known answers, straight on the GPU result."""
    k = torch.zeros(1, 1, 1, 128, 128, device="cuda", dtype=torch.float32)
    v = torch.randn(1, 1, 1, 128, 128, device="cuda")
    q = torch.zeros(1, 1, 128, device="cuda")
    q[0, 0, 0] = 1.0
    out = ctx.attend_decode(k, v, 0, q, [100], rope_base=0.0)          # all scores equal: the mean
    assert torch.allclose(out[0, 0], v[0, 0, 0, :100].mean(dim=0), atol=1e-5)
    k[0, 0, 0, 41, 0] = 2000.0                                          # one key wins
    out = ctx.attend_decode(k, v, 0, q, [100], rope_base=0.0)
    assert torch.allclose(out[0, 0], v[0, 0, 0, 41], atol=1e-5)


def test_attend_7b_shape_one_layer_sampled(ctx):
    """Batch 16 of 7B-shaped caches (32 KV heads, 4096 rows), two layers resident, the second one
    attended: 512 heads x 2.1 MB in one call; sampled heads against the oracle."""
    w = workload(16, 2, 32, 4096, torch.bfloat16, seed=14)
    k, v = synth.make_cache(w, "cuda")
    lens = [4096 - 37 * b for b in range(16)]
    q = queries(16, 32, torch.bfloat16, 8)
    check(ctx, k, v, 1, q, lens, 10000.0, heads=[(0, 0), (15, 31), (7, 13)])


def test_attend_gqa_8b_shape_sampled(ctx):
    w = workload(2, 1, 8, 8192, torch.bfloat16, seed=15)
    k, v = synth.make_cache(w, "cuda")
    check(ctx, k, v, 0, queries(2, 32, torch.bfloat16, 9), [8192, 4098], 500000.0, heads=[(0, 0), (1, 7)])


def test_attend_invalid_arguments(ctx):
    k = torch.zeros(1, 2, 2, 64, 128, device="cuda", dtype=torch.bfloat16)
    v = torch.zeros_like(k)
    q = torch.zeros(1, 2, 128, device="cuda", dtype=torch.bfloat16)
    for bad in ([0], [65]):
        with pytest.raises(fk.FreqKVError) as e:
            ctx.attend_decode(k, v, 0, q, bad)
        assert e.value.status == fk.ERR_INVALID_ARG
    with pytest.raises(fk.FreqKVError) as e:
        ctx.attend_decode(k, v, 2, q, [10])
    assert e.value.status == fk.ERR_INVALID_ARG
    with pytest.raises(fk.FreqKVError) as e:
        ctx.attend_decode(k, v, 0, torch.zeros(1, 6, 128, device="cuda", dtype=torch.bfloat16), [10])  # 3 query heads per KV head
    assert e.value.status == fk.ERR_UNSUPPORTED
    k64 = torch.zeros(1, 1, 1, 64, 64, device="cuda", dtype=torch.bfloat16)
    with pytest.raises(fk.FreqKVError) as e:
        ctx.attend_decode(k64, torch.zeros_like(k64), 0, torch.zeros(1, 1, 64, device="cuda", dtype=torch.bfloat16), [10])
    assert e.value.status == fk.ERR_UNSUPPORTED


@pytest.mark.parametrize("G", [1, 4])
def test_attend_more_sequences_than_one_launch_takes(ctx, G):
    """131 short sequences: the lengths travel as kernel arguments, 128 per launch, and one merge
    launch follows the last of them."""
    w = workload(131, 1, 1, 96, torch.bfloat16, seed=16)
    k, v = synth.make_cache(w, "cuda")
    lens = [96 - (b % 60) for b in range(131)]
    check(ctx, k, v, 0, queries(131, G, torch.bfloat16, 17 + G), lens, 10000.0, heads=[(0, 0), (1, 0), (127, 0), (128, 0), (130, 0)])


@pytest.mark.parametrize("G,H,lens", [(4, 8, [2611]), (1, 4, [193, 7000, 192]), (8, 4, [1400, 17, 385, 600]), (2, 3, [191, 1]),
                                      (1, 32, [900 + 37 * b for b in range(24)])])
def test_attend_splits_and_their_merge(ctx, G, H, lens):
    """A few groups cut into many splits that the last CTA of a group merges (one split, two, lengths around the smallest
    split), and more groups than one wave of CTAs holds, merged by a kernel of its own; the same bits call after call."""
    w = workload(len(lens), 1, H, max(lens) + 5, torch.bfloat16, seed=23)
    k, v = synth.make_cache(w, "cuda")
    q = queries(len(lens), H * G, torch.bfloat16, 24)
    first = ctx.attend_decode(k, v, 0, q, lens)
    for _ in range(3):
        assert torch.equal(ctx.attend_decode(k, v, 0, q, lens), first)
    last = len(lens) - 1
    check(ctx, k, v, 0, q, lens, 10000.0, heads=[(0, 0), (last, H - 1), (last // 2, 1)])


@pytest.mark.parametrize("dtype,G,H,lens", [(torch.bfloat16, 4, 8, [2611]), (torch.bfloat16, 1, 8, [1800, 333, 1900]), (torch.float32, 1, 4, [900, 1500]),
                                            (torch.bfloat16, 1, 32, [900 + 37 * b for b in range(24)]),
                                            (torch.bfloat16, 4, 32, [500 + 50 * b for b in range(24)])])
def test_attend_back_to_back_launches_with_different_contents(ctx, dtype, G, H, lens):
    """A chain of calls that nothing waits between, as a model enqueues them: a token is appended, then every layer attends
    over lengths of its own with the layer before's output as its queries, merged by tickets or by a kernel of its own.  A launch that
    read its inputs or merged its partials before the one in front of it was done would differ from the same chain with a
    synchronisation after every call."""
    layers, B = 3, len(lens)
    w = workload(B, layers, H, max(lens) + 8, dtype, seed=31)
    k0, v0 = synth.make_cache(w, "cuda")
    q0 = queries(B, H * G, dtype, 32)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(33)
    rows = [torch.randn(B, layers, H, 1, 128, generator=gen, device="cuda").to(dtype) for _ in range(2)]

    def chain(wait):
        k, v, q, outs, n = k0.clone(), v0.clone(), q0, [], lens
        torch.cuda.synchronize()
        for _ in range(4):
            n = ctx.append(k, v, rows[0], rows[1], n)
            for layer in range(layers):
                wait()
                q = ctx.attend_decode(k, v, layer, q, [max(1, x - 100 * layer) for x in n], scale=0.02)
                outs.append(q)
                wait()
        torch.cuda.synchronize()
        return torch.stack(outs)

    apart = chain(torch.cuda.synchronize)
    assert torch.isfinite(apart.float()).all() and not torch.equal(apart[0], apart[3])
    for _ in range(3):
        assert torch.equal(chain(lambda: None), apart)


@pytest.mark.parametrize("G,H,lens", [(4, 8, [2611]), (1, 4, [193, 1700, 192]), (1, 32, [900 + 37 * b for b in range(24)])])
def test_attend_captured_into_a_graph(G, H, lens):
    """A decode step of three layers captured and replayed, with eager calls of the same context between the replays: the eager
    calls keep their bits, the replays theirs, new queries are read at each replay.  A captured call merges its splits by a launch of
    its own, never by the ticket counters, which must be zero between the context's calls and which no replay may leave in
    another state.  The two merges sum the splits in another order: fp32 rounding, which can move the one rounding to bf16 by a
    step (2^-8 of the value, stated twice that; values near zero by their fp32 share)."""
    ctx, B = fk.Context(0), len(lens)
    w = workload(B, 3, H, max(lens) + 5, torch.bfloat16, seed=41)
    k, v = synth.make_cache(w, "cuda")
    q, q2 = queries(B, H * G, torch.bfloat16, 42), queries(B, H * G, torch.bfloat16, 43)
    stream = torch.cuda.Stream()
    step = lambda: torch.stack([ctx.attend_decode(k, v, layer, q, lens) for layer in range(3)])  # noqa: E731
    near = lambda a, b: torch.allclose(a.float(), b.float(), rtol=2.0 ** -7, atol=1e-5 * b.float().abs().max().item())  # noqa: E731
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        want = step()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        before = ctx.get_timing()[2]
        with torch.cuda.graph(graph, stream=stream):
            out = step()
        assert ctx.get_timing()[2] - before == 6     # per layer: the attention and the merge
        graph.replay()
        first = out.clone()
        assert near(first, want)
        for i in range(4):
            graph.replay()
            got = out.clone()
            assert torch.equal(got, first) and torch.equal(step(), want), i
        q.copy_(q2)
        graph.replay()
        got, want = out.clone(), step()
        assert near(got, want) and not near(got, first)
        check(ctx, k, v, 1, q, lens, 10000.0, heads=[(0, 0), (B - 1, H - 1)])
        stream.synchronize()
        del graph
    ctx.close()


def test_context_creation_does_not_wait_for_enqueued_work():
    """A context is created while a kernel of 0.2 s or so runs on the default stream: creation returns before it ends."""
    fk.Context(0).close()
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)
    done = torch.cuda.Event()
    done.record()
    ctx = fk.Context(0)
    assert not done.query()
    torch.cuda.synchronize()
    ctx.close()


def test_attend_work_area_follows_growing_lengths_once():
    """A batch whose lengths grow, as a decode stream's do, is split into more and more CTAs: the work area grows once for all
    of it (every time would mean a device synchronisation in the middle of the stream)."""
    k = torch.zeros(64, 1, 8, 2048, 128, device="cuda", dtype=torch.bfloat16)
    q = torch.zeros(64, 64, 128, device="cuda", dtype=torch.bfloat16)
    v, out = torch.ones_like(k), torch.empty_like(q)
    for attempt in range(2):     # the first also loads the kernels, which takes memory of its own
        ctx, free = fk.Context(0), []
        for n in (100, 250, 500, 900, 1400, 2048):
            ctx.attend_decode(k, v, 0, q, [n] * 64, out=out)
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
            assert (out == 1).all()
        ctx.close()
    assert len(set(free)) <= 2, free
