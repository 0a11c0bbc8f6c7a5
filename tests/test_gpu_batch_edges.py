"""GPU parity where the forward changes its path with the number of rows: every case against the oracle on a subset of
its tokens, with the output tolerance of the other parity tests (max |gpu - oracle| / RMS <= 1e-2)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import make_gpu_layer, make_oracle_layer, rel_err
from paper_2503_21135_b200 import binding
from paper_2503_21135_b200 import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-2


def _layer(max_tokens, **kw):
    cfg = wl.scaled(wl.CONFIGS["tiny"], zipf=None, tokens=(max_tokens,), **kw)
    wg, wu, wd = wl.layer_weights(cfg)
    bits = np.array([[2, 3, 4, 8, 6][e % 5] for e in range(cfg.n_experts)] + [8] * cfg.n_shared, np.int32)
    pool = wl.cache_pool(cfg)
    gpu = make_gpu_layer(cfg, wg, wu, wd, bits, pool, max_tokens=max_tokens)
    ora = make_oracle_layer(cfg, wg, wu, wd, bits)
    sets = wl.initial_sig_sets(cfg, pool)
    gpu.set_channel_switch(sets)
    ora.set_channel_switch(sets)
    return cfg, gpu, ora


def _check(cfg, gpu, ora, x, lg, toks):
    y = gpu.forward(x.cuda(), lg.cuda(), binding.F32)
    torch.cuda.synchronize()
    assert gpu.poll_status() == 0 and gpu.debug_check_guards() == 0
    ref = ora.forward(oracle.as_u16(x), lg.numpy(), tokens=np.asarray(toks, np.int32))["y"][toks]
    err = rel_err(y.cpu().numpy()[toks], ref)
    assert err <= TOL, err
    assert torch.equal(gpu.forward(x.cuda(), lg.cuda(), binding.F32), y)


@pytest.mark.parametrize("group_size", [64, 128])
def test_small_experts_beside_large_ones(group_size):
    """More than 1024 rows: the K splits of small experts (at most 32 rows) leave the common buffer.  Row counts on
    both sides of that limit and of the 8-row tiles, an empty expert, the rest on one large expert."""
    counts = [32, 31, 33, 1, 0, 24, 9]
    T = 1030 + sum(counts)
    cfg, gpu, ora = _layer(T, n_experts=8, top_k=1, group_size=group_size)
    e = np.concatenate([np.full(c, i) for i, c in enumerate(counts)] + [np.full(1030, 7)])
    e = e[np.random.default_rng(3).permutation(T)]
    lg = torch.zeros((T, 8))
    lg[torch.arange(T), torch.from_numpy(e)] = 4.0
    x = wl.activations(cfg, T, step=31)
    toks = np.flatnonzero(e != 7)
    _check(cfg, gpu, ora, x, lg, np.concatenate([toks, np.flatnonzero(e == 7)[:8]]))


@pytest.mark.parametrize("group_size", [64, 128])
@pytest.mark.parametrize("down", [False, True])
def test_middle_sized_batches(group_size, down):
    """One kernel for all experts: row counts around its tiles (16 columns an MMA, 64 rows a pass), every bit-width, an
    empty expert; with and without significant hidden units (they read h in this kernel's layout)."""
    counts = [64, 65, 16, 17, 1, 0, 48, 129]
    T = sum(counts)
    cfg, gpu, ora = _layer(T, n_experts=8, top_k=1, group_size=group_size)
    if down:
        wd = wl.layer_weights(cfg)[2]
        pool_d = wl.cache_pool_down(cfg, 32)
        sets_d = wl.sig_sets_down(cfg, pool_d, 16)
        gpu.pack_down_cache(wd.cuda(), np.array([[2, 3, 4, 8, 6][e % 5] for e in range(8)], np.int32), pool_d, 16)
        ora.enable_down_side(oracle.as_u16(wd))
        gpu.set_channel_switch_down(sets_d)
        ora.set_channel_switch_down(sets_d)
    e = np.concatenate([np.full(c, i) for i, c in enumerate(counts)])[np.random.default_rng(4).permutation(T)]
    lg = torch.zeros((T, 8))
    lg[torch.arange(T), torch.from_numpy(e)] = 4.0
    _check(cfg, gpu, ora, wl.activations(cfg, T, step=32), lg, np.arange(T))


@pytest.mark.parametrize("T", [65, 96, 247, 248, 249])
def test_both_ends_of_the_middle_sizes(T):
    cfg, gpu, ora = _layer(256, n_experts=8, top_k=2, group_size=128)
    _check(cfg, gpu, ora, wl.activations(cfg, T, step=33), wl.router_logits(cfg, T, step=33), np.arange(T))


@pytest.mark.parametrize("cfg_kw", [dict(n_experts=8, d_ff=1024), dict(n_experts=48, d_ff=2048), dict(n_experts=24, d_ff=2048),
                                    dict(n_experts=24, d_ff=2048, n_shared=1)])
@pytest.mark.parametrize("T", [7, 9, 17, 25, 33, 49, 64])
def test_items_of_every_size_on_the_streaming_path(cfg_kw, T):
    """Small batches with a skewed router: the first expert has all the tokens, the second half of them, so experts take
    one to eight passes of items of one, two or three tiles, with a remainder, in launches of few and of many items."""
    cfg, gpu, ora = _layer(64, top_k=3, group_size=64, **cfg_kw)
    lg = wl.router_logits(cfg, T, step=34)
    lg[:, 0] += 20.0
    lg[: (T + 1) // 2, 1] += 20.0
    _check(cfg, gpu, ora, wl.activations(cfg, T, step=34), lg, np.arange(T))


@pytest.mark.parametrize("T", [1, 5, 64, 70])
@pytest.mark.parametrize("kind", ["pinned", "pageable", "results_pinned", "shifted"])
def test_host_buffers_of_every_kind(kind, T):
    """Page-locked and aligned buffers are read and written in place, others through copies: the same results."""
    def buffer(t, pin):
        flat = torch.empty(t.numel() + 8, dtype=t.dtype, pin_memory=pin)
        off = 1 if kind == "shifted" else 0
        return flat[off: off + t.numel()].view(t.shape).copy_(t)

    cfg, gpu, _ = _layer(80, n_experts=5, top_k=2, group_size=64)
    x, lg = wl.activations(cfg, T, step=35), wl.router_logits(cfg, T, step=35)
    ins = kind in ("pinned", "shifted")
    for dtype, code in ((torch.float32, binding.F32), (torch.bfloat16, binding.BF16)):
        y = buffer(torch.zeros((T, cfg.d_model), dtype=dtype), kind != "pageable")
        before = gpu.kernel_launches()
        gpu.forward_host(buffer(x, ins), buffer(lg, ins), y, code)
        launched = gpu.kernel_launches() - before
        assert gpu.poll_status() == 0
        before = gpu.kernel_launches()
        assert torch.equal(y, gpu.forward(x.cuda(), lg.cuda(), code).cpu())
        # one launch more where the kernels read the buffers themselves
        assert launched - (gpu.kernel_launches() - before) == (1 if kind == "pinned" else 0)


@pytest.mark.parametrize("large", [1, 3, 7])
def test_small_experts_run_beside_large_ones(large):
    """The kernels of large and of small experts overlap: forwards of different inputs that follow one another without a
    wait in between give what each gives alone."""
    cfg, gpu, _ = _layer(700, n_experts=8, top_k=1, group_size=64)
    runs = []
    for i, T in enumerate((700, 640, 520)):   # (up to 496 tokens one kernel takes all experts of this layer)
        e = np.where(np.arange(T) % 16 < 15, np.arange(T) % large, large + np.arange(T) % (8 - large))
        lg = torch.zeros((T, 8))
        lg[torch.arange(T), torch.from_numpy((e + i) % 8)] = 4.0
        x = wl.activations(cfg, T, step=36 + i).cuda()
        runs.append((x, lg.cuda()))
    before = gpu.kernel_launches()
    gpu.forward(*runs[-1], binding.F32)
    assert gpu.kernel_launches() - before == 8   # the two kernels side by side
    alone = []
    for x, lg in runs:
        alone.append(gpu.forward(x, lg, binding.F32).clone())
        torch.cuda.synchronize()
    for _ in range(5):
        got = [gpu.forward(x, lg, binding.F32) for x, lg in runs]
        assert all(torch.equal(a, b) for a, b in zip(got, alone))
    assert gpu.poll_status() == 0 and gpu.debug_check_guards() == 0


def _everything_on(cfg, gpu, ora):
    """Hidden-unit sets on the d_ff side and activation statistics."""
    wd = wl.layer_weights(cfg)[2]
    pool_d = wl.cache_pool_down(cfg, 32)
    sets_d = wl.sig_sets_down(cfg, pool_d, 16)
    bits = np.array([[2, 3, 4, 8, 6][e % 5] for e in range(cfg.n_experts)] + [8] * cfg.n_shared, np.int32)
    gpu.pack_down_cache(wd.cuda(), bits, pool_d, 16)
    gpu.set_channel_switch_down(sets_d)
    ora.enable_down_side(oracle.as_u16(wd))
    ora.set_channel_switch_down(sets_d)
    gpu.set_stats_collection(True)


def _few_large_experts(T, shift):
    """Router logits of a top-1 layer of eight experts: three of them with most of the tokens, five with a few."""
    e = (np.where(np.arange(T) % 16 < 15, np.arange(T) % 3, 3 + np.arange(T) % 5) + shift) % 8
    lg = torch.zeros((T, 8))
    lg[torch.arange(T), torch.from_numpy(e)] = 4.0
    return lg


@pytest.mark.parametrize("n_shared", [0, 1])
def test_statistics_and_hidden_unit_sets_beside_the_pair_kernel(n_shared):
    """Statistics start beside the gate/up kernels and use the down launch's output as scratch, the d_ff-side correction
    starts beside the down kernels: forwards that follow one another without a wait, all against the oracle."""
    cfg, gpu, ora = _layer(700, n_experts=8, top_k=1, group_size=64, n_shared=n_shared)
    _everything_on(cfg, gpu, ora)
    runs = [(wl.activations(cfg, T, step=41 + i), _few_large_experts(T, i)) for i, T in enumerate((700, 520, 633))]
    dev = [(x.cuda(), lg.cuda()) for x, lg in runs]
    before = gpu.kernel_launches()
    outs = [gpu.forward(x, lg, binding.F32) for x, lg in dev]
    assert gpu.kernel_launches() - before == 3 * 10   # pair and streaming kernels, statistics, correction
    got = gpu.channel_stats().cpu().numpy().astype(np.float64)
    torch.cuda.synchronize()
    assert gpu.poll_status() == 0 and gpu.debug_check_guards() == 0
    pool = wl.cache_pool(cfg)
    stats, n_add = np.zeros((8, cfg.cache_size)), np.zeros(8)
    for (x, lg), y in zip(runs, outs):
        idx, _ = oracle.route(lg.numpy(), 1)
        stats = oracle.channel_stats_update(stats, oracle.as_u16(x), idx, pool)
        n_add += np.bincount(idx.ravel(), minlength=8) + 1
        toks = np.arange(0, x.shape[0], 9, dtype=np.int32)
        ref = ora.forward(oracle.as_u16(x), lg.numpy(), tokens=toks)["y"][toks]
        assert rel_err(y.cpu().numpy()[toks], ref) <= TOL
    # fp32 accumulation of n non-negative terms: |fl(sum) - sum| <= n * 2^-24 * sum
    assert np.all(np.abs(got - stats) <= n_add[:, None] * 2.0 ** -24 * stats)
    for _ in range(5):
        again = [gpu.forward(x, lg, binding.F32) for x, lg in dev]
        assert all(torch.equal(a, b) for a, b in zip(again, outs))


@pytest.mark.parametrize("T", [100, 700])   # fold kernel; pair and streaming kernels side by side
def test_overlapping_launches_in_a_captured_graph(T):
    cfg, gpu, ora = _layer(700, n_experts=8, top_k=1, group_size=128)
    _everything_on(cfg, gpu, ora)
    xs, ls = torch.zeros((T, cfg.d_model), dtype=torch.bfloat16, device="cuda"), torch.zeros((T, 8), device="cuda")
    ys = torch.empty((T, cfg.d_model), device="cuda")
    inputs = [(wl.activations(cfg, T, step=51 + i).cuda(), _few_large_experts(T, i).cuda()) for i in range(2)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        gpu.forward(xs, ls, binding.F32, y=ys)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gpu.forward(xs, ls, binding.F32, y=ys)
        gpu.forward(xs, ls, binding.F32, y=ys)
    for x, lg in inputs:
        want, stats = [], []
        for replay in (False, True):
            gpu.select_significant(0, reset=True)
            if replay:
                xs.copy_(x)
                ls.copy_(lg)
                graph.replay()
                want.append(ys.clone())
            else:
                gpu.forward(x, lg, binding.F32)
                want.append(gpu.forward(x, lg, binding.F32))
            stats.append(gpu.channel_stats().clone())
        torch.cuda.synchronize()
        assert torch.equal(want[0], want[1]) and torch.equal(stats[0], stats[1])
    assert gpu.poll_status() == 0 and gpu.debug_check_guards() == 0


@pytest.mark.parametrize("group_size", [64, 128])
@pytest.mark.parametrize("counts", [[128, 129, 1, 0, 17, 64, 65, 81], [496, 0, 0, 0, 0, 0, 0, 0], [96, 60, 72, 48, 128, 0, 40, 4],
                                    [0, 257, 0, 0, 7, 0, 130, 0]])
def test_popular_experts_of_a_middle_sized_batch(counts, group_size):
    """Experts of more than 128 rows leave for the pair kernel, which starts beside the fold kernel: row counts on both
    sides of that limit, one expert with everything, none that leaves; with statistics and hidden-unit sets (they read
    either kernel's layout)."""
    T = sum(counts)
    cfg, gpu, ora = _layer(T, n_experts=8, top_k=1, group_size=group_size, d_model=1024, d_ff=4096)
    _everything_on(cfg, gpu, ora)
    e = np.concatenate([np.full(c, i) for i, c in enumerate(counts)])[np.random.default_rng(5).permutation(T)]
    lg = torch.zeros((T, 8))
    lg[torch.arange(T), torch.from_numpy(e)] = 4.0
    x = wl.activations(cfg, T, step=71)
    xd, ld = x.cuda(), lg.cuda()
    before = gpu.kernel_launches()
    first = gpu.forward(xd, ld, binding.F32)
    assert gpu.kernel_launches() - before == 10
    for _ in range(5):
        assert torch.equal(gpu.forward(xd, ld, binding.F32), first)
    ends = [t for i in range(8) if counts[i] for t in np.flatnonzero(e == i)[[0, -1]]]
    toks = np.unique(np.array(ends + list(range(0, T, 31)), np.int32))
    _check(cfg, gpu, ora, x, lg, toks)
    stats = oracle.channel_stats_update(np.zeros((8, cfg.cache_size)), oracle.as_u16(x), e[:, None].astype(np.int32), wl.cache_pool(cfg))
    got = gpu.channel_stats().cpu().numpy() / 8.0     # eight forwards of the same tokens
    assert np.all(np.abs(got - stats) <= (np.array(counts)[:, None] + 9) * 2.0 ** -24 * stats)


@pytest.mark.parametrize("T,launches", [(319, 8), (321, 6), (600, 8), (641, 8)])
def test_many_small_experts_in_a_middle_sized_batch(T, launches):
    """32 small experts, top-2, a skewed router, on both sides of the rows per expert from which and up to which they take
    the fold kernel, and of the rows beyond which nothing is split along K."""
    cfg, gpu, ora = _layer(641, n_experts=32, top_k=2, group_size=64, d_ff=2048)
    lg = wl.router_logits(cfg, T, step=72)
    lg -= 1.2 * torch.log(torch.arange(1.0, 33.0))
    assert torch.bincount(lg.topk(2, 1)[1].flatten(), minlength=32).max() > 128
    before = gpu.kernel_launches()
    x = wl.activations(cfg, T, step=72)
    gpu.forward(x.cuda(), lg.cuda(), binding.F32)
    assert gpu.kernel_launches() - before == launches   # streaming and pair, fold, fold and pair, streaming and pair kernel
    _check(cfg, gpu, ora, x, lg, np.arange(0, T, 7))


@pytest.mark.parametrize("group_size", [64, 128])
def test_either_streaming_variant_of_a_small_batch(group_size):
    """Large experts, 9 to 32 tokens: two variants are launched and the device takes the one whose items suit the experts'
    rows.  Routers on both sides of the choice for items of one and of two tiles; with statistics and hidden-unit sets."""
    cfg, gpu, ora = _layer(32, n_experts=3, top_k=1, group_size=group_size, d_model=2048, d_ff=16384)
    _everything_on(cfg, gpu, ora)
    for counts in ([9, 0, 0], [8, 8, 4], [9, 9, 2], [20, 0, 0], [4, 1, 16], [28, 0, 0], [17, 10, 1], [10, 10, 10], [0, 16, 12]):
        T = sum(counts)
        e = np.concatenate([np.full(c, i) for i, c in enumerate(counts)])[np.random.default_rng(T).permutation(T)]
        lg = torch.zeros((T, 3))
        lg[torch.arange(T), torch.from_numpy(e)] = 4.0
        x = wl.activations(cfg, T, step=81)
        before = gpu.kernel_launches()
        gpu.forward(x.cuda(), lg.cuda(), binding.F32)
        assert gpu.kernel_launches() - before == 8   # front, two of either FFN launch, statistics, correction, combine
        ends = [t for i in range(3) if counts[i] for t in np.flatnonzero(e == i)[[0, -1]]]
        _check(cfg, gpu, ora, x, lg, np.unique(np.array(ends, np.int32)))


def _check_pair_tiles(**kw):
    counts = [33, 128, 129, 256, 257, 513, 160, 96]
    T = sum(counts)
    cfg, gpu, ora = _layer(T, n_experts=8, top_k=1, **kw)
    e = np.concatenate([np.full(c, i) for i, c in enumerate(counts)])[np.random.default_rng(7).permutation(T)]
    lg = torch.zeros((T, 8))
    lg[torch.arange(T), torch.from_numpy(e)] = 4.0
    rows = [np.flatnonzero(e == i) for i in range(8)]   # token-ascending inside an expert
    toks = np.concatenate([r[sorted({0, 31, 32, len(r) // 2, 127 % len(r), 128 % len(r), 159 % len(r), 160 % len(r), 255 % len(r),
                                     256 % len(r), len(r) - 1})] for r in rows])
    _check(cfg, gpu, ora, wl.activations(cfg, T, step=36), lg, toks)


@pytest.mark.parametrize("d_model,group_size", [(256, 128), (512, 64), (768, 128)])
def test_token_tiles_of_the_pair_kernel(d_model, group_size):
    """Rows around its tiles (of at most 256 rows, an MMA of 32 at a time) and around 128, up to where two items have
    accumulators of their own; 352 gate/up items for at most 74 pairs of SMs, narrow and wide ones in turn."""
    _check_pair_tiles(d_model=d_model, d_ff=4096, group_size=group_size)


@pytest.mark.parametrize("d_model,d_ff,group_size,cache", [(256, 4096, 64, 0), (256, 4096, 128, 0), (4096, 128, 128, 64),
                                                           (4096, 256, 64, 64), (4096, 384, 128, 0), (4096, 384, 64, 64),
                                                           (4096, 512, 128, 64)])
def test_short_items_of_the_pair_kernel(d_model, d_ff, group_size, cache):
    """Items of one, two, three and four stages, two to five of them a pair of SMs (352 gate/up items without cached channels,
    or 176 down items): an item is wholly dequantized ahead of the epilogue before it, and stage numbers, ring offsets and
    barrier phases run on over items that are shorter than that lead."""
    _check_pair_tiles(d_model=d_model, d_ff=d_ff, group_size=group_size, max_sig=cache // 2, cache_size=cache)
