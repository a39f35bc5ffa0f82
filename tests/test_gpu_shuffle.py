"""GPU parity of the shuffling step: libwash.so (through its C ABI) against the oracle,
bit for bit, on the same seeded inputs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_17517_b200 import binding as B
from paper_2405_17517_b200 import workloads as W
from gpu_util import Case, bits, to_host_bits

pytestmark = pytest.mark.gpu

RAGGED = [1000, 33, 7, 1, 4, 8, 5003, 2048]       # several tiles, ragged tails, tiny tensors


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 16, 20, 24, 32, 33, 64])
def test_shuffle_fp32_matches_oracle(N, layout):
    c = Case(N, RAGGED, layout, seed=N)
    p_layer = [0.3, 1.0, 0.5, 1.0, 0.0, 0.9, 0.05, 0.01]
    for step in (0, 1, (7 << 32) | 5):
        B.wash_shuffle(c.gpu.ctx, step, 0.0, p_layer, seed=0xABCDEF0123456789, stats=c.stats_dev)
        sel, moved = oracle.shuffle(c.ora, c.host, p_layer, seed=0xABCDEF0123456789, step=step)
        c.assert_equal("N=%d layout=%d step=%d" % (N, layout, step))
    # counters accumulate over the three calls
    st = c.gpu_stats()
    c2 = Case(N, RAGGED, layout, seed=N)
    tot = [0, 0]
    for step in (0, 1, (7 << 32) | 5):
        s = oracle.shuffle(c2.ora, c2.host, p_layer, seed=0xABCDEF0123456789, step=step)
        tot[0] += s[0]; tot[1] += s[1]
    assert st == tuple(tot)
    c.close(); c2.close()


@pytest.mark.parametrize("mode", [B.WASH_MODE_STREAM, B.WASH_MODE_SPARSE])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N", [2, 3, 5, 7, 8, 9, 10, 16, 17, 32, 33, 64])
def test_both_kernels_on_many_tiles_match_oracle(N, layout, mode):
    """Both kernels (run-time N) on many tiles with a ragged last tile, both stacks,
    per-layer probabilities from never to always."""
    numel = [70001, 33, 7, 1, 4, 8, 5003, 2048, 300000 if N <= 16 else 30000]
    c = Case(N, numel, layout, "f32", "f32", seed=N)
    B.wash_set_mode(c.gpu.ctx, mode)
    p_layer = [0.3, 1.0, 0.5, 1.0, 0.0, 0.9, 0.05, 0.01, 0.002]
    tot = [0, 0]
    for step in (0, 1, (7 << 32) | 5):
        B.wash_shuffle_both(c.gpu.ctx, step, 0.0, p_layer, seed=0xABCDEF0123456789, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, p_layer, seed=0xABCDEF0123456789, step=step, stack2=c.host_opt)
        tot[0] += s[0]; tot[1] += s[1]
        c.assert_equal("N=%d layout=%d step=%d" % (N, layout, step))
    assert c.gpu_stats() == tuple(tot)
    c.close()


@pytest.mark.parametrize("mode", [B.WASH_MODE_STREAM, B.WASH_MODE_SPARSE, B.WASH_MODE_AUTO])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dtype,opt_dtype", [("f32", "f32"), ("bf16", "f32"), ("bf16", "bf16"), ("f32", "bf16"), ("bf16", None)])
def test_shuffle_both_stacks_and_dtypes(dtype, opt_dtype, layout, mode):
    N = 5
    c = Case(N, RAGGED, layout, dtype, opt_dtype, seed=3)
    B.wash_set_mode(c.gpu.ctx, mode)
    for step in range(3):
        if opt_dtype is None:
            B.wash_shuffle(c.gpu.ctx, step, 0.2, None, seed=9, stats=c.stats_dev)
        else:
            B.wash_shuffle_both(c.gpu.ctx, step, 0.2, None, seed=9, stats=c.stats_dev)
        oracle.shuffle(c.ora, c.host, 0.2, seed=9, step=step, stack2=c.host_opt)
        c.assert_equal("step %d" % step)
    c.close()


@pytest.mark.parametrize("flavour", [-2, -3], ids=["lean", "early"])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,dtype,opt_dtype", [(5, "f32", "f32"), (16, "f32", None), (17, "f32", "f32"), (33, "bf16", "f32"), (64, "f32", None)])
def test_streaming_flavours_on_dense_and_mixed_selection(N, dtype, opt_dtype, layout, flavour):
    """The streaming kernel's two flavours (permutations drawn after or before the wait for the
    copies; the early one serves N > 16 densely from byte columns) on tensors that are selected
    in full, mostly, half, rarely and not at all, with ragged ends."""
    numel = [9000, 33, 4100, 7, 2600, 1, 5003]
    p_layer = [1.0, 1.0, 0.9, 0.5, 0.45, 1.0, 0.02]
    c = Case(N, numel, layout, dtype, opt_dtype, seed=40 + N)
    B.wash_set_launch(c.gpu.ctx, 0, flavour)
    tot = [0, 0]
    for step in (0, 1, (3 << 32) | 9):
        if opt_dtype is None:
            B.wash_shuffle(c.gpu.ctx, step, 0.0, p_layer, seed=123, stats=c.stats_dev)
        else:
            B.wash_shuffle_both(c.gpu.ctx, step, 0.0, p_layer, seed=123, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, p_layer, seed=123, step=step, stack2=c.host_opt)
        tot[0] += s[0]; tot[1] += s[1]
        c.assert_equal("N=%d layout=%d step=%d" % (N, layout, step))
    assert c.gpu_stats() == tuple(tot)
    c.close()


@pytest.mark.parametrize("code", [-4, -5, 0], ids=["resident", "one-trip", "default"])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,dtype,opt_dtype", [(2, "f32", None), (2, "bf16", "f32"), (3, "f32", "f32"), (4, "bf16", None), (4, "f32", None), (8, "f32", None), (17, "bf16", "bf16")])
def test_resident_warp_streaming_kernel(N, dtype, opt_dtype, layout, code):
    """The streaming kernel for small groups (a resident grid of warps walking tiles with two
    shared-memory stages), forced, excluded and as the library chooses, against the oracle: enough
    coordinates for several trips per warp, tensors selected in full, half, rarely and not at
    all, ragged ends, a tensor boundary inside a tile."""
    numel = [2_600_003 if N <= 4 else 200_003, 33, 4100, 7, 260_000, 1, 5003, 90_001]
    p_layer = [0.004, 1.0, 0.9, 0.5, 0.3, 1.0, 0.0, 1.0]
    c = Case(N, numel, layout, dtype, opt_dtype, seed=70 + N)
    B.wash_set_launch(c.gpu.ctx, 0, code)
    tot = [0, 0]
    for step in (0, 1, (5 << 32) | 2):
        if opt_dtype is None:
            B.wash_shuffle(c.gpu.ctx, step, 0.0, p_layer, seed=77, stats=c.stats_dev)
        else:
            B.wash_shuffle_both(c.gpu.ctx, step, 0.0, p_layer, seed=77, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, p_layer, seed=77, step=step, stack2=c.host_opt)
        tot[0] += s[0]; tot[1] += s[1]
        c.assert_equal("N=%d layout=%d step=%d" % (N, layout, step))
    assert c.gpu_stats() == tuple(tot)
    B.wash_check(c.gpu.ctx)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
def test_separate_calls_equal_the_fused_call(layout):
    N = 8
    a = Case(N, RAGGED, layout, "f32", "f32", seed=5)
    b = Case(N, RAGGED, layout, "f32", "f32", seed=5)
    B.wash_shuffle_both(a.gpu.ctx, 4, 0.5, None, seed=1, stats=a.stats_dev)
    B.wash_shuffle(b.gpu.ctx, 4, 0.5, None, seed=1, stats=b.stats_dev)
    B.wash_shuffle_opt_state(b.gpu.ctx, 4, 0.5, None, seed=1)
    torch.cuda.synchronize()
    assert torch.equal(a.dev.view(torch.int32), b.dev.view(torch.int32))
    assert torch.equal(a.dev_opt.view(torch.int32), b.dev_opt.view(torch.int32))
    assert a.gpu_stats() == b.gpu_stats()
    oracle.shuffle(a.ora, a.host, 0.5, seed=1, step=4, stack2=a.host_opt)
    a.assert_equal()
    a.close(); b.close()


@pytest.mark.parametrize("N", [3, 10, 11])
def test_sparse_mode_and_launch_shapes_give_the_same_bits(N):
    ref = Case(N, RAGGED, 0, seed=8)
    oracle.shuffle(ref.ora, ref.host, 0.1, seed=2, step=3)
    for mode in (B.WASH_MODE_STREAM, B.WASH_MODE_SPARSE, B.WASH_MODE_AUTO):
        for threads, bps in ((0, 0), (64, 1), (128, 2), (256, -1), (96, 0), (32, 4), (256, 2), (128, 1), (0, -2), (0, -3), (128, -3), (0, -4), (0, -5)):
            c = Case(N, RAGGED, 0, seed=8)
            B.wash_set_mode(c.gpu.ctx, mode)
            B.wash_set_launch(c.gpu.ctx, threads, bps)
            B.wash_shuffle(c.gpu.ctx, 3, 0.1, None, seed=2)
            torch.cuda.synchronize()
            assert (to_host_bits(c.dev) == bits(ref.host)).all(), (mode, threads, bps)
            c.close()
    ref.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,numel,p", [(2, [511], 1.0), (5, [512], 1.0), (5, [2049], 1.0), (16, [6143, 2], 1.0), (17, [2047, 4100], 1.0),
                                       (32, [8192], 0.3), (33, [2100], 1.0), (64, [5000, 3], 0.9), (2, [3_000_001], 0.9), (10, [400_009], 0.002)])
def test_sparse_queue_at_its_edges(N, numel, p, layout):
    """One, two and several warp tiles per block; a queue that overflows within a tile (a block queues 512
    coordinates, 256 above 32 models) and is served several times; sets that leave pairs without a coordinate."""
    c = Case(N, numel, layout, "f32", "bf16" if N in (5, 17) else None, seed=N)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_SPARSE)
    call = B.wash_shuffle if c.host_opt is None else B.wash_shuffle_both
    call(c.gpu.ctx, 6, p, None, seed=12, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p, seed=12, step=6, stack2=c.host_opt)
    c.assert_equal("N=%d numel=%s p=%g layout=%d" % (N, numel, p, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,numel,p,dtype,opt", [
    (2, [509], 0.3, "f32", None), (2, [512], 0.3, "f32", None), (3, [513, 8], 0.2, "f32", None), (3, [255, 256, 257, 1024], 0.02, "bf16", None),
    (2, [2_000_003], 0.01, "f32", None), (3, [2_400_000, 9, 700_000], 0.0002, "f32", None), (2, [1_500_001], 1.0, "f32", None),
    (4, [900_001, 77], 0.02, "f32", None), (2, [700_001], 0.3, "f32", "f32"), (10, [300_001], 0.6, "f32", None), (17, [40_001], 0.3, "bf16", "f32")])
def test_resident_warp_kernel_serves_a_tiles_groups_together(N, numel, p, dtype, opt, layout):
    """The small-group streaming kernel: tiles of 128 and of 64 groups (below 0.07 % expected selection), ragged and
    single tiles, tensors that end inside a tile, lists of more than 32 coordinates, tiles selected in full."""
    c = Case(N, numel, layout, dtype, opt, seed=N)
    B.wash_set_launch(c.gpu.ctx, 0, -4)
    call = B.wash_shuffle if opt is None else B.wash_shuffle_both
    tot = [0, 0]
    for step in (0, 1):     # twice: the counters' slots must be left zeroed
        call(c.gpu.ctx, step, p, None, seed=31, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, p, seed=31, step=step, stack2=c.host_opt)
        tot[0] += s[0]; tot[1] += s[1]
    c.assert_equal("N=%d numel=%s p=%g layout=%d" % (N, numel, p, layout))
    assert c.gpu_stats() == tuple(tot)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,numel,p,dtype,opt", [
    (17, [30_001], 0.01, "f32", None), (18, [127, 1, 130, 4000], 0.1, "bf16", None), (20, [50_003], 0.25, "bf16", "f32"),
    (32, [40_009], 0.1, "f32", None), (32, [253, 4, 3000], 0.65, "f32", None), (24, [30_011], 0.03, "bf16", "f32"), (33, [255, 9000], 0.2, "f32", None), (63, [20_001], 0.05, "f32", "bf16"), (64, [12_345], 0.28, "f32", "f32")])
def test_wide_population_kernel(N, numel, p, dtype, opt, layout):
    """The streaming kernel of N > 16: permutations of 17 to 64 entries (last Philox block full and partly used), rounds
    of up to 32 and several rounds per warp, few and many coordinates in [N][P] (a lane per pair / per coordinate)."""
    c = Case(N, numel, layout, dtype, opt, seed=N)
    call = B.wash_shuffle if opt is None else B.wash_shuffle_both
    call(c.gpu.ctx, 3, p, None, seed=77, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p, seed=77, step=3, stack2=c.host_opt)
    c.assert_equal("N=%d numel=%s p=%g layout=%d" % (N, numel, p, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


def test_edge_cases_p0_p1_single_element_and_padding():
    # p = 0: identity, nothing written; p = 1: everything selected
    c = Case(4, [1], 0, seed=1)
    B.wash_shuffle(c.gpu.ctx, 0, 0.0, None, seed=0, stats=c.stats_dev)
    c.assert_equal("p=0")
    assert c.gpu_stats() == (0, 0)
    B.wash_shuffle(c.gpu.ctx, 0, 1.0, None, seed=0, stats=c.stats_dev)
    sel, moved = oracle.shuffle(c.ora, c.host, 1.0, seed=0, step=0)
    c.assert_equal("p=1")     # compares the padding too: it must still hold its NaN pattern
    assert c.gpu_stats() == (1, moved) and sel == 1
    c.close()
    for numel in ([3], [4], [5], [8], [9], [31, 33], [1, 1, 1, 1]):
        for layout in (0, 1):
            c = Case(3, numel, layout, seed=2)
            B.wash_shuffle(c.gpu.ctx, 11, 1.0, None, seed=5)
            oracle.shuffle(c.ora, c.host, 1.0, seed=5, step=11)
            c.assert_equal(str(numel))
            c.close()


def test_last_layer_untouched_and_schedules_agree_with_oracle():
    numel = [640, 1280, 320, 2560, 100]
    c = Case(5, numel, 0, seed=4)
    before = to_host_bits(c.dev).reshape(5, c.P)[:, c.off[-1]:c.off[-1] + 100].copy()
    for sched in (0, 1, 2):
        assert np.array_equal(B.wash_layer_probs(len(numel), 0.4, sched), oracle.layer_probs(len(numel), 0.4, sched))
    pl = B.wash_layer_probs(len(numel), 0.4)
    for step in range(5):
        B.wash_shuffle(c.gpu.ctx, step, 0.4, pl, seed=step)
        oracle.shuffle(c.ora, c.host, pl, seed=step, step=step)
    c.assert_equal()
    after = to_host_bits(c.dev).reshape(5, c.P)[:, c.off[-1]:c.off[-1] + 100]
    assert (before == after).all()
    c.close()


@pytest.mark.parametrize("p", [0.25, 0.6])
@pytest.mark.parametrize("N,dtype,opt", [(2, "f32", None), (8, "f32", None), (16, "bf16", None), (16, "f32", None), (12, "f32", None),
                                         (4, "f32", "f32"), (10, "bf16", "f32"), (20, "f32", None)])
def test_coordinate_major_images_with_and_without_padding(N, dtype, opt, p):
    """[P][N], below and above the share from which some populations' images are padded."""
    c = Case(N, [30_001, 9, 2048], 1, dtype, opt, seed=N)
    call = B.wash_shuffle if opt is None else B.wash_shuffle_both
    call(c.gpu.ctx, 1, p, None, seed=6, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p, seed=6, step=1, stack2=c.host_opt)
    c.assert_equal("N=%d" % N)
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,numel,p,dtype,opt", [
    (2, [9_000_001], [0.03], "f32", None),                       # several waves of blocks, loaded evenly
    (3, [5_000_003, 30_000], [0.0005, 1.0], "f32", "f32"),       # one wave by the mean, a few blocks loaded far above it
    (9, [2_000_001], [0.01], "bf16", None), (20, [1_000_001], [0.004], "f32", None)])
def test_sparse_blocks_take_what_a_wave_leaves_them(N, numel, p, dtype, opt, layout):
    c = Case(N, numel, layout, dtype, opt, seed=N)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_SPARSE)
    call = B.wash_shuffle if opt is None else B.wash_shuffle_both
    call(c.gpu.ctx, 2, max(p), p, seed=3, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p, seed=3, step=2, stack2=c.host_opt)
    c.assert_equal("N=%d layout=%d" % (N, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("dtype,opt", [("f32", None), ("bf16", None), ("bf16", "f32")])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6])
def test_resident_warp_kernel_for_each_compiled_population(N, dtype, opt, layout):
    """Populations of 2 to 5 models have kernels of their own and 6 the one that reads N at run time: rare and common
    selection, a tensor selected in full, a ragged last tile."""
    numel = [150_001, 3, 127, 40_000]
    c = Case(N, numel, layout, dtype, opt, seed=N)
    B.wash_set_launch(c.gpu.ctx, 0, -4)
    p = [0.02, 0.5, 1.0, 0.4]
    call = B.wash_shuffle if opt is None else B.wash_shuffle_both
    call(c.gpu.ctx, 3, 0.5, p, seed=8, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p, seed=8, step=3, stack2=c.host_opt)
    c.assert_equal("N=%d layout=%d" % (N, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("N,dtype,opt", [(2, "f32", None), (2, "bf16", None), (4, "f32", None), (4, "bf16", None),
                                         (8, "f32", None), (16, "bf16", None), (4, "f32", "f32")])
@pytest.mark.parametrize("p", [0.25, 0.6])
def test_resident_warp_kernel_with_a_padded_coordinate_major_image(N, dtype, opt, p):
    """[P][N]: from half of the coordinates on the shared-memory image is padded against bank conflicts where a group is a
    multiple of 128 bytes (64 in two stacks): N = 8 in fp32, 16 in bf16, two fp32 stacks of N = 4 at p = 0.6; the
    small-group streaming kernel, forced here, fetches and serves a padded image by a path of its own."""
    c = Case(N, [300_007, 12, 40_000], 1, dtype, opt, seed=90 + N)
    B.wash_set_launch(c.gpu.ctx, 0, -4)
    shuffle = B.wash_shuffle_both if opt else B.wash_shuffle
    tot = [0, 0]
    for step in (0, 1):
        shuffle(c.gpu.ctx, step, p, None, seed=5, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, p, seed=5, step=step, stack2=c.host_opt)
        tot[0] += s[0]; tot[1] += s[1]
        c.assert_equal("N=%d %s step=%d" % (N, dtype, step))
    assert c.gpu_stats() == tuple(tot)
    c.close()


@pytest.mark.parametrize("N", [2, 4])
def test_shards_reproduce_the_unsharded_shuffle(N):
    """Coordinate shards keyed by the global (tensor, coordinate) need no communication
    (N = 2 goes through the streaming kernel for small groups, N = 4 through the one-trip kernel)."""
    numel = [4000, 1000, 36]
    full = Case(N, numel, 0, seed=6)
    dense = W.from_stack(full.host, N, numel, full.off, full.P)
    oracle.shuffle(full.ora, full.host, 0.3, seed=77, step=5)
    want = W.from_stack(full.host, N, numel, full.off, full.P)
    # shard A: tensor 0 [0, 2000) ; shard B: tensor 0 [2000, 4000), tensor 1, tensor 2
    shards = [([2000], [0], [0], dense[:, :2000]),
              ([2000, 1000, 36], [0, 1, 2], [2000, 0, 0], dense[:, 2000:])]
    got = []
    for nm, tid, cb, d in shards:
        c = Case(N, nm, 0, tensor_id=tid, coord_begin=cb, dense=np.ascontiguousarray(d))
        B.wash_shuffle(c.gpu.ctx, 5, 0.3, None, seed=77)
        torch.cuda.synchronize()
        host = to_host_bits(c.dev).view(np.float32)
        got.append(W.from_stack(host, N, nm, c.off, c.P))
        c.close()
    assert (np.concatenate(got, axis=1).view(np.uint32) == want.view(np.uint32)).all()
    full.close()


def test_config1_hundred_steps_then_ema_and_average():
    """N = 3, one flat fp32 vector of 2^20 elements, N(0, 0.05), p = 0.01, 100 steps with
    the step index as the RNG counter; then PAPA's EMA and the final average."""
    N, d = 3, 1 << 20
    c = Case(N, [d], 0, dense=W.flat_population(N, d, seed=0, std=0.05))
    tot = [0, 0]
    for step in range(100):
        B.wash_shuffle(c.gpu.ctx, step, 0.01, None, seed=0, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, 0.01, seed=0, step=step)
        tot[0] += s[0]; tot[1] += s[1]
        if step < 10 or step == 99:
            c.assert_equal("step %d" % step)
    assert c.gpu_stats() == tuple(tot)
    for alpha in (0.99, 0.01):
        B.papa_ema(c.gpu.ctx, B.WASH_STACK_PARAMS, alpha)
        oracle.papa_ema(c.ora, c.host, alpha)
        c.assert_equal("ema %g" % alpha)     # designed to be bit-exact; the bar is 2 ulp
    out = torch.zeros(c.P, dtype=torch.float32, device="cuda")
    B.population_average(c.gpu.ctx, B.WASH_STACK_PARAMS, out, B.WASH_F32)
    want = np.zeros(c.P, dtype=np.float32)
    oracle.population_average(c.ora, c.host, want)
    assert (to_host_bits(out) == want.view(np.uint32)).all()
    c.close()


def test_argument_and_state_errors():
    ctx = B.wash_create(3, [100])
    with pytest.raises(B.WashError) as e:
        B.wash_shuffle(ctx, 0, 0.5)
    assert e.value.code == B.WASH_ERR_STATE
    P, _ = B.wash_stack_elems(ctx, 1)
    t = torch.zeros(3 * P, device="cuda")
    with pytest.raises(B.WashError) as e:
        B.wash_bind(ctx, 0, B.WASH_F32, t, 3 * P - 1)
    assert e.value.code == B.WASH_ERR_ARG
    B.wash_bind(ctx, 0, B.WASH_F32, t, 3 * P)
    for bad in (dict(p=1.5), dict(p=float("nan")), dict(p=-0.1), dict(p=0.5, step=1 << 56), dict(p=0.5, p_layer=[2.0])):
        with pytest.raises(B.WashError) as e:
            B.wash_shuffle(ctx, bad.get("step", 0), bad["p"], bad.get("p_layer"))
        assert e.value.code == B.WASH_ERR_ARG
    with pytest.raises(B.WashError) as e:
        B.wash_shuffle_both(ctx, 0, 0.5)
    assert e.value.code == B.WASH_ERR_STATE
    with pytest.raises(B.WashError):
        B.papa_ema(ctx, 0, 1.0)
    assert (t == 0).all()
    B.wash_check(ctx)
    B.wash_destroy(ctx)


def test_a_rejected_probability_vector_leaves_the_context_consistent():
    """A call refused for one bad entry of p_layer must not change the thresholds the next
    call compares with: the following valid call (which repeats the good entries) has to
    upload its table and match the oracle."""
    N, numel = 4, [3000, 2000, 500]
    c = Case(N, numel, 0, "f32", "f32", seed=13)
    B.wash_shuffle_both(c.gpu.ctx, 0, 0.0, [0.1, 0.1, 0.1], seed=3, stats=c.stats_dev)
    st = list(oracle.shuffle(c.ora, c.host, [0.1, 0.1, 0.1], seed=3, step=0, stack2=c.host_opt))
    for bad in ([0.5, 2.0, 0.0], [0.5, 0.25, float("nan")]):
        with pytest.raises(B.WashError) as e:
            B.wash_shuffle_both(c.gpu.ctx, 1, 0.0, bad, seed=3, stats=c.stats_dev)
        assert e.value.code == B.WASH_ERR_ARG
    c.assert_equal("after the refused calls")          # nothing ran
    for step, pl in ((1, [0.5, 0.0, 0.0]), (2, [0.5, 0.25, 0.0]), (3, [0.1, 0.1, 0.1])):
        B.wash_shuffle_both(c.gpu.ctx, step, 0.0, pl, seed=3, stats=c.stats_dev)
        s = oracle.shuffle(c.ora, c.host, pl, seed=3, step=step, stack2=c.host_opt)
        st[0] += s[0]; st[1] += s[1]
        c.assert_equal("step %d" % step)
    assert c.gpu_stats() == tuple(st)
    c.close()


def test_resume_from_a_host_copy_continues_bit_identically():
    """The shuffle is a pure function of (stack bits, seed, step, tensor table, p): 20 steps
    in one context equal 10 steps, a round trip of the stacks through host memory into a
    fresh context, and 10 more steps."""
    N, numel = 5, [3000, 17, 640]
    a = Case(N, numel, 0, "f32", "f32", seed=31)
    for step in range(20):
        B.wash_shuffle_both(a.gpu.ctx, step, 0.05, None, seed=77)
    b = Case(N, numel, 0, "f32", "f32", seed=31)
    for step in range(10):
        B.wash_shuffle_both(b.gpu.ctx, step, 0.05, None, seed=77)
    torch.cuda.synchronize()
    saved, saved_opt = b.dev.cpu(), b.dev_opt.cpu()
    b.close()
    c = Case(N, numel, 0, "f32", "f32", seed=99)          # different contents, overwritten below
    c.dev.copy_(saved); c.dev_opt.copy_(saved_opt)
    for step in range(10, 20):
        B.wash_shuffle_both(c.gpu.ctx, step, 0.05, None, seed=77)
    torch.cuda.synchronize()
    assert torch.equal(a.dev.view(torch.int32), c.dev.view(torch.int32))
    assert torch.equal(a.dev_opt.view(torch.int32), c.dev_opt.view(torch.int32))
    a.close(); c.close()


def test_auto_mode_takes_either_kernel_and_keeps_the_bits():
    """WASH_MODE_AUTO picks the sparse kernel below a share of expected selection (N = 6 in [N][P]:
    5.8 %) and the streaming one above; a per-layer vector is judged by its expectation over the whole model."""
    N = 6
    numel = [70000, 9, 3000]
    c = Case(N, numel, 0, "f32", "f32", seed=21)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_AUTO)
    for step, (p, pl) in enumerate([(0.001, None), (0.5, None), (0.0, [0.01, 1.0, 0.2]), (0.0, [0.2, 0.0, 0.0])]):
        B.wash_shuffle_both(c.gpu.ctx, step, p, pl, seed=77, stats=c.stats_dev)
        oracle.shuffle(c.ora, c.host, p if pl is None else pl, seed=77, step=step, stack2=c.host_opt)
        c.assert_equal("step %d" % step)
    c.close()


@pytest.mark.parametrize("seed", [11, 12, 13])
def test_random_configurations_match_oracle(seed):
    """Seeded random draws of population size, layout, dtypes, tensor table, probabilities (uniform
    or per layer), kernel family and forced streaming flavour: stacks, padding and counters equal
    the oracle's after two steps each."""
    import random
    rng = random.Random(seed)
    for it in range(40):
        N = rng.choice([2, 2, 3, 3, 4, 4, 5, 6, 8, 9, 12, 16, 17, 24, 32, 33])
        layout = rng.randint(0, 1)
        dtype = rng.choice(["f32", "bf16"])
        opt = rng.choice([None, None, "f32", "bf16"])
        T = rng.randint(1, 6)
        big = rng.choice([20000, 200000, 700000 if N <= 8 else 60000])
        numel = [rng.choice([1, 3, 4, 5, 8, 31, 33, 260, 4099, rng.randint(1, big)]) for _ in range(T)]
        numel[rng.randrange(T)] = rng.randint(big // 2, big)
        mode = rng.choice([B.WASH_MODE_STREAM, B.WASH_MODE_STREAM, B.WASH_MODE_SPARSE, B.WASH_MODE_AUTO])
        code = rng.choice([0, 0, -4, -5, -2, -3])
        uniform = rng.random() < 0.5
        p = rng.choice([0.0005, 0.003, 0.01, 0.03, 0.1, 0.25, 0.6, 1.0]) if uniform else 0.0
        pl = None if uniform else [rng.choice([0.0, 0.002, 0.01, 0.05, 0.3, 1.0]) for _ in range(T)]
        what = "seed %d case %d: N=%d layout=%d %s/%s numel=%s mode=%d code=%d p=%s" % (seed, it, N, layout, dtype, opt, numel, mode, code, p if uniform else pl)
        c = Case(N, numel, layout, dtype, opt, seed=1000 * seed + it)
        B.wash_set_mode(c.gpu.ctx, mode)
        B.wash_set_launch(c.gpu.ctx, 0, code)
        tot = [0, 0]
        for step in (it, (it << 33) | 7):
            if opt is None:
                B.wash_shuffle(c.gpu.ctx, step, p, pl, seed=it * 77 + 1, stats=c.stats_dev)
            else:
                B.wash_shuffle_both(c.gpu.ctx, step, p, pl, seed=it * 77 + 1, stats=c.stats_dev)
            s = oracle.shuffle(c.ora, c.host, p if uniform else pl, seed=it * 77 + 1, step=step, stack2=c.host_opt)
            tot[0] += s[0]; tot[1] += s[1]
            c.assert_equal(what)
        assert c.gpu_stats() == tuple(tot), what
        B.wash_check(c.gpu.ctx)
        c.close()


@pytest.mark.parametrize("N,dtype,opt,layout,p", [(5, "f32", None, 1, 0.01), (6, "f32", None, 0, 0.01), (12, "bf16", None, 0, 0.03), (10, "bf16", None, 1, 0.02),
                                                  (3, "f32", "f32", 1, 0.01), (8, "bf16", None, 0, 0.1), (4, "f32", None, 1, 0.1)])
def test_groups_of_49_to_96_bytes_by_default(N, dtype, opt, layout, p):
    c = Case(N, [260_003, 17, 9000], layout, dtype, opt, seed=N)
    call = B.wash_shuffle if opt is None else B.wash_shuffle_both
    call(c.gpu.ctx, 2, p, None, seed=6, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p, seed=6, step=2, stack2=c.host_opt)
    c.assert_equal("N=%d" % N)
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("captured", [False, True], ids=["stream", "graph"])
def test_calls_that_follow_each_other_at_once(captured):
    """Kernels are launched so that one may start while the one before it ends: a chain of calls on shared stacks with
    other kernels, copies and changes of the probabilities (a table upload) in between must see every result before it,
    launched on a side stream and replayed from a graph (no upload there: the probabilities stay)."""
    N, numel = 5, [120_001, 64, 30_003]
    c = Case(N, numel, 0, "f32", "f32", seed=3)
    avg = torch.zeros(c.P, dtype=torch.float32, device="cuda")
    seen, scale = [torch.zeros_like(avg) for _ in range(4)], torch.full((1,), 0.5, device="cuda")

    def chain(stream):
        for i in range(4):
            B.wash_set_mode(c.gpu.ctx, (B.WASH_MODE_SPARSE, B.WASH_MODE_STREAM)[i & 1])
            p = 0.05 if captured else (0.05, 0.05, 0.2, 0.01)[i]
            B.wash_shuffle_both(c.gpu.ctx, i, p, None, seed=4, stream=stream, stats=c.stats_dev)
            B.wash_shuffle(c.gpu.ctx, 100 + i, p, None, seed=4, stream=stream, stats=c.stats_dev)
            B.papa_ema(c.gpu.ctx, B.WASH_STACK_PARAMS, 0.75, stream=stream)
            if i == 2:
                c.dev.mul_(scale)                              # another library's kernel between two of ours
            B.population_average(c.gpu.ctx, B.WASH_STACK_PARAMS, avg, B.WASH_F32, stream=stream)
            seen[i].copy_(avg)

    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    repeats = 1
    if captured:
        B.wash_shuffle(c.gpu.ctx, 7, 0.05, None, seed=4, stream=s)      # the table is uploaded before the capture
        oracle.shuffle(c.ora, c.host, 0.05, seed=4, step=7)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            chain(s)
        torch.cuda.current_stream().wait_stream(s)
        repeats = 3
        for _ in range(repeats):
            g.replay()
    else:
        with torch.cuda.stream(s):
            chain(s)
    torch.cuda.synchronize()
    tot, want = [0, 0], np.zeros(c.P, dtype=np.float32)
    for _ in range(repeats):
        for i in range(4):
            p = 0.05 if captured else (0.05, 0.05, 0.2, 0.01)[i]
            for st in (oracle.shuffle(c.ora, c.host, p, seed=4, step=i, stack2=c.host_opt), oracle.shuffle(c.ora, c.host, p, seed=4, step=100 + i)):
                tot[0] += st[0]; tot[1] += st[1]
            oracle.papa_ema(c.ora, c.host, 0.75)
            if i == 2:
                c.host *= np.float32(0.5)
            oracle.population_average(c.ora, c.host, want)
            got = to_host_bits(seen[i])
            if repeats == 1:
                assert (got == bits(want)).all(), i
    assert (to_host_bits(seen[3]) == bits(want)).all()
    got, h = to_host_bits(c.dev), bits(c.host)
    finite = ~np.isnan(c.host.reshape(-1))
    assert (got[finite] == h[finite]).all()
    assert (to_host_bits(c.dev_opt) == bits(c.host_opt)).all()
    assert c.gpu_stats() == tuple(tot)
    c.close()


@pytest.mark.parametrize("mode", [B.WASH_MODE_STREAM, B.WASH_MODE_SPARSE], ids=["stream", "sparse"])
@pytest.mark.parametrize("N,p", [(2, 0.02), (5, 0.01), (8, 0.001), (20, 0.001), (20, 0.5)])
def test_counters_in_mapped_host_memory(N, p, mode):
    """The counts are the oracle's, call after call, and a launch does not pay an atomic over PCIe (a microsecond each) per
    reporting block: with counters in pinned memory it takes no more than three times as long as with counters on the
    device, plus 50 us (one more kernel and a few such atomics; with one per block it was 430 us and more)."""
    numel = [400_001, 300]
    c = Case(N, numel, seed=N)
    B.wash_set_mode(c.gpu.ctx, mode)
    pinned = torch.zeros(2, dtype=torch.int64).pin_memory()
    want = np.zeros(2, dtype=np.int64)
    for step in range(2):
        B.wash_shuffle(c.gpu.ctx, step, p, None, seed=3, stats=pinned)
        want += np.array(oracle.shuffle(c.ora, c.host, p, seed=3, step=step), dtype=np.int64)
    c.assert_equal("N=%d" % N)
    assert (pinned.numpy() == want).all()

    def us(stats):
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for i in range(10):
                B.wash_shuffle(c.gpu.ctx, i, p, None, seed=3, stats=stats)
            b.record()
            b.synchronize()
            best = min(best, 100.0 * a.elapsed_time(b))
        return best
    on_device, in_host_memory = us(c.stats_dev), us(pinned)
    assert in_host_memory < 3 * on_device + 50, (in_host_memory, on_device)
    c.close()


def test_counters_in_mapped_host_memory_without_a_context():
    for N, p in ((3, 0.02), (8, 0.001)):
        c = Case(N, [300_001, 9], seed=N)
        pinned = torch.zeros(2, dtype=torch.int64).pin_memory()
        B.wash_shuffle_noalloc(N, c.numel, 0, B.WASH_F32, c.dev, c.dev.numel(), 5, p, None, seed=2, stats=pinned)
        want = oracle.shuffle(c.ora, c.host, p, seed=2, step=5)
        c.assert_equal("N=%d" % N)
        assert tuple(pinned.tolist()) == tuple(want)
        c.close()


@pytest.mark.parametrize("N,dtype,opt", [(5, "f32", None), (3, "bf16", "f32"), (10, "bf16", None)])
def test_streaming_is_not_bound_by_the_launch_of_its_blocks(N, dtype, opt):
    """A long row, few coordinates selected: the kernel reads the stacks once.  A copy of them (which reads and writes) is the
    measure: half of its time is the bound, 0.50-0.52 was measured, 0.67-0.70 when every block released the next kernel."""
    P = 1 << 24
    pop = B.Population(N, [P], B.WASH_LAYOUT_NP, 0)
    stacks = []
    for role, dt in ((B.WASH_STACK_PARAMS, dtype), (B.WASH_STACK_OPT, opt)):
        if dt:
            stacks.append(torch.zeros(N * P, dtype=torch.float32 if dt == "f32" else torch.bfloat16, device="cuda"))
            pop.bind(role, stacks[-1])
    spare = [torch.empty_like(s) for s in stacks]
    step = B.wash_shuffle_both if opt else B.wash_shuffle

    def us(call):
        best = 1e9
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for i in range(10):
                call(i)
            b.record()
            b.synchronize()
            best = min(best, 100.0 * a.elapsed_time(b))
        return best
    copied = us(lambda i: [d.copy_(s) for d, s in zip(spare, stacks)])
    shuffled = us(lambda i: step(pop.ctx, i, 1e-4, None, seed=1))
    assert shuffled < 0.61 * copied, (shuffled, copied)
    pop.close()


def test_short_launches_that_follow_each_other_stay_spread_over_the_gpu():
    """EMA of small populations, call after call: no slower than the same calls with another library's
    kernel between them (which keeps them from overlapping), less that kernel's own time, with 30 % and 1 us for noise
    (6.4, 10.2 and 8.2 us a call were measured, 13.9, 20.6 and 16.0 when every launch let the next one start before its own wait)."""
    for N, dtype, layout in ((16, "bf16", 0), (20, "bf16", 1), (24, "bf16", 0)):
        c = Case(N, [1 << 17], layout, dtype, seed=N)
        scratch = torch.zeros(1 << 16, device="cuda")

        def us(call):
            best = 1e9
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for i in range(100):
                    call()
                b.record()
                b.synchronize()
                best = min(best, 10.0 * a.elapsed_time(b))
            return best
        chained = us(lambda: B.papa_ema(c.gpu.ctx, 0, 0.9))
        apart = us(lambda: (B.papa_ema(c.gpu.ctx, 0, 0.9), scratch.zero_())) - us(lambda: scratch.zero_())
        assert chained < 1.3 * apart + 1.0, (N, chained, apart)
        c.close()


@pytest.mark.parametrize("N,layout,numel,p,dtype,opt", [
    (2, 1, [70_001, 9], 0.3, "f32", None), (3, 1, [511], 1.0, "f32", None), (4, 1, [2_000_003, 33], 0.16, "f32", None), (5, 1, [512, 7], 0.9, "bf16", None),
    (8, 1, [100_003], 0.45, "bf16", None), (10, 1, [513, 60_001], 0.31, "f32", None), (12, 1, [30_001, 1, 5], 1.0, "bf16", None), (15, 1, [40_001], 0.8, "f32", None),
    (18, 0, [200_001, 31], 0.06, "f32", None), (20, 0, [2_047, 90_001], 0.2, "bf16", "f32"), (32, 0, [100_003], 0.39, "bf16", None), (33, 0, [65_537, 9], 0.1, "f32", "f32"),
    (64, 0, [70_003], 0.026, "f32", None), (64, 0, [511], 0.1, "bf16", "bf16")])
def test_sparse_warps_that_serve_by_themselves(N, layout, numel, p, dtype, opt):
    """Dense selections of the sparse kernel, a warp's list from tile to tile: lists of a full tile and none, ranges that
    end inside a tile and a tensor, more warps than tiles, permutations packed and in shared memory; also twice in a row."""
    c = Case(N, numel, layout, dtype, opt, seed=N + 3)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_SPARSE)
    want = np.zeros(2, dtype=np.int64)
    for step in (0, 1):
        (B.wash_shuffle_both if opt else B.wash_shuffle)(c.gpu.ctx, step, p, None, seed=21, stats=c.stats_dev)
        want += np.array(oracle.shuffle(c.ora, c.host, p, seed=21, step=step, stack2=c.host_opt), dtype=np.int64)
    c.assert_equal("N=%d layout=%d p=%g" % (N, layout, p))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("N,tiles", [(2, 1), (2, 300), (2, 148 * 22 - 1), (2, 148 * 22), (2, 148 * 22 + 1), (3, 1500), (3, 2400)])
def test_resident_warps_with_one_tile_and_with_more(N, tiles):
    """As many warps as tiles, where masks are drawn before the wait for the kernel before, and one tile more; the counters,
    a word per slot, over calls that follow each other at once."""
    c = Case(N, [512 * tiles - 3], 0, seed=N)
    B.wash_set_launch(c.gpu.ctx, 0, -4)
    want = np.zeros(2, dtype=np.int64)
    for step in range(4):
        B.wash_shuffle(c.gpu.ctx, step, 0.05, None, seed=3, stats=c.stats_dev)
    for step in range(4):
        want += np.array(oracle.shuffle(c.ora, c.host, 0.05, seed=3, step=step), dtype=np.int64)
    c.assert_equal("N=%d tiles=%d" % (N, tiles))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("N,numel,p,dtype,opt", [
    (20, [30_001], 0.1, "bf16", None), (24, [9_001, 2], 0.5, "f32", None), (28, [253, 4, 3000], 0.9, "f32", None), (32, [40_009], 0.02, "f32", None),
    (32, [16_390], 0.3, "bf16", "f32"), (36, [8_191], 0.6, "f32", "f32"), (48, [10_003], 0.4, "bf16", None), (60, [5_001], 0.2, "f32", "bf16"), (64, [4_099], 0.65, "f32", None), (47, [6_001], 0.5, "f32", None)])
def test_wide_populations_coordinate_major(N, numel, p, dtype, opt):
    """[P][N], N > 16: four models to a thread, the block's permutations drawn by some of its warps in one and in several
    rounds, one and two threads to a group, and a population that is no multiple of four."""
    c = Case(N, numel, 1, dtype, opt, seed=N)
    for step in (0, 1):
        (B.wash_shuffle_both if opt else B.wash_shuffle)(c.gpu.ctx, step, p, None, seed=8, stats=c.stats_dev)
    want = np.array(oracle.shuffle(c.ora, c.host, p, seed=8, step=0, stack2=c.host_opt), dtype=np.int64)
    want += np.array(oracle.shuffle(c.ora, c.host, p, seed=8, step=1, stack2=c.host_opt), dtype=np.int64)
    c.assert_equal("N=%d p=%g" % (N, p))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,p,dtype,opt", [(2, 0.03, "f32", None), (5, 0.004, "f32", "f32"), (8, 0.01, "bf16", "f32"), (16, 0.02, "bf16", None), (20, 0.05, "f32", None),
                                           (32, 0.001, "f32", "bf16"), (64, 0.004, "bf16", None), (3, 0.0004, "f32", None), (5, 0.0002, "f32", "f32")])
def test_sparse_loads_of_half_lines(N, p, dtype, opt, layout):
    """Selections about which the sparse kernel's loads ask for 64 bytes (pairs, rows and warps that serve by themselves) and
    two that are too rare for it; three steps in a row, the second drawing while the first still serves."""
    numel = [700_001, 9, 120_000] if N <= 16 else [150_001, 9]
    c = Case(N, numel, layout, dtype, opt, seed=N)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_SPARSE)
    want = np.zeros(2, dtype=np.int64)
    for step in range(3):
        (B.wash_shuffle_both if opt else B.wash_shuffle)(c.gpu.ctx, step, p, None, seed=17, stats=c.stats_dev)
        want += np.array(oracle.shuffle(c.ora, c.host, p, seed=17, step=step, stack2=c.host_opt), dtype=np.int64)
    c.assert_equal("N=%d p=%g layout=%d" % (N, p, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


def _half_wave_row(at_least_blocks_over=1.5):
    """Coordinates for which a launch of a warp tile (512 coordinates) a warp would take more blocks of four warps than half a wave
    holds (eight blocks an SM are a wave)."""
    half = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    return int(at_least_blocks_over * half) * 4 * 512 + 3


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N,p,dtype,opt", [(2, 1e-3, "f32", None), (3, 4e-4, "bf16", None), (5, 2e-4, "f32", "f32"), (8, 3e-4, "bf16", "f32"), (16, 2e-4, "f32", None), (20, 2e-4, "bf16", None), (40, 1e-4, "bf16", None)])
def test_sparse_half_a_wave_of_blocks(N, p, dtype, opt, layout):
    """Selections rare enough for half a wave of blocks, in rows that would fill more, three steps in a row: the
    second draws its masks beside the first one's serving."""
    c = Case(N, [_half_wave_row(), 5, 2047], layout, dtype, opt, seed=N)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_SPARSE)
    want = np.zeros(2, dtype=np.int64)
    for step in range(3):
        (B.wash_shuffle_both if opt else B.wash_shuffle)(c.gpu.ctx, step, p, None, seed=23, stats=c.stats_dev)
        want += np.array(oracle.shuffle(c.ora, c.host, p, seed=23, step=step, stack2=c.host_opt), dtype=np.int64)
    c.assert_equal("N=%d p=%g layout=%d" % (N, p, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("N", [2, 5, 16])
def test_sparse_half_a_wave_with_everything_selected_in_one_place(N, layout):
    """A schedule that is rare on the whole, and selects in one tensor what fills the queue (512 entries) of the block whose range it is
    several times over."""
    c = Case(N, [_half_wave_row() // 2, 1900, _half_wave_row() // 2], layout, "f32", "f32", seed=N)
    B.wash_set_mode(c.gpu.ctx, B.WASH_MODE_SPARSE)
    p_layer = [1e-5, 1.0, 1e-5]
    want = np.zeros(2, dtype=np.int64)
    for step in range(2):
        B.wash_shuffle_both(c.gpu.ctx, step, 0.0, p_layer, seed=29, stats=c.stats_dev)
        want += np.array(oracle.shuffle(c.ora, c.host, p_layer, seed=29, step=step, stack2=c.host_opt), dtype=np.int64)
    c.assert_equal("N=%d layout=%d" % (N, layout))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("code", [-4, -5], ids=["resident", "one-trip"])
@pytest.mark.parametrize("dtype,opt", [("f32", None), ("bf16", None), ("f32", "bf16"), ("bf16", "f32"), ("f32", "f32")])
@pytest.mark.parametrize("N", [2, 4, 6, 8, 10, 14, 16])
def test_neighbouring_models_stored_together(N, dtype, opt, code):
    """[P][N], dealt serving: two or four models' values with one store (N even, N a multiple of 4), fixed points
    among them, counted as not moved; in tensors that end inside a group, and up to the selection that is served densely or, with
    two stacks of 8 models and more, is not."""
    c = Case(N, [9001, 3, 130, 2046, 3001], 1, dtype, opt, seed=N)
    B.wash_set_launch(c.gpu.ctx, 0, code)
    p_layer = [0.1, 1.0, 0.45, 0.25, 0.9]
    (B.wash_shuffle_both if opt else B.wash_shuffle)(c.gpu.ctx, 4, 0.0, p_layer, seed=5, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p_layer, seed=5, step=4, stack2=c.host_opt)
    c.assert_equal("N=%d %s/%s" % (N, dtype, opt))
    assert c.gpu_stats() == tuple(want)
    c.close()


@pytest.mark.parametrize("code", [-4, -5], ids=["resident", "one-trip"])
@pytest.mark.parametrize("N,dtype,opt", [(2, "f32", None), (2, "bf16", "f32"), (4, "bf16", None), (4, "bf16", "f32"), (6, "f32", "f32"), (8, "f32", None), (10, "bf16", None), (14, "f32", "bf16")])
def test_dense_serving_by_the_tensors_threshold(N, dtype, opt, code):
    """[P][N], even populations: neighbouring tensors on both sides of the threshold from which a tensor is served densely (0.56 of the coordinates for two
    models, 0.78 to 0.87 above), small ones, so that warps hold groups of both, ragged ones, and one whose threshold is reached by none of its words."""
    c = Case(N, [130, 7, 1021, 64, 300, 5003, 12, 260, 900, 33, 2050], 1, dtype, opt, seed=N)
    B.wash_set_launch(c.gpu.ctx, 0, code)
    p_layer = [0.55, 0.57, 0.5, 0.79, 0.77, 0.9, 1.0, 0.86, 0.88, 0.0, 0.8]
    (B.wash_shuffle_both if opt else B.wash_shuffle)(c.gpu.ctx, 3, 0.0, p_layer, seed=11, stats=c.stats_dev)
    want = oracle.shuffle(c.ora, c.host, p_layer, seed=11, step=3, stack2=c.host_opt)
    c.assert_equal("N=%d %s/%s" % (N, dtype, opt))
    assert c.gpu_stats() == tuple(want)
    c.close()
