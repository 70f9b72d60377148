"""The step as one kernel: sizes at the edges of the in-kernel compaction (words of the bitmap,
the largest number of positions it takes, masks at any address), of the claimed rows and of the
merge, against the oracle."""
import pytest
import torch

import workloads as WL
from oracle import rpd_oracle as O

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from gpu_util import DeviceRunner, bits  # noqa: E402
from parity import compare_block_step, compare_step  # noqa: E402


def make(seed, K, N, d, V):
    W, g = WL.make_head(V, d, seed, w_std=0.08)
    cv = WL.make_hidden(W, K, N, seed + 1000, WL.u_profile(N, 0.5, 3.0),
                        WL.calibrated_sigma(V, d, 0.08, 3.0), flip_frac=0.1)
    return W, g, cv.hidden


@pytest.mark.parametrize("N,count", [(1, 1), (15, 7), (16, 16), (31, 2), (33, 33), (64, 1), (320, 200),
                                     (321, 9)])
@pytest.mark.parametrize("offset", [0, 1, 8])
def test_compaction_at_word_edges_and_any_mask_address(N, count, offset):
    K, d, V = 2, 128, 1024
    W, g, hidden = make(700 + N, K, N, d, V)
    mask = WL.uniform_fraction_mask(N, count / N, N)
    ref = O.rpd_step(bits(hidden), mask.numpy(), bits(g), bits(W), 1e-6, 0.9, 1.0, "llada")
    runner = DeviceRunner(W, g, K)
    try:
        room = torch.zeros(N + 32, dtype=torch.uint8, device="cuda")
        m = room[offset:offset + N]
        m.copy_(mask)
        h = hidden.cuda()
        out = runner._alloc(1, N)
        runner.ctx.step(h, m, 0.9, 1.0, out["commit"][0], out["token"][0], out["stats"][0])
        got = runner._fetch(out, m.reshape(1, N), 1)[0]
        assert int(room.sum()) == int(m.sum())  # nothing beside the mask was written
    finally:
        runner.close()
    compare_step(ref, got)


@pytest.mark.parametrize("B,N", [(8, 1024), (9, 911), (3, 2731)])  # 8192, 8199 and 8193 positions
@pytest.mark.parametrize("block", [0, 32])
def test_batches_around_the_compaction_limit(B, N, block):
    K, d, V = 1, 64, 512
    W, g = WL.make_head(V, d, 41, w_std=0.08)
    gen = torch.Generator().manual_seed(B)
    hidden = torch.randn(K, B, N, d, generator=gen).to(torch.bfloat16) * 2
    masks = torch.stack([WL.uniform_fraction_mask(N, 0.02 + 0.9 * b / B, 50 + b) for b in range(B)])
    masks[1] = 0
    runner = DeviceRunner(W, g, K, rule="llada_block" if block else "llada")
    try:
        got = runner.step_batched(hidden, masks, [0.9] * B, [1.5] * B)
    finally:
        runner.close()
    for b in (0, 1, 2, B - 1):
        args = (bits(hidden[:, b].contiguous()), masks[b].numpy(), bits(g), bits(W), 1e-6, 0.9)
        ref = O.rpd_block_step(*args, "llada", block) if block else O.rpd_step(*args, 1.5, "llada")
        (compare_block_step if block else compare_step)(ref, got[b])
        assert got[b]["stats"]["n_rows"] == got[0]["stats"]["n_rows"]


def test_more_rows_than_the_grid_has_warps_and_splits_of_every_width():
    """Rows that warps claim several at a time (over 2432), and merges of 1 to 32 lanes per row."""
    for V, N in [(300, 640), (2048, 650), (20000, 5)]:
        K, d = 4, 64
        W, g, hidden = make(90 + N, K, N, d, V)
        mask = torch.ones(N, dtype=torch.uint8)
        ref = O.rpd_step(bits(hidden), mask.numpy(), bits(g), bits(W), 1e-6, 0.9, 1.0, "llada")
        runner = DeviceRunner(W, g, K)
        try:
            compare_step(ref, runner.step(hidden, mask, 0.9, 1.0))
        finally:
            runner.close()


@pytest.mark.parametrize("tau,prefix", [(0.9, 0), (0.62, 0), (0.9, 96)])  # a band, a thin one, nothing masked
@pytest.mark.parametrize("projection", ["lazy", "auto"])
@pytest.mark.parametrize("N", [96, 700])
def test_two_pass_steps_one_after_another(N, projection, tau, prefix):
    """The first pass selects the second's positions, or scores the canvas itself when there are
    none; the steps that follow on the same context find its counters as they should be."""
    K, d, V = 6, 128, 2048
    W, g, hidden = make(60 + N, K, N, d, V)
    mask = torch.ones(N, dtype=torch.uint8)
    if prefix:
        mask[:] = 0
    runner = DeviceRunner(W, g, K)
    try:
        for mode in (projection, "all", projection):
            runner.ctx.set_projection(mode)
            got = runner.step(hidden, mask, tau, 1.0)
            ref = O.rpd_step(bits(hidden), mask.numpy(), bits(g), bits(W), 1e-6, tau, 1.0, "llada")
            lazy = got["stats"]["n_rows"] < K * int(mask.sum())
            compare_step(ref, got, lazy=lazy)
    finally:
        runner.close()


@pytest.mark.parametrize("V,N,d", [(4100, 200, 128),    # under half a wave: only half tiles, the last one empty
                                   (9728, 200, 128),    # half a wave exactly
                                   (20480, 200, 128),   # one wave and four tiles: whole tiles only at this depth,
                                   (19713, 300, 128),   # here too
                                   (9728, 600, 128),    # and here
                                   (20480, 400, 4096),  # two waves and eight tiles of two row tiles
                                   (19713, 500, 4096),  # two waves and four tiles, a last half tile of one entry
                                   (15872, 748, 4096)]) # three row tiles of 62: two waves and 34 tiles
def test_pair_tiles_with_a_split_tail(V, N, d):
    """Whole waves of pair tiles and a rest of half tiles, whose rows have two partials per tile."""
    K = 1
    w_std = 0.08 if d < 1024 else 0.02
    W, g = WL.make_head(V, d, 800 + N, w_std=w_std)
    hidden = WL.make_hidden(W, K, N, 1800 + N, WL.u_profile(N, 0.5, 3.0), WL.calibrated_sigma(V, d, w_std, 3.0),
                            flip_frac=0.1).hidden
    mask = torch.ones(N, dtype=torch.uint8)
    ref = O.rpd_step(bits(hidden), mask.numpy(), bits(g), bits(W), 1e-6, 0.9, 1.0, "llada")
    runner = DeviceRunner(W, g, K)
    try:
        got = runner.step(hidden, mask, 0.9, 1.0)
        runner.ctx.set_head_tiling("pair")  # without the split
        whole = runner.step(hidden, mask, 0.9, 1.0)
    finally:
        runner.close()
    compare_step(ref, got)
    compare_step(ref, whole)


def test_maps_of_many_positions_hold_up_no_step():
    """The compaction's maps (for the kernels after the head kernel) are written by the whole grid:
    8192 positions cost a step a few us more than 64 with as many masked (25 us by a single warp)."""
    K, d, V = 1, 64, 1024
    W, g, _ = make(5, K, 8, d, V)
    runner = DeviceRunner(W, g, K)
    runner.ctx.set_vocab_shard(0, V)
    try:
        times = []
        for N in (64, 8192):
            hidden = torch.zeros(K, N, d, dtype=torch.bfloat16, device="cuda")
            mask = torch.zeros(N, dtype=torch.uint8, device="cuda")
            mask[:32] = 1
            out = torch.zeros(K, N, 4, device="cuda")
            best = 1e9
            for _ in range(30):
                t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                t0.record()
                for _ in range(20):
                    runner.ctx.step_shard_partials(hidden, mask, out)
                t1.record()
                t1.synchronize()
                best = min(best, t0.elapsed_time(t1) / 20 * 1e3)
            times.append(best)
    finally:
        runner.close()
    assert times[1] < times[0] + 12, times


@pytest.mark.parametrize("B,N,projection,launches", [
    (1, 256, "all", 1), (1, 2048, "all", 1), (1, 256, "lazy", 2), (1, 256, "auto", 2),  # everything in the head kernel
    (1, 2049, "all", 2), (1, 8192, "lazy", 3),   # a long canvas, and several, are scored apart
    (8, 1024, "all", 2), (8, 1024, "lazy", 3),
    (9, 911, "all", 3), (9, 911, "lazy", 5)])    # more positions than the head kernel compacts: also compaction, band
def test_kernels_launched_by_a_step(B, N, projection, launches):
    K, d, V = 2, 64, 512
    W, g = WL.make_head(V, d, 3, w_std=0.08)
    gen = torch.Generator().manual_seed(N)
    hidden = torch.randn(K, B, N, d, generator=gen).to(torch.bfloat16) * 2
    masks = torch.stack([WL.uniform_fraction_mask(N, 0.3, 20 + b) for b in range(B)])
    runner = DeviceRunner(W, g, K)
    try:
        runner.ctx.set_projection(projection)
        runner.ctx.profile(True)
        got = runner.step_batched(hidden, masks, [0.9] * B, [1.5] * B)
        count = sum(n for _, n in runner.ctx.kernel_times().values())
    finally:
        runner.close()
    assert count == launches
    for b in {0, B - 1}:
        ref = O.rpd_step(bits(hidden[:, b].contiguous()), masks[b].numpy(), bits(g), bits(W), 1e-6, 0.9, 1.5, "llada")
        compare_step(ref, got[b], lazy=projection != "all" and got[b]["stats"]["n_rows"] < K * int(masks.sum()))


@pytest.mark.parametrize("K,B,N,d,V", [(3, 4, 1000, 72, 300),     # claims of 4 rows, one trip over a row
                                       (2, 4, 1900, 1048, 300),   # claims of 6, a second trip of 3 vectors
                                       (16, 2, 700, 64, 256)])    # claims of 8
def test_claims_of_several_rows_in_a_batch(K, B, N, d, V):
    """Batches of more rows than two a warp, gathered two at a time; the last claim is a part one."""
    W, g = WL.make_head(V, d, 17, w_std=0.08)
    gen = torch.Generator().manual_seed(N)
    hidden = torch.randn(K, B, N, d, generator=gen).to(torch.bfloat16) * 2
    masks = torch.stack([WL.uniform_fraction_mask(N, 0.9, 30 + b) for b in range(B)])
    runner = DeviceRunner(W, g, K)
    try:
        got = runner.step_batched(hidden, masks, [0.9] * B, [1.5] * B)
    finally:
        runner.close()
    for b in (0, B - 1):
        ref = O.rpd_step(bits(hidden[:, b].contiguous()), masks[b].numpy(), bits(g), bits(W), 1e-6, 0.9, 1.5, "llada")
        compare_step(ref, got[b])


def test_many_rows_of_a_batch_are_in_flight_together():
    """A further row of a large batch costs under 1.2 ns (1.5 with one row a warp at a time)."""
    B, N, d, V = 8, 1024, 64, 256
    W, g, _ = make(5, 1, 8, d, V)
    times = []
    for K in (4, 16):
        runner = DeviceRunner(W, g, K)
        try:
            hidden = torch.ones(K, B, N, d, dtype=torch.bfloat16, device="cuda")
            start = torch.ones(B, N, dtype=torch.uint8, device="cuda")
            mask = start.clone()
            commit, token = torch.zeros_like(mask), torch.zeros(B, N, dtype=torch.int32, device="cuda")
            stats = torch.zeros(B, runner.rpd.STATS_WORDS, dtype=torch.int32, device="cuda")
            best = 1e9
            for _ in range(100):
                mask.copy_(start)
                t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                t0.record()
                runner.ctx.step_batched(hidden, mask, [0.9] * B, [1.0] * B, commit, token, stats)
                t1.record()
                t1.synchronize()
                best = min(best, t0.elapsed_time(t1) * 1e6)
            times.append(best)
        finally:
            runner.close()
    assert (times[1] - times[0]) / (12 * B * N) < 1.2, times


@pytest.mark.parametrize("N", [2048, 2049, 8192])
def test_host_buffers_of_long_canvases(N):
    """rpd_step_host equals rpd_step on both sides of the length up to which the head kernel scores."""
    K, d, V = 2, 64, 512
    W, g, hidden = make(30 + N, K, N, d, V)
    runner = DeviceRunner(W, g, K)
    try:
        for count in (N, 700, 1):
            mask = torch.zeros(N, dtype=torch.uint8)
            mask[N - count:] = 1
            want = runner.step(hidden, mask, 0.9, 1.0)
            m, commit = mask.clone(), torch.full((N,), 7, dtype=torch.uint8)
            token = torch.full((N,), -5, dtype=torch.int32)
            stats = torch.zeros(runner.rpd.STATS_WORDS, dtype=torch.int32)
            runner.ctx.step_host(hidden.pin_memory(), m, 0.9, 1.0, commit, token, stats)
            assert (commit.numpy() == want["commit"]).all() and (token.numpy() == want["token"]).all()
            assert (m.numpy() == want["new_mask"]).all() and runner.rpd.stats_dict(stats) == want["stats"]
    finally:
        runner.close()
