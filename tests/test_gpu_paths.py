"""The branches a dispatch on sizes and id ranges can take, each at sizes where it can go wrong, bit
for bit against the oracle."""
import numpy as np
import pytest

from paper_2609_40247_b200 import synth
from runners import DEVICE_MASK
from test_gpu_parity import both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,distinct,spread", [
    (0.02, 700, 700),            # dense rows
    (0.02, 4097, 400_000),       # marked cells: ids in reach of a direct bitmap, few of them used
    (0.02, 1, 1),                # a single symbol
    (0.02, 3000, 1 << 31),       # symbol table, few cells
    (0.05, 90_000, 1 << 31),     # symbol table and marked cells
    (0.08, 140_000, 1 << 31),    # more distinct symbols than the table holds: grouped by sorting
])
def test_aggregate_row_paths(scale, distinct, spread):
    wl = synth.make_workload("c1", scale, truth=False)
    ev = wl.events.copy()
    rng = np.random.default_rng(distinct)
    ids = rng.choice(spread, size=distinct, replace=False) if spread < 10**7 else \
        np.unique(rng.integers(-2**31, 2**31, size=distinct + distinct // 8))
    if distinct > 1:
        ids[0], ids[-1] = ids.min(), ids.max()
        pick = rng.integers(0, len(ids), size=len(ev))
        pick[:len(ids)] = np.arange(len(ids))[:len(pick)]  # every symbol occurs
    else:
        pick = np.zeros(len(ev), dtype=np.int64)
    ev["name_id"] = ids[pick].astype(np.int32)
    o, g = both(ev, wl.win_off, wl.win_t0, wl.win_t1, comm_sizes=wl.comm_sizes, agg_masks=(DEVICE_MASK, 1 << 2, 63))
    assert len(o["agg2_g_count"]) >= min(distinct, len(ev)) // 2


@pytest.mark.parametrize("scale,dup,multi", [(0.004, 0.0, 0.0), (0.02, 0.2, 0.0), (0.02, 0.0, 0.3), (0.1, 0.05, 0.05)])
@pytest.mark.parametrize("hashed", [False, True])
def test_join_with_any_ids_and_several_kernels_per_launch(scale, dup, multi, hashed):
    """Both ways to address the join's table, with launch ids used twice and with launches that own
    several kernels (graph replays: their kernels reach the operators from the device side)."""
    wl = synth.make_workload("c3", scale, truth=False)
    ev = wl.events.copy()
    rng = np.random.default_rng(int(1000 * scale + 10 * dup + 100 * multi))
    joins = np.isin(ev["kind"], (2, 3, 4))
    if hashed:
        with np.errstate(over="ignore"):
            ev["corr_id"][joins] *= np.int64(-7046029254386353131)
        ev["corr_id"][np.nonzero(joins)[0][:2]] = (-2**63, 2**63 - 1)
    for kinds, frac in (((2,), dup), ((3, 4), multi)):
        at = np.nonzero(np.isin(ev["kind"], kinds))[0]
        take = rng.choice(at, size=int(len(at) * frac), replace=False)
        for pid in np.unique(ev["pid"]):
            mine = take[ev["pid"][take] == pid]
            pool = at[ev["pid"][at] == pid]
            if len(mine):
                ev["corr_id"][mine] = ev["corr_id"][rng.choice(pool, size=len(mine))]
    o, g = both(ev, wl.win_off, wl.win_t0, wl.win_t1, comm_sizes=wl.comm_sizes)
    if multi:
        assert int(o["kernels_of_launch"].max()) > 1 and int(o["op_n_kernels"].sum()) > 1000
    if dup:
        assert int(o["join_sum"]["n_dup_launch"].sum()) > 0


@pytest.mark.parametrize("bad", [1, 2, 255, 257, 4097, 16384, 16385])
def test_dropped_tail_ranked_by_counting_and_by_sorting(bad):
    """Dropped records around the size where the tail's order is no longer found by counting, with
    equal tuples among them, in two windows."""
    wl = synth.make_workload("c4", 0.05, truth=False, n_windows=2)
    ev = wl.events.copy()
    rng = np.random.default_rng(bad)
    at = rng.choice(len(ev), size=bad, replace=False)
    ev[at] = ev[rng.choice(at, size=bad)]  # equal records
    ev["kind"][at] = rng.choice((9, -1, 6), size=bad)
    both(ev, wl.win_off, wl.win_t0, wl.win_t1, comm_sizes=wl.comm_sizes)


@pytest.mark.parametrize("n", [104_857, 104_858, 700_001])
def test_pageable_records_around_the_threshold_of_the_staged_upload(n):
    """Host records just below and above four megabytes and over several rings of buffers, twice."""
    from runners import assert_same, run_gpu
    wl = synth.make_workload("c2", 0.05, truth=False)
    ev = np.ascontiguousarray(wl.events[:n])
    assert len(ev) == n
    off = [0, n]
    a = run_gpu(ev, off, wl.win_t0, wl.win_t1, on_device=True)
    for _ in range(2):
        assert_same(a, run_gpu(ev, off, wl.win_t0, wl.win_t1, on_device=False))


@pytest.mark.parametrize("scale,gap", [(0.02, 4_990_000), (0.12, 4_990_000)])
def test_critical_path_with_a_short_and_a_long_list_of_waits(scale, gap):
    """Prefill windows wait once per step: some three thousand waits (walked by one CTA) and some
    twenty thousand (pointer doubling over many)."""
    wl = synth.make_workload("c2", scale, truth=False)
    both(wl.events, wl.win_off, wl.win_t0, wl.win_t1, min_gap=gap)
    assert ((wl.events["kind"] == 1).sum() > 16_384) == (scale > 0.1)


@pytest.mark.parametrize("windows,per", [(2, 20_000), (9, 38_460), (40, 20_000)])
def test_many_windows_counted_by_window_and_lane(windows, per):
    """Batches whose lane histograms come from counts per window and lane, some records dropped."""
    wl = synth.make_workload("c4", per * 512 / (1 << 28), truth=False, n_windows=windows)
    ev = wl.events.copy()
    ev["kind"][::97] = 8
    assert len(ev) // windows >= 8192
    both(ev, wl.win_off, wl.win_t0, wl.win_t1, comm_sizes=wl.comm_sizes)


@pytest.mark.parametrize("n", [1, 511, 512, 513, 1023, 1024, 1025, 1536, 60_001])
def test_records_at_an_odd_eight_bytes(n, monkeypatch):
    """A device buffer that begins at eight bytes past a multiple of sixteen, around the size of the
    tiles that are copied in bulk."""
    import torch
    from paper_2609_40247_b200 import ta

    class Shifted(ta.Window):
        def __init__(self, events, *args, **kw):
            room = torch.zeros(events.numel() + 40, dtype=torch.uint8, device="cuda")
            room[8:8 + events.numel()] = events
            assert room.data_ptr() % 16 == 0
            super().__init__(room[8:8 + events.numel()], *args, **kw)

    monkeypatch.setattr(ta, "Window", Shifted)
    wl = synth.make_workload("c3", 0.002, truth=False)
    ev = np.ascontiguousarray(wl.events[:n])
    assert len(ev) == n
    both(ev, [0, n], wl.win_t0, wl.win_t1, comm_sizes=wl.comm_sizes)


@pytest.mark.parametrize("name,scale", [("c2", 0.004), ("c2", 0.03), ("c3", 0.01)])
def test_operators_with_kernels_far_apart(name, scale):
    """Kernels that start up to seconds after their launch or run for up to seconds: the row's kernel
    times do not fit the 32-bit reductions of the attribution, nor do the lanes end in ascending order."""
    wl = synth.make_workload(name, scale, truth=False)
    ev = wl.events.copy()
    rng = np.random.default_rng(5)
    k = np.nonzero(ev["kind"] == 3)[0]
    late = rng.choice(k, size=len(k) // 50, replace=False)
    shift = rng.integers(0, 3_000_000_000, size=len(late))
    ev["ts_start"][late] += shift
    ev["ts_end"][late] += shift
    long = rng.choice(k, size=len(k) // 50, replace=False)
    ev["ts_end"][long] += rng.integers(0, 1 << 33, size=len(long))
    both(ev, wl.win_off, wl.win_t0, np.asarray(wl.win_t1) + 4_000_000_000, comm_sizes=wl.comm_sizes)


@pytest.mark.parametrize("n", [255, 4_096, 4_097, 8_191, 8_192, 8_193, 16_385, 65_536, 65_537, 131_072, 131_073, 524_289])
def test_one_deep_host_lane_of_many_tiles(n):
    """A single host lane whose operators stay open across hundreds of tiles, around the sizes where
    the stacks in front of a tile are folded by the tile itself, where the attribution's last step
    moves into the operators' launch, and where tiles grow."""
    rng = np.random.default_rng(n)
    ev = np.zeros(n, dtype=synth.EVENT_DTYPE)
    ev["pid"], ev["kind"] = 7, 0
    ev["name_id"] = rng.integers(0, 5, size=n)
    t0, span = 1_000_000, 4 * n + 64
    ev["ts_start"] = t0 + 32 + 4 * np.arange(n)
    ev["ts_end"] = ev["ts_start"] + 1
    enc = 5  # nested operators around everything else
    for d in range(enc):
        ev["ts_start"][d], ev["ts_end"][d] = t0 + d, t0 + span - d
    middle = [enc + (d + 1) * n // 5 for d in range(3)]
    for k in middle:  # and around a seventh of the rest
        ev["ts_end"][k] = ev["ts_start"][min(n - 1, k + n // 7)] - 1
    launch = enc + 1 + np.arange((n - enc - 1) // 3) * 3
    launch = launch[~np.isin(launch, middle)]
    ev["kind"][launch] = 2
    ev["corr_id"][launch] = np.arange(len(launch)) + 5
    dev = launch[rng.random(len(launch)) < 0.5] + 1
    dev = dev[(dev < n) & ~np.isin(dev, middle)]
    ev["kind"][dev], ev["stream"][dev], ev["corr_id"][dev] = 3, 4, ev["corr_id"][dev - 1]
    ev = ev[rng.permutation(n)]
    o, _ = both(ev, np.array([0, n]), np.array([t0]), np.array([t0 + span + 1]))
    assert o["attr_status"] == 0 and int(o["attr_sum"]["max_depth"].max()) >= 6


@pytest.mark.parametrize("run", [1, 2, 3, 31, 32, 33, 47, 48, 49])
@pytest.mark.parametrize("shift", [0, 5])
def test_runs_of_one_coarse_time(run, shift):
    """Records of one lane that begin at the same instant or a few ns apart, in runs inside a warp,
    across its edge and beyond the length that is ranked in place."""
    n = 20_000
    rng = np.random.default_rng(run * 8 + shift)
    ev = np.zeros(n, dtype=synth.EVENT_DTYPE)
    ev["pid"], ev["kind"], ev["stream"] = 3, 3, 1 + (np.arange(n) < shift)
    group = np.arange(n) // run
    ev["ts_start"] = 500 + group * 1_500_000 + rng.integers(0, 3, size=n)
    ev["ts_end"] = ev["ts_start"] + rng.integers(0, 3, size=n)
    ev["corr_id"] = rng.integers(0, 50, size=n)
    ev["name_id"] = rng.integers(0, 9, size=n)
    ev = ev[rng.permutation(n)]
    both(ev, np.array([0, n]), np.array([0]), np.array([int(ev["ts_end"].max()) + 1]))


@pytest.mark.parametrize("n", [2_047, 2_048, 2_049, 4_097, 2_097_152, 2_097_153])
def test_sort_around_its_tiles_and_where_they_grow(n):
    wl = synth.make_workload("c1", max(0.002, 1.03 * n / 4_194_304), truth=False)
    ev = np.ascontiguousarray(wl.events[:n])
    assert len(ev) == n
    both(ev, [0, n], wl.win_t0, wl.win_t1, comm_sizes=wl.comm_sizes)


def _many_small_windows(windows, pids, rng):
    """A few records per process and window: an operator, a launch of two kernels (one of them in
    a third of the windows), a wait, a collective and now and then a damaged record."""
    rows = np.zeros((windows, pids, 6), dtype=synth.EVENT_DTYPE)
    span = 5_000
    t0 = 1_000_000 + span * np.arange(windows, dtype=np.int64)
    at = t0[:, None] + rng.integers(0, 900, size=(windows, pids))
    rows["pid"] = np.arange(pids)[None, :, None]
    rows["name_id"] = rng.integers(0, 7, size=rows.shape)
    for k, (kind, stream, begin, length) in enumerate((
            (0, 0, 0, 2_000), (2, 0, 20, 30), (3, 1, 200, 300), (3, 1, 700, 250), (1, 0, 400, 1_200), (5, 1, 1_100, 100))):
        e = rows[:, :, k]
        e["kind"], e["stream"] = kind, stream
        e["ts_start"] = at + begin + rng.integers(0, 15, size=at.shape)
        e["ts_end"] = e["ts_start"] + length + rng.integers(0, 50, size=at.shape)
    rows["corr_id"][:, :, 1:4] = 5 + rng.integers(0, 3, size=(windows, pids, 1))
    rows["corr_id"][::3, :, 3] = -1
    rows["corr_id"][:, :, 5], rows["seq"][:, :, 5] = 77, rng.integers(0, 2, size=(windows, 1))
    rows["kind"][::5, 0, 4] = 9
    ev = rows.reshape(windows, -1)
    ev = ev[np.arange(windows)[:, None], rng.permuted(np.tile(np.arange(pids * 6), (windows, 1)), axis=1)]
    off = pids * 6 * np.arange(windows + 1, dtype=np.int64)
    return np.ascontiguousarray(ev).reshape(-1), off, t0, t0 + span, [(77, pids)]


@pytest.mark.parametrize("windows,pids", [(86, 16), (1_100, 16), (1_600, 1), (2_500, 1), (3_500, 1), (5_600, 1)])
def test_summaries_too_large_for_the_staging_kernel(windows, pids):
    """Tables of more than 128 KB come back by real copies, behind the call's last kernel: the path
    figures of 1376 processes, the id ranges of 17 600, and the summaries of thousands of windows."""
    from runners import assert_same, run_gpu, run_oracle
    rng = np.random.default_rng(windows)
    ev, off, t0, t1, sizes = _many_small_windows(windows, pids, rng)
    work = (rng.uniform(1e9, 1e12, len(ev)), rng.uniform(1e6, 1e9, len(ev)), synth.PEAK_FLOPS, synth.PEAK_BW)
    o = run_oracle(ev, off, t0, t1, min_gap=100, comm_sizes=sizes, op_work=work)
    g = run_gpu(ev, off, t0, t1, min_gap=100, comm_sizes=sizes, op_work=work)
    assert o["attr_status"] == 0 and int(o["join_sum"]["n_matched"].min()) > 0
    assert int(o["sol_sum"]["n_resolved"].min()) > 0 and int(o["roll_sum"].sum()) > 0
    assert_same(o, g)


def test_hashed_ids_with_a_number_in_their_upper_bits_share_no_chains():
    """Ids that carry a rank or a thread in bits 40 and up, on 64 processes of 32 threads: the join
    takes about as long as with ids of no structure."""
    import time
    import torch
    from paper_2609_40247_b200 import ta
    P, T, per = 64, 32, 500
    p, t, k = (x.astype(np.int64) for x in np.ogrid[:P, :T, :per])
    ev = np.zeros((P, T, per, 2), dtype=synth.EVENT_DTYPE)
    ev["pid"], ev["stream"] = p[..., None], t[..., None]
    ev["kind"][..., 0], ev["kind"][..., 1] = 2, 3
    ev["ts_start"] = 1_000 + k[..., None] * 1_000 + np.array([0, 400])
    ev["ts_end"] = ev["ts_start"] + 300

    def join(ids):
        ev["corr_id"] = np.broadcast_to(ids, (P, T, per))[..., None]
        flat = np.ascontiguousarray(ev).reshape(-1)
        buf = torch.from_numpy(flat.view(np.uint8)).cuda()
        best = 1e9
        for _ in range(5):
            with ta.Window(buf, [0, len(flat)], [0], [per * 1_000 + 5_000]) as w:
                w.sort_timeline()
                torch.cuda.synchronize()
                at = time.perf_counter()
                j = w.correlate_launches()
                best = min(best, time.perf_counter() - at)
                assert int(j.join_sum["n_matched"][0]) == P * T * per and int(j.join_sum["n_dup_launch"][0]) == 0
        return best

    mixed = join(((t << 40) | (p << 48) | k) * np.int64(-7046029254386353131))
    assert join((t << 40) | k) < 4 * mixed
    assert join((p << 40) | (t << 32) | k) < 4 * mixed


@pytest.mark.parametrize("n", [40, 129, 700])
def test_operators_at_the_first_instant_there_is(n):
    """Records at the smallest time of all, over several tiles: an empty operator there encloses the
    empty records behind it."""
    import torch
    from oracle.ta_oracle import Oracle
    from paper_2609_40247_b200 import ta
    first = -2**63
    ev = np.zeros(n, dtype=synth.EVENT_DTYPE)
    ev["ts_start"] = ev["ts_end"] = first
    ev["kind"] = 1
    ev["kind"][0] = 0
    ev["ts_end"][1], ev["kind"][1] = first + 50, 0
    o = Oracle(ev, [0, n], [first], [first + 1_000])
    o.load(), o.sort(), o.correlate(), o.attribute()
    assert (o.get("parent") >= 0).sum() == n - 1
    buf = torch.from_numpy(ev.view(np.uint8)).cuda()
    with ta.Window(buf, [0, n], [first], [first + 1_000]) as w:
        s = w.sort_timeline()
        w.correlate_launches()
        a = w.attribute_operators()
        assert np.array_equal(s.numpy("perm"), o.get("perm"))
        for k in ("parent", "depth"):
            assert np.array_equal(a.numpy(k), o.get(k)), k


@pytest.mark.parametrize("hashed", [False, True])
def test_join_of_more_records_than_launches_are_counted_on_the_way(hashed):
    """From 24 M records on, launches with a kernel are counted by a pass of their own, which also
    tells whether some have several (graph replays): both ways to address the table."""
    import torch
    from oracle.ta_oracle import Oracle
    from paper_2609_40247_b200 import ta
    from runners import ATTR_KEYS, JOIN_KEYS, ROLLUP_KEYS, assert_same
    wl = synth.make_workload("c3", 0.39, truth=False)
    ev = wl.events
    assert len(ev) > 24 << 20
    kernels = np.nonzero(ev["kind"] == 3)[0]
    again = kernels[5::97]  # the kernel of the record two kernels before in the list gets a second one
    same = ev["pid"][again] == ev["pid"][kernels[3::97][:len(again)]]
    ev["corr_id"][again[same]] = ev["corr_id"][kernels[3::97][:len(again)][same]]
    if hashed:
        joins = ev["kind"] != 5
        with np.errstate(over="ignore"):
            ev["corr_id"][joins] *= np.int64(-7046029254386353131)
    o = Oracle(ev, wl.win_off, wl.win_t0, wl.win_t1)
    o.load()
    o.sort()
    o.correlate()
    assert o.attribute() == 0
    o.rollup()
    want = {k: o.get(k) for k in JOIN_KEYS + ATTR_KEYS + ROLLUP_KEYS}
    assert int(want["kernels_of_launch"].max()) > 1 and int(want["join_sum"]["n_orphan_launch"].sum()) > 0
    buf = torch.from_numpy(np.ascontiguousarray(ev).view(np.uint8).reshape(-1)).cuda()
    with ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1) as w:
        w.sort_timeline()
        j, a = w.correlate_launches(), w.attribute_operators()
        r = w.rollup_operators()
        got = {k: res.numpy(k) for res, names in ((j, JOIN_KEYS), (a, ATTR_KEYS), (r, ROLLUP_KEYS)) for k in names}
    assert_same(want, got)
