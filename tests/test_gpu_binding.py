"""What the Python binding promises about results: arrays hold what the device holds when they are
asked for."""
import numpy as np
import pytest

from paper_2609_40247_b200 import synth, ta

pytestmark = pytest.mark.gpu


def _window(scale=0.02, name="c1"):
    import torch
    wl = synth.make_workload(name, scale, truth=False)
    buf = torch.from_numpy(np.ascontiguousarray(wl.events).view(np.uint8).reshape(-1)).cuda()
    return wl, buf


@pytest.mark.parametrize("tensor_first", [False, True])
def test_arrays_show_what_was_written_to_a_tensor(tensor_first):
    """Small tables come to the host together; a table the caller writes to is read again."""
    import torch
    wl, buf = _window()
    with ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1) as w:
        s = w.sort_timeline()
        t = s.tensor("lane_pid") if tensor_first else None
        before = s.numpy("lane_window").copy()  # brings the other lane tables along
        if t is None:
            t = s.tensor("lane_pid")
        t.view(torch.int32).fill_(77)
        assert (s.numpy("lane_pid") == 77).all()
        t.view(torch.int32).fill_(78)
        assert (s.numpy("lane_pid") == 78).all()
        assert np.array_equal(s.numpy("lane_window"), before)


def test_no_table_of_a_closed_window():
    wl, buf = _window()
    w = ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1)
    s = w.sort_timeline()
    s.numpy("lane_window")
    w.close()
    for name in ("lane_pid", "lane_off", "lane_window"):
        with pytest.raises(ta.TaError):
            s.numpy(name)


def test_threads_read_results_of_a_window_that_is_being_analysed():
    """Three threads read every table and column of a window's results over and over, as arrays and
    as tensors, while a fourth makes further calls on the window."""
    import threading
    import torch
    from runners import AGG_KEYS, GAP_KEYS, SORT_KEYS
    wl, buf = _window(0.05)
    with ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1) as w:
        s = w.sort_timeline()
        g = w.stream_gaps(500_000)
        k = w.aggregate_ops(ta.DEVICE_KINDS, 0)
        tables = [(s, SORT_KEYS), (g, GAP_KEYS), (k, AGG_KEYS)]
        want = [[r.numpy(n).copy() for n in names] for r, names in tables]
        errors, stop = [], threading.Event()

        def reader(seed):
            try:
                torch.cuda.set_device(buf.device)
                rng = np.random.default_rng(seed)
                for _ in range(60):
                    i = rng.integers(len(tables))
                    r, names = tables[i]
                    for j in rng.permutation(len(names)):
                        if rng.random() < 0.5:
                            got = r.numpy(names[j])
                        else:
                            got = r.tensor(names[j]).cpu().numpy().view(want[i][j].dtype).reshape(want[i][j].shape)
                        assert np.array_equal(got, want[i][j]), names[j]
            except BaseException as e:  # reported in the main thread
                errors.append(e)

        def caller():
            try:
                torch.cuda.set_device(buf.device)
                for _ in range(300):  # (what a call returns stays until the window is closed)
                    if stop.is_set():
                        break
                    again = w.stream_gaps(500_000)
                    assert np.array_equal(again.numpy("lane_gaps"), want[1][GAP_KEYS.index("lane_gaps")])
                    del again
                    assert w.aggregate_ops(ta.DEVICE_KINDS, 0).n_groups == k.n_groups
            except BaseException as e:
                errors.append(e)

        call = threading.Thread(target=caller)
        readers = [threading.Thread(target=reader, args=(q,)) for q in range(3)]
        call.start()
        for t in readers:
            t.start()
        for t in readers:
            t.join()
        stop.set()
        call.join()
        if errors:
            raise errors[0]


@pytest.mark.parametrize("memory", ["torch", "pieces", "library"])
def test_tensors_of_a_window_opened_in_inference_mode_are_ordinary(memory):
    """They can be written to, and hold the results, outside of that mode and inside."""
    import torch
    wl, buf = _window()
    kw = {"torch": {}, "library": {"use_torch_allocator": False},
          "pieces": {"alloc_fn": lambda n: torch.cuda.caching_allocator_alloc(n, buf.device.index),
                     "release_fn": torch.cuda.caching_allocator_delete}}[memory]
    with torch.inference_mode():
        w = ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1, **kw)
        s = w.sort_timeline()
        k = w.aggregate_ops(0, 0)
        made = [s.tensor("perm"), k.tensor("g_name")]
    with w:
        made += [s.tensor("lane_off"), k.tensor("g_count")]
        assert not any(t.is_inference() for t in made)
        for t in made:
            t.add_(0)
        assert (s.numpy("perm") == made[0].view(torch.int32).cpu().numpy()).all()


def test_no_block_up_front_where_torch_would_fill_it_or_cannot_give_it(monkeypatch):
    """Deterministic mode writes to all fresh memory of a tensor; another allocator may refuse in
    its own words.  The window then takes its memory in pieces."""
    import torch
    wl, buf = _window()

    def lanes():
        with ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1) as w:
            return w._handle.chunk, w.sort_timeline().numpy("lane_off")

    chunk, want = lanes()
    assert chunk
    torch.use_deterministic_algorithms(True)
    try:
        chunk, got = lanes()
    finally:
        torch.use_deterministic_algorithms(False)
    assert not chunk and np.array_equal(got, want)

    def refuse(*args, **kw):
        raise RuntimeError("no")

    monkeypatch.setattr(torch, "empty", refuse)
    chunk, got = lanes()
    assert not chunk and np.array_equal(got, want)


_BLOCKING = """
import ctypes, sys, time
cuda = ctypes.CDLL("libcuda.so.1")
assert cuda.cuInit(0) == 0
assert cuda.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0  # CU_CTX_SCHED_BLOCKING_SYNC
sys.path[:0] = [%r, %r]
import numpy as np, torch
from paper_2609_40247_b200 import synth, ta
wl = synth.make_workload("c1", 0.02, truth=False)
buf = torch.from_numpy(np.ascontiguousarray(wl.events).view(np.uint8).reshape(-1)).cuda()
for _ in range(2):
    with ta.Window(buf, wl.win_off, wl.win_t0, wl.win_t1) as w:
        torch.cuda.synchronize()
        torch.cuda._sleep(1_000_000_000)  # half a second of the stream's time in front of the call
        wall, cpu = time.perf_counter(), time.thread_time()
        s = w.sort_timeline()
        wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
        g = w.stream_gaps(1000)
        l = int(np.nonzero(s.numpy("lane_domain") == 1)[0][0])
        a, b = s.numpy("lane_off")[l:l + 2]
        ts, te = (s.tensor(k).view(torch.int64)[a:b].contiguous() for k in ("ts_start", "ts_end"))
        torch.cuda.synchronize()
        torch.cuda._sleep(1_000_000_000)
        wall2, cpu2 = time.perf_counter(), time.thread_time()
        _, row = ta.lane_gaps_noalloc(ts, te, int(wl.win_t0[0]), int(wl.win_t1[0]))
        wall2, cpu2 = time.perf_counter() - wall2, time.thread_time() - cpu2
        assert row == g.numpy("lane_gaps")[l]
print(wall, cpu, wall2, cpu2)
assert wall > 0.2 and wall2 > 0.2, "nothing was waited for"
assert cpu < 0.25 * wall and cpu2 < 0.25 * wall2, "the host thread was busy while it waited"
"""


def test_calls_block_where_the_device_is_set_to_blocking():
    """A process that has asked the driver for blocking waits keeps its cores while a call waits."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _BLOCKING % (root, os.path.join(root, "tests"))], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
