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
