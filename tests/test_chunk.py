"""ta_chunk_*: pieces of one block of memory, handed out without touching it (no GPU needed)."""
import ctypes

import numpy as np
import pytest

from paper_2609_40247_b200 import ta

_ALLOC, _RELEASE = ta._ALLOC_T, ta._RELEASE_T


class Chunk:
    """A chunk over addresses that are never touched; what does not fit is asked of `outside`."""

    def __init__(self, base, size):
        self.lib = ta.lib()
        self.asked, self.returned = [], []
        self.cb = (_ALLOC(lambda n, ctx: self.asked.append(n) or 0x7000 + 256 * len(self.asked)),
                   _RELEASE(lambda p, ctx: self.returned.append(p)))
        self.ptr = self.lib.ta_chunk_open(base, size, *self.cb, None)
        assert self.ptr

    def alloc(self, n):
        return self.lib.chunk_alloc(n, self.ptr)

    def release(self, p):
        self.lib.chunk_release(p, self.ptr)


@pytest.mark.parametrize("base", [1 << 40, (1 << 40) + 8, (1 << 40) + 255, (1 << 40) + 256 + 16])
@pytest.mark.parametrize("size", [0, 100, 256, 511, 4096, 1 << 20])
def test_pieces_are_aligned_and_inside_the_block(base, size):
    c = Chunk(base, size)
    rng = np.random.default_rng(size)
    live = {}
    for _ in range(2000):
        if live and rng.random() < 0.45:
            p = list(live)[rng.integers(len(live))]
            del live[p]
            c.release(p)
            continue
        n = int(rng.integers(1, 700))
        before = len(c.asked)
        p = c.alloc(n)
        if len(c.asked) > before:  # did not fit
            assert p == 0x7000 + 256 * len(c.asked) and c.asked[-1] == n
            c.release(p)
            assert c.returned[-1] == p
            continue
        assert p % 256 == 0 and base <= p and p + n <= base + size
        assert all(p + n <= q or q + m <= p for q, m in live.items())
        live[p] = n
    for p in live:
        c.release(p)
    room = (size - (-base % 256)) // 256 * 256
    if room > 0:  # all of it is one piece again
        assert c.alloc(room) == base + -base % 256
    c.lib.ta_chunk_close(c.ptr)


_NO_MEMORY = """
import resource, sys
sys.path[:0] = [%r, %r]
from test_chunk import Chunk
c = Chunk(1 << 40, 1 << 40)
for _ in range(1000):  # whatever Python and the loader set up on first use
    c.release(c.alloc(1))
now = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (now + (3 << 20), now + (3 << 20)))
alloc, ptr, i = c.lib.chunk_alloc, c.ptr, 0
while i < 2000000 and not c.asked:
    p = alloc(1, ptr)
    i += 1
assert c.asked == [1] and p == 0x7000 + 256 and i > 1000, (c.asked, i)
print("ok", i)
"""


def test_a_list_that_cannot_grow_is_no_exception():
    """The list of pieces needs host memory; without any more the request goes to the caller."""
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", _NO_MEMORY % (os.path.dirname(here), here)], capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stdout, r.stderr)
