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
