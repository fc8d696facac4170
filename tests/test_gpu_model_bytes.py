"""The device memory that the batching form's admission counts for a run holds
the run: compared with the memory pool's high-water mark of the run itself, for
graphs whose largest part is the vertices', the edges', the dense counts' and
the hubs' tables.  (It can be well above: a run need not pass through the
largest dense block count that it might.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2305_18663_gb300 as P  # noqa: E402
from test_gpu_graph import _pool_high  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,hub,dense_max_B", [
    (200_000, 50_000, 0, 64),       # vertices
    (200_000, 200_000, 0, 1024),
    (2_000, 2_000_000, 0, 64),      # edges
    (20_000, 400_000, 0, 4096),     # dense counts
    (3_000, 30_000, 0, 4096),       # ... at every block count
    (60_000, 60_000, 40_000, 256),  # a hub's tables in global memory
])
def test_admission_counts_what_a_run_takes(n, m, hub, dense_max_B):
    rng = np.random.default_rng(n + m)
    src, dst = rng.integers(0, n, m), rng.integers(0, n, m)
    if hub:
        src, dst = np.concatenate([src, np.zeros(hub, np.int64)]), np.concatenate([dst, rng.permutation(n)[:hub]])
    pg = P.Graph(n, src.astype(np.int32), dst.astype(np.int32))
    prm = P.Params.default(seed=1, dense_max_B=dense_max_B, max_sweeps=3, merge_proposals=2)
    count = P.sbp_model_bytes(pg.h, dense_max_B)
    high = _pool_high(lambda: pg.partition(prm))
    assert 0 < high <= count, (high, count)
