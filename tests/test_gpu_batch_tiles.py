"""A batch's tensor-core tiles (member-local columns, only the tiles inside members) against
the hash path: bit-exact."""
import numpy as np
import pytest

from conftest import csr_of
from test_gpu_batch import run_batch
from test_gpu_bit_rows import random_edges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_wave_edges", [0, 700])
def test_batch_tiles_inside_members(hglib, max_wave_edges):
    # the tile path of a batch (member-local columns, only the tiles inside members) against
    # the hash path: members without a heavy hyperedge, members of one tile, members whose
    # rows begin inside another's tile
    rng = np.random.default_rng(2)
    members = []
    for k, (nv, ne, lo, hi) in enumerate([(30, 90, 2, 6), (200, 400, 1, 9), (12, 20, 1, 3),
                                          (150, 300, 3, 40), (500, 200, 2, 60), (40, 1, 5, 5),
                                          (64, 260, 4, 20)]):
        members.append((nv, *csr_of(random_edges(nv, ne, lo, hi, 10 * k + int(rng.integers(9))))))
    members.insert(2, (4, np.zeros(1, dtype=np.int64), np.zeros(0, dtype=np.int32)))
    want = run_batch(hglib, members, max_wave_edges=max_wave_edges, dense_min_size=-1)
    got = run_batch(hglib, members, max_wave_edges=max_wave_edges, dense_min_size=5,
                    dense_max_count=100_000)
    assert got[0].tolist() == want[0].tolist()
    assert got[6].tolist() == want[6].tolist()
    for k in ("W", "W_c", "connected", "max_deg"):
        assert got[1][k].tolist() == want[1][k].tolist(), k
