"""Owners that bit rows cannot hold go to the walking team of their shape: the counts and who
closes them, against the oracle or the global-table teams.  Integers: bit-exact."""
import numpy as np
import pytest

from conftest import csr_of
from test_gpu_bit_rows import random_edges
from test_gpu_parity import check_against_oracle, gpu_count

pytestmark = pytest.mark.gpu


def star(nv, ne, size, seed, first):
    """ne hyperedges of vertex `first` and size - 1 others of the next nv."""
    rng = np.random.default_rng(seed)
    rows = np.sort(rng.integers(1, nv, (ne, size - 1)), axis=1) + first
    return csr_of([[first, *r.tolist()] for r in rows])


@pytest.mark.parametrize("ne", [420, 2001])
def test_full_hash_returns_owners_to_the_block_teams(hglib, ne):
    # ids beyond the bit maps' 262,144 vertices; 2,001 hyperedges of 20 vertices out of 30,000:
    # the largest owners have more distinct vertices than the hash has slots, the smallest
    # have few and stay; 420 (within the oracle's time) fill half of it
    first, nv = 300_000, 30_000
    e_ptr, e_idx = star(nv, ne, 20, ne, first)
    counts, st = gpu_count(hglib, first + nv, e_ptr, e_idx)
    assert int(counts[0]) == ne * (ne - 1) * (ne - 2) // 6   # all share the first vertex
    assert st["close"]["bucket_teams"][6] == 0   # none left to the global-table blocks
    if ne == 420:
        check_against_oracle(hglib, first + nv, e_ptr, e_idx)
    wide, ws = gpu_count(hglib, first + nv, e_ptr, e_idx, close_mode=1)
    assert counts.tolist() == wide.tolist() and st["masks"] == ws["masks"]
    for k in ("probes", "gathers", "out_entries"):
        assert st["close"][k] == ws["close"][k], k


def test_out_degrees_beyond_the_bit_rows(hglib):
    # 4,400 of the hyperedges of 30-32 out of 60 vertices beside 262,000 unused ones: nearly
    # all meet, and owners of out-degree 4,000 and more do not fit a bit-row team
    edges = random_edges(60, 4400, 30, 32, 8)
    e_ptr, e_idx = csr_of([[v + 262_000 for v in e] for e in edges])
    counts, st = gpu_count(hglib, 262_060, e_ptr, e_idx)
    wide, ws = gpu_count(hglib, 262_060, e_ptr, e_idx, close_mode=1)
    assert counts.tolist() == wide.tolist() and st["masks"] == ws["masks"]
    assert st["max_out_deg"] > 4000 and st["close"]["bucket_teams"][6] == 0
    for k in ("probes", "gathers", "out_entries"):
        assert st["close"][k] == ws["close"][k], k
