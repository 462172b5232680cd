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


def closed_by(hg, nv, e_ptr, e_idx):
    """(counts, masks, names of the closure kernels that ran)"""
    import torch

    g = hg.hg_load_csr(nv, len(e_ptr) - 1, e_ptr, e_idx, stream=torch.cuda.Stream().cuda_stream)
    try:
        hg.hg_set_timing(g, True)
        hg.hg_build_wedges(g)
        counts = hg.hg_count_patterns(g)
        return counts, {k for k in hg.hg_kernel_times(g) if k.startswith("close_")}
    finally:
        hg.hg_free(g)


@pytest.mark.parametrize("nv,ne,lo,hi,shift,bits", [
    (3000, 120, 400, 800, 0, False),      # |e_u| of hundreds over few others: walked
    (300, 420, 33, 38, 50_000, True),     # beyond the direct map: bit rows all the same
    (300, 420, 33, 38, 300_000, False),   # the hash dictionary is for dense ones alone
])
def test_owners_of_more_than_32_vertices(hglib, nv, ne, lo, hi, shift, bits):
    edges = random_edges(nv, ne, lo, hi, ne)
    e_ptr, e_idx = csr_of([[v + shift for v in e] for e in edges])
    check_against_oracle(hglib, nv + shift, e_ptr, e_idx)
    _, kernels = closed_by(hglib, nv + shift, e_ptr, e_idx)
    assert kernels >= ({"close_bits_large"} if bits else {"close_wide"})
    if not bits:
        assert "close_bits_large" not in kernels


def test_sparse_owners_with_long_neighbours_go_to_the_block_teams(hglib):
    # 300 small hyperedges and 60 of 300-500 vertices meet in vertex 0: the small ones rank
    # lowest, have out-degrees above 256, and their neighbours' vertices are many and private
    rng = np.random.default_rng(4)
    edges = {(0, 1 + k, 301 + k) for k in range(300)}
    edges |= {tuple([0] + (1000 + np.sort(rng.choice(40_000, int(n), replace=False))).tolist())
              for n in rng.integers(300, 500, 60)}
    e_ptr, e_idx = csr_of([list(e) for e in sorted(edges)])
    check_against_oracle(hglib, 41_000, e_ptr, e_idx)
    _, kernels = closed_by(hglib, 41_000, e_ptr, e_idx)
    assert "close_block2048" in kernels


@pytest.mark.parametrize("ne", [1201, 3001])
def test_unpacked_block_teams(hglib, ne):
    # the same star beside one hyperedge of 300 vertices that gives the two-array row layout:
    # block teams of that layout up to out-degree 4,096
    first, nv = 300_000, 40_000
    e_ptr, e_idx = star(nv, ne, 24, ne, first)
    e_ptr = np.concatenate([e_ptr, [e_ptr[-1] + 300]]).astype(np.int64)
    e_idx = np.concatenate([e_idx, np.arange(300, dtype=np.int32)])
    counts, st = gpu_count(hglib, first + nv, e_ptr, e_idx)
    wide, ws = gpu_count(hglib, first + nv, e_ptr, e_idx, close_mode=1)
    assert int(counts[0]) == ne * (ne - 1) * (ne - 2) // 6
    assert counts.tolist() == wide.tolist() and st["masks"] == ws["masks"]
    _, kernels = closed_by(hglib, first + nv, e_ptr, e_idx)
    assert ("close_block8192" if ne > 2048 else "close_block2048") in kernels
