"""The large bit-row teams by vertex dictionary, column chunks and place of the column lists, on
owners that the choice by ratio sends there: bit-exact, and by the kernels that ran."""
import itertools

import numpy as np
import pytest

from conftest import csr_of
from test_gpu_bit_rows import random_edges
from test_gpu_close_routes import closed_by
from test_gpu_parity import check_against_oracle, gpu_count

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 40_000, 262_000])
def test_more_than_32_vertices(hglib, shift):
    # |e_u| of two mask words, nearly all meet: the direct map (|V| up to 32,768) and the bit
    # maps with columns in scratch (up to 262,144)
    edges = random_edges(60, 420, 33, 36, 21)
    e_ptr, e_idx = csr_of([[v + shift for v in e] for e in edges])
    check_against_oracle(hglib, 60 + shift, e_ptr, e_idx)
    _, kernels = closed_by(hglib, 60 + shift, e_ptr, e_idx)
    assert "close_bits_large" in kernels and "close_wide" not in kernels


def test_dictionaries_agree(hglib):
    # 2,400 sets of 4 or 5 out of 14 vertices: out-degrees up to about 1,900, the ratio far above
    # 80; the same hypergraph with the direct map, the bit maps and the hash
    sets = [c for k in (4, 5) for c in itertools.combinations(range(14), k)]
    pick = np.random.default_rng(6).permutation(len(sets))[:2400]
    edges = [list(sets[k]) for k in sorted(pick)]
    e_ptr, e_idx = csr_of(edges)
    wide, ws = gpu_count(hglib, 14, e_ptr, e_idx, close_mode=1)
    for shift in (0, 40_000, 300_000):
        counts, st = gpu_count(hglib, 14 + shift, e_ptr, e_idx + shift)
        assert counts.tolist() == wide.tolist() and st["masks"] == ws["masks"], shift
        _, kernels = closed_by(hglib, 14 + shift, e_ptr, e_idx + shift)
        assert "close_bits_large" in kernels and not kernels & {"close_wide", "close_block4096"}


def test_columns_in_chunks(hglib):
    # 400 hyperedges of vertex 0 and 45 of 4,500 others: about 4,000 shared vertices for 13 words
    # of out-neighbours, which shared memory does not hold at once
    rng = np.random.default_rng(8)
    edges = [[0, *(1 + np.sort(rng.choice(4500, 45, replace=False))).tolist()] for _ in range(400)]
    e_ptr, e_idx = csr_of(edges)
    shared = int((np.bincount(e_idx) >= 2).sum())
    assert 4 * shared * 13 > 230_400 - 2 * 48 * 399
    check_against_oracle(hglib, 4501, e_ptr, e_idx)
    _, kernels = closed_by(hglib, 4501, e_ptr, e_idx)
    assert "close_bits_large" in kernels and "close_wide" not in kernels


def test_column_lists_in_scratch(hglib):
    # 1,300 hyperedges of 90-110 out of 3,000 vertices: the lists of the largest owners (130,000
    # entries of two bytes) are larger than shared memory
    edges = random_edges(3000, 1300, 90, 110, 9)
    e_ptr, e_idx = csr_of(edges)
    assert 2 * len(e_idx) > 232_448
    counts, st = gpu_count(hglib, 3000, e_ptr, e_idx)
    wide, ws = gpu_count(hglib, 3000, e_ptr, e_idx, close_mode=1)
    assert counts.tolist() == wide.tolist() and st["masks"] == ws["masks"]
    _, kernels = closed_by(hglib, 3000, e_ptr, e_idx)
    assert "close_bits_large" in kernels
