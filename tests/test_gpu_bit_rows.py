"""The closure by bit rows (k_bits.cu) at the sizes where it can go wrong, against the oracle
and the list walk: bit-exact."""
import itertools

import numpy as np
import pytest

from conftest import csr_of
from test_gpu_parity import check_against_oracle, gpu_count

pytestmark = pytest.mark.gpu


def random_edges(nv, ne, lo, hi, seed):
    rng = np.random.default_rng(seed)
    out = set()
    while len(out) < ne:
        out.add(tuple(sorted(rng.choice(nv, int(rng.integers(lo, hi + 1)), replace=False).tolist())))
    return [list(e) for e in sorted(out)]


@pytest.mark.parametrize("ne", [620, 900])
def test_dense_small_teams(hglib, ne):
    # few vertices, so that most hyperedges meet: out-degrees from 2 to several hundred, all
    # in shared-memory teams of every size (the walk's ratio is above its line)
    e_ptr, e_idx = csr_of(random_edges(24, ne, 2, 5, ne))
    check_against_oracle(hglib, 24, e_ptr, e_idx)


@pytest.mark.parametrize("shift", [0, 40_000, 262_084, 300_000])
def test_large_teams_direct_and_hash_dictionary(hglib, shift):
    # out-degrees up to 329 over hyperedges of 24-32 vertices: column lists beyond the
    # shared-memory teams, and more distinct row masks than the mask table holds; ids beyond
    # the direct map's range send the same teams through the maps with columns in scratch (up to
    # 262,144 vertices) and the hash dictionary
    edges = random_edges(60, 330, 24, 32, 3)
    e_ptr, e_idx = csr_of([[v + shift for v in e] for e in edges])
    counts, st = check_against_oracle(hglib, 60 + shift, e_ptr, e_idx)
    assert st["close"]["bucket_teams"][3] > 0 and st["close"]["bucket_teams"][6] == 0


def test_large_teams_few_masks(hglib):
    # lists of the same length whose hyperedges meet an owner in few ways (a common vertex,
    # a subset of four others, rarely one more): the mask table's path
    rng = np.random.default_rng(9)
    edges = {tuple([0] + [1 + k for k in range(4) if rng.random() < 0.5] +
                   (5 + np.sort(rng.choice(3000, 26, replace=False))).tolist())
             for _ in range(340)}
    e_ptr, e_idx = csr_of([list(e) for e in sorted(edges)])
    check_against_oracle(hglib, 3005, e_ptr, e_idx)


def test_shared_counts_beyond_eight_digits(hglib):
    # hyperedges of 300-450 vertices over 600: any two share more than 255 vertices outside a
    # third, and |e_u| is beyond one mask word
    edges = random_edges(600, 40, 300, 450, 5)
    edges += [[600 + k, k] for k in range(3)]   # low-ranked owners of small size
    e_ptr, e_idx = csr_of(edges)
    check_against_oracle(hglib, 603, e_ptr, e_idx)


@pytest.mark.parametrize("sizes", [(1, 9), (1, 4)])
def test_inclusion_patterns(hglib, sizes):
    # every subset (of these sizes) of nine vertices: all patterns with inclusions, many of
    # each; out-degrees above 64 closed by bit rows
    edges = [list(c) for n in range(sizes[0], sizes[1] + 1)
             for c in itertools.combinations(range(9), n)]
    e_ptr, e_idx = csr_of(edges)
    ref, _ = check_against_oracle(hglib, 9, e_ptr, e_idx)
    counts, st = gpu_count(hglib, 9, e_ptr, e_idx, warp_team_max=64)
    assert counts.tolist() == ref.tolist()
    assert st["close"]["bucket_teams"][1] == st["close"]["bucket_teams"][2] == 0
    assert all(int(c) > 0 for c in ref[1:9])
    # the work counters do not depend on the path
    _, walked = gpu_count(hglib, 9, e_ptr, e_idx, close_mode=1)
    for k in ("probes", "gathers", "out_entries"):
        assert st["close"][k] == walked["close"][k], k
