"""Draws whose third hyperedge has a size around the lines between scanning and searching its
vertices, against the oracle: bit-exact."""
import numpy as np
import pytest

from conftest import csr_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [False, True])
def test_third_hyperedge_around_the_scan_lines(hglib, wide):
    # sizes 7-9 and 31-34 over 60 vertices: every hyperedge meets nearly every other one, in
    # one vertex to thirty; a hyperedge of 300 gives the two-array row layout
    import oracle
    import torch

    rng = np.random.default_rng(12)
    edges = {tuple(np.sort(rng.choice(60, int(k), replace=False)).tolist())
             for k in rng.choice([7, 8, 9, 31, 32, 33, 34], 260)}
    nv = 60
    if wide:
        edges.add(tuple(range(50, 350)))
        nv = 350
    e_ptr, e_idx = csr_of([list(e) for e in sorted(edges)])
    g = hglib.hg_load_csr(nv, len(e_ptr) - 1, e_ptr, e_idx,
                          stream=torch.cuda.Stream().cuda_stream)
    try:
        hglib.hg_build_wedges(g)
        raw, est = hglib.hg_sample_estimate(g, 5, 0, 4000)
        raw7, est7, _ = hglib.hg_sample_estimate_adv(g, 5, 0, 4000)
    finally:
        hglib.hg_free(g)
    ref = oracle.sample_estimate(e_ptr, e_idx, nv, seed=5, first=0, num=4000)
    ref7 = oracle.sample_estimate_adv(e_ptr, e_idx, nv, seed=5, first=0, num=4000)
    assert raw.tolist() == ref.raw.tolist() and est.tolist() == ref.est.tolist()
    assert raw7.tolist() == ref7.raw.tolist() and est7.tolist() == ref7.est.tolist()
