"""The sampler's rows around the sizes where their sort and their staging change, against the
oracle: bit-exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spokes", [500, 520, 1100])
@pytest.mark.parametrize("long_edge", [0, 300])
def test_sampler_rows_around_the_warp_sort(hglib, spokes, long_edge):
    # rows just below and above the 512 entries that one warp sorts, and searched rows beyond
    # the staged 384; a hyperedge of 300 vertices gives the two-array row layout
    import hgen
    import oracle
    import torch

    nv, e_ptr, e_idx = hgen.hub(spokes, 60, 3)
    if long_edge:
        e_ptr = np.concatenate([e_ptr, [e_ptr[-1] + long_edge]]).astype(np.int64)
        e_idx = np.concatenate([e_idx, np.arange(long_edge, dtype=np.int32)])
        nv = max(nv, long_edge)
    g = hglib.hg_load_csr(nv, len(e_ptr) - 1, e_ptr, e_idx,
                          stream=torch.cuda.Stream().cuda_stream)
    try:
        hglib.hg_build_wedges(g)
        raw, est = hglib.hg_sample_estimate(g, 11, 0, 3000)
        raw7, est7, _ = hglib.hg_sample_estimate_adv(g, 11, 0, 3000)
    finally:
        hglib.hg_free(g)
    ref = oracle.sample_estimate(e_ptr, e_idx, nv, seed=11, first=0, num=3000)
    ref7 = oracle.sample_estimate_adv(e_ptr, e_idx, nv, seed=11, first=0, num=3000)
    assert raw.tolist() == ref.raw.tolist() and est.tolist() == ref.est.tolist()
    assert raw7.tolist() == ref7.raw.tolist() and est7.tolist() == ref7.est.tolist()
