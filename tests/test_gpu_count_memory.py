"""Device memory that a count holds at a time, seen through the allocator hooks."""
import pytest

from conftest import csr_of
from test_gpu_bit_rows import random_edges

pytestmark = pytest.mark.gpu


class Counting:
    """Hooks over torch's allocator that keep the bytes of every live block and the peak."""

    def __init__(self, hg):
        import torch

        self.live, self.peak = {}, 0
        self.on_change = None
        self.largest = None   # larger requests get no memory

        def alloc(nbytes, stream, _ctx):
            if self.largest is not None and nbytes > self.largest:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(),
                                                   int(stream or 0))
            self.live[p] = int(nbytes)
            self.peak = max(self.peak, sum(self.live.values()))
            if self.on_change:
                self.on_change(self.live)
            return p

        def free(p, _nbytes, _stream, _ctx):
            self.live.pop(p)
            torch.cuda.caching_allocator_delete(int(p))

        self.hooks = (hg.hg._ALLOC_FN(alloc), hg.hg._FREE_FN(free))
        hg.hg_set_allocator(*self.hooks)


def test_one_scratch_of_the_global_table_teams_at_a_time(hglib):
    # hyperedges of 60-70 vertices (global-table teams) and of 20-32 (handed over to the same
    # teams by close_mode 2): the scratch of the second launch takes the place of the first's
    import torch

    edges = random_edges(400, 150, 60, 70, 1) + random_edges(400, 250, 20, 32, 2)
    e_ptr, e_idx = csr_of(edges)
    count = Counting(hglib)
    try:
        big = []
        g = hglib.hg_load_csr(400, len(e_ptr) - 1, e_ptr, e_idx,
                              stream=torch.cuda.Stream().cuda_stream)
        hglib.hg_build_wedges(g, close_mode=2)
        built = set(count.live)

        def watch(live):
            big.append(sum(1 for p, n in live.items() if p not in built and n > (4 << 20)))

        count.on_change = watch
        two = hglib.hg_count_patterns(g)
        st = hglib.hg_close_stats_get(g)
        count.on_change = None
        hglib.hg_free(g)
        assert not count.live
    finally:
        hglib.use_torch_allocator()
    assert st["bucket_teams"][6] > 150   # both kinds were closed by the global-table teams
    assert max(big) == 1, big
    g = hglib.hg_load_csr(400, len(e_ptr) - 1, e_ptr, e_idx)
    hglib.hg_build_wedges(g)
    assert hglib.hg_count_patterns(g).tolist() == two.tolist()
    hglib.hg_free(g)


@pytest.mark.parametrize("shape", ["long", "coauthor", "tag"])
def test_server_admits_by_what_an_evaluation_takes(hglib, shape):
    # the bytes that the server books for a query against the peak of the same calls on a handle
    # of the same hypergraph (the long shape has the 8-byte row layout)
    from dataclasses import replace

    import hgen
    import torch

    spec = {"long": replace(hgen.TAG_HEAVY, num_edges=12_000, num_vertices=20_000, size_p1=2.5,
                            size_hi=600, degree_cap=100),
            "coauthor": replace(hgen.COAUTHOR, num_edges=31_000, num_vertices=6_200),
            "tag": replace(hgen.TAG_HEAVY, num_edges=5_000)}[shape]
    e_ptr, e_idx = hgen.generate(spec)
    nv, ne = spec.num_vertices, len(e_ptr) - 1
    booked, peak = [], []
    for kind in (hglib.HG_Q_COUNTS, hglib.HG_Q_ESTIMATE):
        srv = hglib.Server(workers=1)
        try:
            gid = srv.add_graph(nv, e_ptr, e_idx)
            assert srv.wait(srv.submit(kind, gid, seed=1, num_samples=1000))["status"] == 0
            booked.append(srv.stats()["max_in_flight_bytes"])
        finally:
            srv.close()
        count = Counting(hglib)
        try:
            g = hglib.hg_load_csr(nv, ne, e_ptr, e_idx, stream=torch.cuda.Stream().cuda_stream)
            hglib.hg_build_wedges(g)
            if kind == hglib.HG_Q_COUNTS:
                hglib.hg_count_patterns(g)
            else:
                hglib.hg_sample_estimate(g, 1, 0, 1000)
            hglib.hg_free(g)
        finally:
            hglib.use_torch_allocator()
        peak.append(count.peak)
    assert all(b >= p for b, p in zip(booked, peak)), (booked, peak)
    assert booked[0] < 4 * peak[0] + (64 << 20)   # not so much that it admits nothing


def test_bit_rows_on_fewer_blocks_when_memory_is_short(hglib):
    # column lists of 130,000 entries per block: no room for a slice of scratch on every SM
    import torch

    edges = random_edges(3000, 1300, 90, 110, 9)
    e_ptr, e_idx = csr_of(edges)
    count = Counting(hglib)
    try:
        g = hglib.hg_load_csr(3000, len(e_ptr) - 1, e_ptr, e_idx,
                              stream=torch.cuda.Stream().cuda_stream)
        hglib.hg_build_wedges(g)
        want = hglib.hg_count_patterns(g)
        assert max(count.live.values()) > (12 << 20)   # a slice for each of up to 152 blocks
        count.largest = 3 << 20
        got = hglib.hg_count_patterns(g)
        hglib.hg_free(g)
    finally:
        hglib.use_torch_allocator()
    assert got.tolist() == want.tolist()
