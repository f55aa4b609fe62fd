"""The library's own memory for lattices: reused between lattices, bounded, and
given back by lbm_set_allocator (None, None)."""
import threading

import pytest
import torch

from paper_1111_1129_gb300 import SparseLattice, build, capi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    capi.load()


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_idle_memory_is_bounded_and_given_back():
    bed = inputs.bed_medium(0)
    flags = torch.from_numpy(bed.flags).cuda()
    capi.lbm_set_allocator(None, None)
    before = _free()
    for _ in range(3):
        lat = SparseLattice(flags, "hilbert", periodic=bed.periodic)
        capi.lbm_sparse_info(lat.handle)   # the public links too
        lat.close()
    kept = before - _free()
    assert 0 <= kept <= torch.cuda.mem_get_info()[1] // 64 + (64 << 20)
    capi.lbm_set_allocator(None, None)
    assert before - _free() <= 64 << 20


def test_threads_and_streams_share_it():
    """Four threads, each on its own stream, build and release lattices; every
    one must come out as the first did."""
    bed = inputs.bed_small(1)
    flags = torch.from_numpy(bed.flags).cuda()
    ref = SparseLattice(flags, "morton1", periodic=bed.periodic)
    want = ref.cells(), ref.adjacency(), ref.inverse()
    torch.cuda.synchronize()
    bad = []

    def work():
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for _ in range(20):
                lat = SparseLattice(flags, "morton1", periodic=bed.periodic)
                got = lat.cells(), lat.adjacency(), lat.inverse()
                stream.synchronize()
                bad.extend(k for k in range(3) if not torch.equal(got[k], want[k]))
                lat.close()

    threads = [threading.Thread(target=work) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    ref.close()
