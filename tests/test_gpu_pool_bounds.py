"""What the library's pool keeps: never more than 1/64 of the device's memory,
also after a lattice of nearly twice that; and a lattice that fits in what is
kept takes no memory from the device."""
import pytest
import torch

from paper_1111_1129_gb300 import SparseLattice, build, capi, inputs

pytestmark = pytest.mark.gpu

SLACK = 64 << 20   # the driver's own granularity


@pytest.fixture(autouse=True)
def _empty_pool():
    build.build()
    capi.load()
    capi.lbm_set_allocator(None, None)
    yield
    capi.lbm_set_allocator(None, None)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_a_large_lattice_gives_back_what_exceeds_the_bound():
    flags = torch.zeros((256, 256, 1024), dtype=torch.uint8, device="cuda")
    bound = torch.cuda.mem_get_info()[1] // 64
    before = _free()
    lat = SparseLattice(flags, "lex", periodic=7)
    capi.lbm_sparse_info(lat.handle)   # the public links too
    assert before - _free() > 1.5 * bound
    lat.close()
    assert 0 < before - _free() <= bound + SLACK


def test_the_next_lattice_takes_the_same_memory():
    bed = inputs.bed_medium(0)
    flags = torch.from_numpy(bed.flags).cuda()
    before = _free()
    SparseLattice(flags, "hilbert", periodic=bed.periodic).close()
    kept = before - _free()
    assert kept >= 38 * bed.n_fluid   # its links at least
    lat = SparseLattice(flags, "hilbert", periodic=bed.periodic)
    assert before - _free() <= kept
    lat.close()
    assert before - _free() <= kept
