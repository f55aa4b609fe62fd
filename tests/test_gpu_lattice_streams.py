"""Copies of a lattice's arrays asked for on another stream than its own: a
lattice closed while they are still queued, and another one built in the
memory it gave back, must leave them as they were."""
import pytest
import torch

from paper_1111_1129_gb300 import SparseLattice, build, capi, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bed", ["bed_small", "bed_medium"])
def test_queued_copies_outlive_the_lattice(bed):
    build.build()
    capi.load()
    bed = getattr(inputs, bed)(0)
    flags = torch.from_numpy(bed.flags).cuda()
    other = flags.flip(0, 1, 2).contiguous()   # as many cells in other places
    own, reader = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    lat = SparseLattice(flags, "lex", periodic=bed.periodic, stream=own)
    want = lat.cells(), lat.adjacency(), lat.inverse()
    torch.cuda.synchronize()
    with torch.cuda.stream(reader):
        torch.cuda._sleep(100_000_000)   # ~50 ms of other work before the copies
        got = lat.cells(), lat.adjacency(), lat.inverse()
    lat.close()
    following = SparseLattice(other, "lex", periodic=bed.periodic, stream=own)
    assert following.n == want[0].numel()
    with torch.cuda.stream(own):
        theirs = following.cells(), following.adjacency(), following.inverse()
    torch.cuda.synchronize()
    for a, b, c in zip(want, got, theirs):
        assert torch.equal(a, b) and not torch.equal(a, c)
    following.close()
