"""The cached step graph and a damping field that is removed and set again.

FP64 storage keeps the damping in two allocations, and a step bakes both
addresses in.  An allocator may give one of them its old address back and not
the other; long calls (graph replays) must then still equal short ones
(individual launches) bit for bit.  The allocator here hands out blocks of
buffers it keeps for the whole test."""
import pytest
import torch

from paper_1111_1129_gb300 import LBMState, SparseLattice, build, capi, inputs, omega_minus

pytestmark = pytest.mark.gpu

WP = 1.0 / 0.8
WM = omega_minus(WP)
F = (0.0, 0.0, 1e-5)


class _Blocks:
    """Blocks by size, the one freed last first."""

    def __init__(self):
        self.buffers, self.size, self.idle, self.given = {}, {}, {}, []

    def alloc(self, nbytes, stream):
        idle = self.idle.get(nbytes, [])
        if idle:
            ptr = idle.pop()
        else:
            buf = torch.zeros(max(nbytes, 1), dtype=torch.uint8, device="cuda")
            ptr = buf.data_ptr()
            self.buffers[ptr], self.size[ptr] = buf, nbytes
        self.given.append((nbytes, ptr))
        return ptr

    def release(self, ptr, stream):
        self.idle.setdefault(self.size[ptr], []).append(ptr)


@pytest.mark.parametrize("form", ["f64x", "f64", "f32s"])
def test_damping_set_again_at_other_addresses(form):
    build.build()
    capi.load()
    bed = inputs.bed_small(3)
    flags = torch.from_numpy(bed.flags).cuda()
    blocks = _Blocks()
    capi.lbm_set_allocator(blocks.alloc, blocks.release)
    try:
        lat = SparseLattice(flags, "lex", periodic=bed.periodic)
        g = torch.Generator(device="cuda").manual_seed(1)
        a1, a2 = (0.05 * torch.rand(lat.n, generator=g, dtype=torch.float64, device="cuda")
                  for _ in range(2))
        got = []
        for chunk in (400, 100):   # replays of 128 steps; launches only
            st = LBMState(lat, form)

            def steps():
                for _ in range(400 // chunk):
                    st.step(chunk, WP, WM, F)

            blocks.given.clear()
            st.set_damping(a1)
            first = list(blocks.given)
            steps()
            st.set_damping(None)
            # every block of the field but its first is taken by someone else
            for nbytes, ptr in first[1:]:
                blocks.idle[nbytes].remove(ptr)
            blocks.given.clear()
            st.set_damping(a2)
            assert blocks.given[0] == first[0]
            assert all(p != q for (_, p), (_, q) in zip(blocks.given[1:], first[1:]))
            assert len(first) == (2 if form == "f64x" else 1)
            steps()
            got.append((st.get_raw(), st.reduce_flux(2)))
            st.close()
        lat.close()
        torch.cuda.synchronize()
    finally:
        capi.lbm_set_allocator(None, None)
    assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
