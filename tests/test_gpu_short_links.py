"""Short links: lists of more than two waves keep each link in 16 bits.

The lists here are just above two waves of the device (of 4 blocks of 256
threads per SM), one just below, with every kind of end: a multiple of 64
cells, one more, one less, odd and even.  The public adjacency, decoded from the short
links, must equal the oracle's bit for bit.  Steps through them must match the
oracle in the FP64 forms, and in every form one call (pair sweeps, then the
reducing step) must equal single steps (the reducing step alone) bit for bit.
"""
import numpy as np
import pytest
import torch

import fp64_measures
import oracle
from paper_1111_1129_gb300 import LBMState, SparseLattice, build, capi, omega_minus

pytestmark = pytest.mark.gpu

WP = 1.3
F = (1e-5, -2e-5, 3e-5)
ORDERS = {"lex": oracle.ORDER_LEX, "blocked": oracle.ORDER_BLOCKED,
          "morton2": oracle.ORDER_MORTON2, "hilbert": oracle.ORDER_HILBERT}


def _flags(shape, rest, seed):
    """A box of mostly fluid cells whose number is `rest` modulo 64."""
    rng = np.random.default_rng(seed)
    flags = (rng.random(shape) < 0.05).astype(np.uint8)
    fluid = np.flatnonzero(flags.ravel() == 0)
    flags.ravel()[rng.choice(fluid, (len(fluid) - rest) % 64, replace=False)] = 1
    return flags


@pytest.mark.parametrize("shape,rest,ordering,periodic",
                         [((70, 70, 70), 0, "lex", 0b100), ((70, 71, 70), 1, "blocked", 0b111),
                          ((40, 90, 95), 63, "hilbert", 0b010), ((130, 9, 300), 2, "morton2", 0b001),
                          ((70, 74, 72), 33, "lex", 0b101), ((71, 70, 73), 62, "hilbert", 0b000),
                          ((68, 69, 69), 5, "lex", 0b110)])
def test_links_and_steps(shape, rest, ordering, periodic):
    build.build()
    capi.load()
    flags = _flags(shape, rest, sum(shape))
    lat = SparseLattice(torch.from_numpy(flags).cuda(), ordering, (8, 8, 8), periodic)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (lat.n > 2 * 4 * 256 * sms) == (shape != (68, 69, 69)) and lat.n % 64 == rest
    cells, _, adj = oracle.build_sparse(flags, ORDERS[ordering], block=(8, 8, 8),
                                        periodic=periodic)
    np.testing.assert_array_equal(lat.cells().cpu().numpy(), cells)
    np.testing.assert_array_equal(lat.adjacency().cpu().numpy(), adj)
    rng = np.random.default_rng(5)
    f0 = oracle.rest_state(flags) * (1 + 1e-3 * rng.standard_normal((19,) + shape))
    start = torch.from_numpy(oracle.to_sparse(f0, cells).copy())
    alpha = rng.uniform(0.0, 0.05, shape)
    wm = omega_minus(WP)
    for damped in (False, True):
        f_ref, _, _, u_ref = oracle.run(flags, periodic, WP, wm, F, 4,
                                        alpha=alpha if damped else None, f=f0)
        for form in ("f64", "f64x", "f32", "f32s", "f16s", "bf16s"):
            got = []
            for calls in ([4], [1] * 4):
                st = LBMState(lat, form, 20 if form in ("f16s", "bf16s") else 0)
                if damped:
                    st.set_damping(torch.from_numpy(alpha.ravel()[cells].copy()))
                st.set_pdfs(start)
                for k in calls:
                    st.step(k, WP, wm, F)
                got.append((st.get_raw(), st.reduce_flux(1), st.moments()))
                if form in ("f64", "f64x"):
                    fp64_measures.check(st.get_pdfs().cpu().numpy(),
                                        oracle.to_sparse(f_ref, cells), 4,
                                        got[-1][2][1].cpu().numpy(),
                                        oracle.to_sparse(u_ref, cells),
                                        label=f"short links {ordering} {form} {damped}")
                st.close()
            assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
            assert all(torch.equal(a, b) for a, b in zip(got[0][2], got[1][2]))
    lat.close()
