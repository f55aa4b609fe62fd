"""The fixed-point FP64-storage step over the range of relaxation rates.

The even-part factor (1 - w+)/2 is a power of two of either sign, zero, or a
general product, and the odd-part factor runs to the ends of its range; each
takes its own form of the fixed-point products.  A few steps from a random
state in the fast range must match the oracle within the FP64 round-off
bound, and the stored mass must not change, with and without damping."""
import numpy as np
import pytest
import torch

import fp64_measures
import oracle
from paper_1111_1129_gb300 import LBMState, SparseLattice, build, capi, omega_minus

pytestmark = pytest.mark.gpu

WBITS = np.array([0x3FD5555555555555] + [0x3FAC71C71C71C71C] * 6 + [0x3F9C71C71C71C71C] * 12,
                 dtype=np.int64)
SHIFT = np.array([4] + [1] * 6 + [0] * 12, dtype=np.int64)


def _mass(f):
    bits = np.ascontiguousarray(f).view(np.int64)
    assert np.all((bits >> 52) == (WBITS[:, None] >> 52))
    return sum(((bits - WBITS[:, None]) << SHIFT[:, None]).ravel().tolist())


@pytest.mark.parametrize("damped", [False, True])
@pytest.mark.parametrize("wp", [1e-9, 0.5, 0.75, 1.0, 1.25, 1.5, 1.61, 1.99])
def test_rates_against_oracle(wp, damped):
    build.build()
    capi.load()
    rng = np.random.default_rng(int(wp * 1000) + damped)
    shape, steps = (9, 8, 13), 6
    flags = (rng.random(shape) < 0.3).astype(np.uint8)
    f0 = oracle.rest_state(flags) * (1 + 1e-3 * rng.standard_normal((19,) + shape))
    wm, F = omega_minus(wp), 1e-5 * rng.standard_normal(3)
    alpha = rng.uniform(0.0, 0.05, shape) if damped else None
    lat = SparseLattice(torch.from_numpy(flags).cuda(), "lex", periodic=0b101)
    cells = lat.cells().cpu().numpy()
    st = LBMState(lat, "f64x")
    if damped:
        st.set_damping(torch.from_numpy(alpha.ravel()[cells].copy()))
    st.set_pdfs(torch.from_numpy(oracle.to_sparse(f0, cells).copy()))
    before = _mass(st.get_pdfs().cpu().numpy())
    st.step(steps, wp, wm, F)
    got = st.get_pdfs().cpu().numpy()
    assert _mass(got) == before
    kw = {"alpha": alpha} if damped else {}
    f_ref, _, _, u_ref = oracle.run(flags, 0b101, wp, wm, F, steps, f=f0, **kw)
    _, u = st.moments()
    fp64_measures.check(got, oracle.to_sparse(f_ref, cells), steps, u.cpu().numpy(),
                        oracle.to_sparse(u_ref, cells), label=f"f64x w+={wp} damped={damped}")
    st.close()
    lat.close()
