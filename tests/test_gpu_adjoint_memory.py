"""The adjoint's memory plan: velocities of the last steps, checkpoints and
recomputed segments before them.

The stride sets how much memory there is, hence how many steps are kept and in
how many segments the others are recomputed; results must not depend on it,
bit for bit, nor on a second reverse pass, nor on the state moving on after
the forward pass.  A list with short links is checked against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1111_1129_gb300 import Adjoint, LBMState, SparseLattice, build, capi, omega_minus

pytestmark = pytest.mark.gpu

WP = 1.0 / 0.8
WM = omega_minus(WP)
F = (1e-5, -2e-5, 1e-4)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    capi.load()


def _random(shape, seed, scale):
    rng = np.random.default_rng(seed)
    flags = (rng.random(shape) < 0.2).astype(np.uint8)
    return flags, 0.05 * rng.random(shape), oracle.rest_state(flags) * (
        1 + scale * rng.standard_normal((19,) + shape))


def _state(lat, precision, f0, alpha):
    cells = lat.cells().cpu().numpy()
    st = LBMState(lat, precision, 18 if precision in ("f16s", "bf16s") else 0)
    st.set_pdfs(torch.from_numpy(oracle.to_sparse(f0, cells).copy()))
    if alpha is not None:
        st.set_damping(torch.from_numpy(alpha.ravel()[cells].copy()))
    return st


@pytest.mark.parametrize("precision", ["f64", "f64x", "f32s", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("K", [1, 2, 3, 40, 301])
def test_strides_and_second_pass_agree(precision, K):
    flags, alpha, f0 = _random((5, 6, 7), K, 1e-3)
    lat = SparseLattice(torch.from_numpy(flags).cuda(), "lex", periodic=0b011)
    ref = None
    for stride in (1, 0, K):
        st = _state(lat, precision, f0, alpha)
        adj = Adjoint(st, K, stride)
        for again in range(2):   # a second forward pass from the same state
            J = adj.forward(WP, WM, F, 2)
            if again:
                st.step(3, WP, WM, F)   # the reverse pass must not need the state's PDFs
            for _ in range(2):
                dF, da, df0 = adj.backward(want_alpha=True, want_f0=True)
                got = (J, dF, da, df0)
                if ref is None:
                    ref = got
                assert got[:2] == ref[:2]
                assert torch.equal(da, ref[2]) and torch.equal(df0, ref[3])
            dF_only, none, _ = adj.backward(want_alpha=False)
            assert none is None and dF_only == ref[1]
        adj.close()
        st.close()
    lat.close()


@pytest.mark.parametrize("damped", [False, True])
@pytest.mark.parametrize("precision", ["f64", "f64x"])
def test_list_with_short_links_matches_oracle(precision, damped):
    flags, alpha, f0 = _random((75, 74, 73), 3, 1e-3)
    lat = SparseLattice(torch.from_numpy(flags).cuda(), "hilbert", periodic=0b101)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert lat.n > 2 * 4 * 256 * sms
    alpha = alpha if damped else None
    J_ref, dF_ref, da_ref, lam_ref = oracle.adjoint(flags, 0b101, WP, WM, np.array(F), 4, 1,
                                                    alpha=alpha, f0=f0)
    st = _state(lat, precision, f0, alpha)
    adj = Adjoint(st, 4)
    J = adj.forward(WP, WM, F, 1)
    dF, da, df0 = adj.backward(want_alpha=True, want_f0=True)
    cells = lat.cells().cpu().numpy()

    def rel(a, b):
        return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))
    assert abs(J - J_ref) <= 1e-10 * abs(J_ref)
    assert rel(dF, dF_ref) < 1e-10
    assert rel(da.cpu().numpy(), da_ref.ravel()[cells]) < 1e-10
    assert rel(df0.cpu().numpy(), oracle.to_sparse(lam_ref, cells)) < 1e-10
    adj.close()
    st.close()
    lat.close()


@pytest.mark.parametrize("damped", [False, True])
@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("precision", ["f32s", "f16s"])
def test_two_cells_a_thread_match_one(precision, odd, damped):
    """Five copies of a periodic box, long enough for short links and the reverse
    step of two cells a thread, against one copy with a cell a thread: the same
    mean velocity, and each cell's gradient a fifth.  The seeds 1/N round
    differently; a value takes ~10 roundings of 2^-24 in each of 4 steps, which
    1e-5 of the norm covers."""
    flags, alpha, f0 = _random((45, 44, 43), 11, 1e-3)
    fluid = np.argwhere(flags == 0)
    if (len(fluid) % 2 == 1) != odd:
        flags[tuple(fluid[777])] = 1
        f0 = f0 * (flags == 0)
    got = []
    for copies in (1, 5):
        tile = lambda a: np.concatenate([a] * copies, axis=-3)
        lat = SparseLattice(torch.from_numpy(tile(flags)).cuda(), "lex", periodic=7)
        st = _state(lat, precision, tile(f0), tile(alpha) if damped else None)
        adj = Adjoint(st, 4)
        J = adj.forward(WP, WM, F, 0)
        dF, da, _ = adj.backward(want_alpha=True)
        got.append((J, np.array(dF), da.cpu().numpy() * copies, lat.n))
        adj.close()
        st.close()
        lat.close()
    (J1, dF1, da1, n1), (J5, dF5, da5, n5) = got
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n1 % 2 == odd and n1 <= 2 * 4 * 256 * sms < n5 == 5 * n1

    def rel(a, b):
        return np.linalg.norm(a - b) / np.linalg.norm(b)
    assert abs(J5 - J1) <= 1e-5 * abs(J1)
    assert rel(dF5, dF1) < 1e-5
    assert rel(da5.reshape(5, n1), da1[None].repeat(5, 0)) < 1e-5
