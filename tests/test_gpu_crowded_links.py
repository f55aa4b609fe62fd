"""Large lists that keep 32-bit links: a tile of 64 cells meets more pages of
the list than a short link can name.

Membranes one cell thick, across z, with one open cell in each row: in
lexicographic order a run of 64 such cells has neighbours all over the layers
below and above.  The public adjacency must equal the oracle's, steps match
the oracle in the FP64 forms and not depend on how calls are split in any
form, and the gradients match the oracle's adjoint: 1e-10 in FP64; in FP16,
whose 11 significant bits of f - w are rounded once a step, 5e-3 for dJ/dalpha,
which is proportional to the kept velocities.  In 16-bit storage a step moves
148 bytes a cell against 224 in FP32: on a bed of 16 million cells it must be
at least 1.38 times as fast (1.46 measured; 1.31 with one cell a thread)."""
import numpy as np
import pytest
import torch

import fp64_measures
import oracle
from paper_1111_1129_gb300 import Adjoint, LBMState, SparseLattice, build, capi, omega_minus

pytestmark = pytest.mark.gpu

WP = 1.3
WM = omega_minus(WP)
F = (1e-5, -2e-5, 3e-5)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    capi.load()


def _most_pages(adj, n):
    """The most pages of 2048 cells that the links of one tile name."""
    tiles = -(-n // 64)
    page = np.full((18, 64 * tiles), -1)
    page[:, :n] = np.where(adj // n == np.arange(1, 19)[:, None], adj % n // 2048, -1)
    page = np.sort(page.reshape(18, tiles, 64).transpose(1, 0, 2).reshape(tiles, -1), axis=1)
    return int(((page[:, 1:] != page[:, :-1]) & (page[:, 1:] >= 0)).sum(1).max()) + 1


def _norm_rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


@pytest.mark.parametrize("shape,ordering,kind,block,periodic",
                         [((3, 100, 2048), "lex", oracle.ORDER_LEX, (1, 1, 1), 0b001),
                          ((3, 101, 2047), "blocked", oracle.ORDER_BLOCKED, (4096, 4096, 1), 0b110)])
def test_membrane(shape, ordering, kind, block, periodic):
    flags = np.zeros(shape, np.uint8)
    flags[1] = 1
    flags[1, :, 5] = 0
    lat = SparseLattice(torch.from_numpy(flags).cuda(), ordering, block, periodic)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cells, _, adj = oracle.build_sparse(flags, kind, block=block, periodic=periodic)
    assert lat.n > 2 * 4 * 256 * sms and _most_pages(adj, lat.n) > 30
    np.testing.assert_array_equal(lat.cells().cpu().numpy(), cells)
    np.testing.assert_array_equal(lat.adjacency().cpu().numpy(), adj)
    rng = np.random.default_rng(7)
    f0 = oracle.rest_state(flags) * (1 + 1e-3 * rng.standard_normal((19,) + shape))
    start = torch.from_numpy(oracle.to_sparse(f0, cells).copy())
    alpha = rng.uniform(0.0, 0.05, shape)
    field = torch.from_numpy(alpha.ravel()[cells].copy())
    for damped in (False, True):
        f_ref, _, _, u_ref = oracle.run(flags, periodic, WP, WM, F, 4,
                                        alpha=alpha if damped else None, f=f0)
        for form in ("f64", "f64x", "f32", "f32s", "f16s", "bf16s"):
            got = []
            for calls in ([4], [1] * 4):
                st = LBMState(lat, form, 20 if form in ("f16s", "bf16s") else 0)
                if damped:
                    st.set_damping(field)
                st.set_pdfs(start)
                for k in calls:
                    st.step(k, WP, WM, F)
                got.append((st.get_raw(), st.reduce_flux(1), st.moments()))
                if form in ("f64", "f64x"):
                    fp64_measures.check(st.get_pdfs().cpu().numpy(),
                                        oracle.to_sparse(f_ref, cells), 4,
                                        got[-1][2][1].cpu().numpy(),
                                        oracle.to_sparse(u_ref, cells),
                                        label=f"crowded links {ordering} {form} {damped}")
                st.close()
            assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
            assert all(torch.equal(a, b) for a, b in zip(got[0][2], got[1][2]))
    J_ref, dF_ref, da_ref, _ = oracle.adjoint(flags, periodic, WP, WM, F, 3, 1, alpha=alpha, f0=f0)
    for form, tol in (("f64", 1e-10), ("f64x", 1e-10), ("f16s", 5e-3)):
        st = LBMState(lat, form, 20 if form == "f16s" else 0)
        st.set_damping(field)
        st.set_pdfs(start)
        adjoint = Adjoint(st, 3)
        adjoint.forward(WP, WM, F, 1)
        dF, da, _ = adjoint.backward()
        assert _norm_rel(da.cpu().numpy(), oracle.to_sparse(da_ref, cells)) <= tol, form
        assert _norm_rel(dF, dF_ref) <= tol, form
        adjoint.close()
        st.close()
    lat.close()


def test_16_bit_steps_keep_their_lead():
    flags = np.ones((64, 256, 1024), np.uint8)
    flags[1:-1, 1:-1] = 0
    flags[32] = 1
    flags[32, 1:-1, 512] = 0   # a plate with a slit
    lat = SparseLattice(torch.from_numpy(flags).cuda(), "lex", periodic=1)
    rate = {}
    for form in ("f32s", "f16s", "bf16s"):
        st = LBMState(lat, form, 0 if form == "f32s" else 20)
        st.step(20, WP, WM, F)
        rate[form] = 1 / min(st.step_timed(20, WP, WM, F) for _ in range(5))
        st.close()
    lat.close()
    assert min(rate["f16s"], rate["bf16s"]) >= 1.38 * rate["f32s"], rate
