"""The integer conversions of set_pdfs / get_pdfs against PyTorch's, bit for bit,
and the fixed-point moments against FP64 sums, cells out of range included."""
import numpy as np
import pytest
import torch

from paper_1111_1129_gb300 import LBMState, SparseLattice, build, capi, inputs, omega_minus

pytestmark = pytest.mark.gpu
W = torch.from_numpy(np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12))[:, None]
# one cell in flight and several per thread; an odd number of cells
BOXES = [(5, 5, 7), (61, 97, 101)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    capi.load()


def _lattice(box):
    return SparseLattice(torch.zeros(box, dtype=torch.uint8, device="cuda"), "lex",
                         periodic=7)


def _same_bits(a, b):
    both_nan = torch.isnan(a) & torch.isnan(b)
    return bool(((a.view(torch.int64) == b.view(torch.int64)) | both_nan).all())


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("form,dtype,bits", [("f32", torch.float32, 32), ("f32s", torch.float32, 32),
                                             ("f16s", torch.float16, 16),
                                             ("bf16s", torch.bfloat16, 16)])
def test_copies_are_exact(box, form, dtype, bits):
    lat = _lattice(box)
    scale = 20 if bits == 16 else 0
    st = LBMState(lat, form, scale)
    shifted = form != "f32"
    rng = np.random.default_rng(lat.n)
    word = {32: np.int32, 16: np.int16}[bits]
    raw = rng.integers(-2 ** (bits - 1), 2 ** (bits - 1), (19, lat.n)).astype(word)
    # zeros, subnormals and infinities among them
    special = {torch.float32: [0, 1, 0x7FFFFF, 0x800000, 0x7F7FFFFF, 0x7F800000],
               torch.float16: [0, 1, 0x3FF, 0x400, 0x7BFF, 0x7C00],
               torch.bfloat16: [0, 1, 0x7F, 0x80, 0x7F7F, 0x7F80]}[dtype]
    for k, v in enumerate(special):
        raw[k, ::2], raw[k + 6, ::3] = v, np.array([v], word) | np.iinfo(word).min
    raw = torch.from_numpy(raw)
    st.set_raw(raw.cuda())
    v = (raw.view(dtype).float() * 2.0 ** -scale).double()
    assert _same_bits(st.get_pdfs().cpu(), W + v if shifted else v)

    # to the storage form: values across the whole range, ties and near ties
    x = rng.standard_normal((19, lat.n)) * 10.0 ** rng.uniform(-47, 39, (19, lat.n))
    b = x.view(np.int64)
    b[:, ::3] = (b[:, ::3] & ~0x1FFFFFFF) | 0x10000000
    b[:, 1::6] |= 0x1FFFFFFF
    x[:, 5::7] = 0.0
    x[:, 6::7] = -0.0
    x[:, 11::13] *= 1e-30
    x[0, :4] = [np.inf, -np.inf, 3.4028235677973366e38, 1.1754943157898258e-38]
    x = torch.from_numpy(x) + (W if shifted else 0.0)
    st.set_pdfs(x.cuda())
    c = (x - W if shifted else x).float()
    want = (c * 2.0 ** scale).to(dtype)
    got = st.get_raw().cpu().view(dtype)
    assert _same_bits(got.double(), want.double())


@pytest.mark.parametrize("damped", [False, True])
@pytest.mark.parametrize("form", ["f64", "f64x"])
@pytest.mark.parametrize("size", ["small", "medium"])   # 32-bit and 16-bit links
def test_moments(size, form, damped):
    bed = inputs.bed_small(0) if size == "small" else inputs.bed_medium(0)
    lat = SparseLattice(torch.from_numpy(bed.flags).cuda(), "lex", periodic=bed.periodic)
    st = LBMState(lat, form)
    g = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)
    w = W.cuda()
    f = w * (1.0 + 1e-3 * (rand(19, lat.n) - 0.5))
    out = torch.randint(0, lat.n, (lat.n // 50,), generator=g, device="cuda")
    f[:, out] *= 0.2 + 3.0 * rand(19, out.numel())   # beyond a binary range
    f[3, out[:50]] = -0.1
    force = (1e-4, -2e-4, 3e-5)
    st.set_pdfs(f)
    alpha = 0.8 * rand(lat.n) if damped else None
    if damped:
        st.set_damping(alpha)
    st.step(1, 1.25, omega_minus(1.25), force)
    rho, u = st.moments()
    pulled = f.clone()
    pulled[1:] = f.reshape(-1)[lat.adjacency().long()]
    c = torch.tensor(_velocities(), dtype=torch.float64, device="cuda")
    want_rho = pulled.sum(0)
    want_u = c.T @ pulled + 0.5 * torch.tensor(force, dtype=torch.float64, device="cuda")[:, None]
    if damped:
        want_u = want_u / (1.0 + 0.5 * alpha)
    # either side rounds at most 20 sums of magnitude below sum |f|
    tol = 2 * 20 * 2.0 ** -53 * pulled.abs().sum(0)
    assert bool(((rho - want_rho).abs() <= tol).all())
    assert bool(((u - want_u).abs() <= tol).all())


def _velocities():
    c = [(0, 0, 0)]
    for a in [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1),
              (0, 1, 1), (0, 1, -1)]:
        c += [a, tuple(-x for x in a)]
    return c
