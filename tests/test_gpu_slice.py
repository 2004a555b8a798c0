"""The sliced FP64 product (exact digit products on the tensor cores) against extended precision."""
import numpy as np
import pytest

from paper_2308_09782_gb300 import vgtb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    vgtb.load()


def _matrix(rng, m, k, kind):
    x = rng.normal(size=(m, k)) + 1j * rng.normal(size=(m, k))
    if kind == "decay":      # S^-1, D and H fall off away from the diagonal
        x *= np.exp(-0.3 * np.abs(np.arange(m)[:, None] - np.arange(k)[None]))
    elif kind == "coherent":  # every digit product at its largest: the exactness bound of a run is met
        x = np.full((m, k), (1.0 - 2.0 ** -20) * (1 + 1j))
    elif kind == "rows":     # row scales over the exponent range
        x *= 10.0 ** rng.uniform(-150, 150, size=(m, 1))
    return x


# tile edges: one row, partial and whole 64-wide k-panels, 128-column and 256-row tiles, runs of 512 k
SHAPES = [(1, 1, 1), (5, 7, 3), (33, 64, 65), (128, 128, 128), (257, 129, 513), (300, 260, 600)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["random", "decay", "coherent", "rows"])
def test_slice_product_is_as_exact_as_fp64(shape, kind):
    """Operands are held to 2^-55 of their row's largest part, so each of the 2 k real products of a
    part is off by at most 2 x 2^-55 of the row maxima (the pairs left out are far below), and the
    result is rounded once: |error| <= 2^-52 |c| + 2 k 2^-54 max|a_row| max|r_row|."""
    m, n, k = shape
    rng = np.random.default_rng(m + n + k)
    a, r = _matrix(rng, m, k, kind), _matrix(rng, n, k, kind)
    c = vgtb.diag_slice_product(a, r)
    e = a.astype(np.clongdouble) @ r.conj().T.astype(np.clongdouble)
    part = lambda x: np.maximum(np.abs(x.real), np.abs(x.imag))  # noqa: E731
    scale = part(a).max(1)[:, None] * part(r).max(1)[None]
    bound = 2.0 ** -52 * part(e) + 2 * k * 2.0 ** -54 * scale
    assert np.all(part(c - e) <= bound)


def test_slice_product_real_operand_planes_and_nonfinite_rows():
    rng = np.random.default_rng(5)
    a, r = _matrix(rng, 70, 90, "decay"), _matrix(rng, 65, 90, "decay")
    real = a.real + 0j
    assert np.array_equal(vgtb.diag_slice_product(real, r, a_real=True), vgtb.diag_slice_product(real, r))
    assert np.array_equal(vgtb.diag_slice_product(a, r, planes=19), vgtb.diag_slice_product(a, r))
    a[3, 5], a[7, 1], r[9, 9] = np.inf, np.nan, -np.inf
    bad = ~np.isfinite(vgtb.diag_slice_product(a, r))
    want = np.zeros_like(bad)
    want[[3, 7]] = True
    want[:, 9] = True
    assert np.array_equal(bad, want)
