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


def _mixed_system(kgrid):
    """64 diamond sites, 24 of them with a single s orbital: N = 184, uneven blocks, no block-sparse kernel."""
    from paper_2308_09782_gb300 import inputs
    sysd = inputs.diamond_si(2, 0.05, seed=64, kgrid=kgrid)
    light = np.zeros(64, bool)
    light[np.random.default_rng(2).permutation(64)[:24]] = True
    norb = np.where(light, 1, 4)
    ijl = sysd["blk_ijl"]
    a = np.arange(4)
    keep = ((a[None, :, None] < norb[ijl[:, 0]][:, None, None]) & (a[None, None, :] < norb[ijl[:, 1]][:, None, None])).ravel()
    z = np.where(light, 1.0, 4.0)
    return {**sysd, "orb_offset": np.concatenate([[0], np.cumsum(norb)]).astype(np.int32), "h0": sysd["h0"][keep],
            "s": sysd["s"][keep], "ds": np.ascontiguousarray(sysd["ds"][:, keep]), "z_ref": z,
            "n_electrons": float(z.sum())}


@pytest.mark.parametrize("kgrid", ["gamma", "mp2"])
@pytest.mark.parametrize("form", ["fp64", "fp64_delta", "cn", "split", "split_batch"])
def test_uneven_orbitals_match_oracle(form, kgrid):
    """Every product route with uneven atom blocks and an N off every tile size, at a real and at
    complex S_k, over graph-free steps: the FP64 bounds of the parity tests (J 1e-8, D 1e-10), the
    split form's J bound of 1e-4."""
    import oracle as O
    from oracle import crank_nicolson as ocn
    from paper_2308_09782_gb300 import inputs
    sysd = _mixed_system(kgrid)
    n = 6
    A = inputs.pulse_field(n, sysd["dt"], 0.01, 0.1, pol=(1.0, 0.5, 0.2), duration=40.0)
    cx = O.setup(sysd)
    nocc = int(sysd["n_electrons"]) // 2
    C = [O.occupied_states(H, S, nocc)[0] for H, S in zip(cx["H0"], cx["S"])]
    D = [2.0 * (c @ c.conj().T) for c in C]
    cn = form == "cn"
    ref = ocn.propagate_cn(sysd, A, n, C, ctx=cx) if cn else O.propagate(sysd, A, n, D, ctx=cx)
    split = form.startswith("split")
    traj = [0, 0] if form == "split_batch" else [0]
    with vgtb.Context([sysd], traj_sys=traj, init=vgtb.INIT_USER, delta_form=int(form == "fp64_delta"),
                      precision=vgtb.SPLIT_BF16X3 if split else vgtb.FP64,
                      integrator=vgtb.CRANK_NICOLSON if cn else vgtb.LEAPFROG) as c:
        for k in range(len(C)):
            (c.set_coefficients if cn else c.set_density)(0, k, C[k] if cn else D[k])
        for t in range(len(traj)):
            c.set_field(t, A)
        c.propagate(n)
        for t in range(len(traj)):
            J, E, q = c.observables(t)
            err = np.linalg.norm(J - ref["J"]) / np.linalg.norm(ref["J"])
            assert err <= (1e-4 if split else 1e-8), err
            assert np.max(np.abs(q - ref["q"])) <= (1e-5 if split else 1e-9)
            if not cn:
                X = np.stack([c.get_density(t, k) for k in range(len(C))])
                R = np.stack(ref["D"])
                assert np.linalg.norm(X - R) / np.linalg.norm(R) <= (1e-4 if split else 1e-10)


@pytest.mark.parametrize("planes", [8, 19])
def test_group_sums_are_exact_where_digits_correlate(planes):
    """[x | x] [x | -x]^dagger is zero.  Built from digits in [-127, 127], x has these digits and -x their
    negatives, so every group sum is zero too and the result has to be exactly zero.  The squares of
    equal digits (the pair (4, 4)) add up to 2 x 2048 x 127 x 128 / 3 = 2.2e7 > 2^24 half way through
    k = 4096, which FP32 does not hold unless the sums are taken out in time."""
    rng = np.random.default_rng(17)
    d = rng.integers(-127, 128, (2, 7, 40, 2048))
    d[:, 0] = rng.integers(64, 121, (2, 40, 2048))       # row maxima in [1/4, 1/2): every scale is 1
    d[:, 6] = 4 * rng.integers(-31, 32, (2, 40, 2048))   # 53 bits
    x = sum(d[:, s].astype(float) * 2.0 ** (-8 * (s + 1)) for s in range(7))
    x = x[0] + 1j * x[1]
    c = vgtb.diag_slice_product(np.hstack([x, x]), np.hstack([x, -x]), planes=planes)
    assert not np.any(c)


@pytest.mark.parametrize("shape", [(40, 33, 96), (257, 129, 513)])
@pytest.mark.parametrize("fall", [0.0, 0.05])
def test_slice_product_holds_more_than_fp64_rows(shape, fall):
    """Eight digits: with 2^e <= 4.07 of the row's largest part (slice_field) an entry is off by at most
    2^-65 2^e, a real product by 1.02 x 2^-62 of the row maxima, and the pairs left out (s + t > 10, at
    most 6.1 x 2^14 2^-88 of 2^eA 2^eR) add 2^-67: |error| <= 2^-53 |c| + 2 k 1.1 x 2^-62 max|a_row| max|r_row|,
    also for the elements that rows falling off from the diagonal make small."""
    if np.finfo(np.longdouble).nmant < 100:
        pytest.skip("the reference needs a 128-bit long double")
    m, n, k = shape
    rng = np.random.default_rng(m + k)
    a, r = ((rng.normal(size=(q, k)) + 1j * rng.normal(size=(q, k)))
            * np.exp(-fall * np.abs(np.arange(q)[:, None] - np.arange(k)[None])) for q in (m, n))
    e = a.astype(np.clongdouble) @ r.conj().T.astype(np.clongdouble)
    part = lambda x: np.maximum(np.abs(x.real), np.abs(x.imag))  # noqa: E731
    scale = part(a).max(1)[:, None] * part(r).max(1)[None]
    for planes in (8, 19):
        d = vgtb.diag_slice_product(a, r, planes=planes).astype(np.clongdouble) - e
        for got, val in ((d.real, e.real), (d.imag, e.imag)):
            assert np.all(np.abs(got) <= 2.0 ** -53 * np.abs(val) * (1 + 2.0 ** -40) + 2.2 * k * 2.0 ** -62 * scale)


@pytest.mark.parametrize("form", ["fp64", "fp64_delta", "cn"])
def test_rounds_that_share_scratch_equal_single_runs(form):
    """The digits and planes of a step's items take at most 32 GB (a quarter of the free memory): 512 atoms at
    134 MB of digits a matrix and 302 MB of planes need more than one round from 57 (32, 39) trajectories
    on.  Every trajectory equals its own single run bit for bit, whichever round holds it."""
    from paper_2308_09782_gb300 import inputs
    from tests._gpu_util import oracle_ground, system
    sysd, _, _ = system("si512_kick")
    _, gs = oracle_ground("si512_kick")
    dig, planes = 2 * 8 * 2048 * 2 * 2048, 4 * 9 * 2048 * 2 * 2048
    n_traj = int(32e9 / {"fp64": 2 * dig + planes, "fp64_delta": 3 * dig + 2 * planes, "cn": 4 * dig + planes}[form]) + 2
    n = 2
    fields = [inputs.kick_field(n, 0.001 * (1.0 + 0.1 * t), np.array([1.0, 0.1 * t, 0.0])) for t in range(n_traj)]

    def run(which):
        c = vgtb.Context([sysd], traj_sys=[0] * len(which), init=vgtb.INIT_USER, delta_form=int(form == "fp64_delta"),
                         integrator=vgtb.CRANK_NICOLSON if form == "cn" else vgtb.LEAPFROG, graph_steps=1)
        (c.set_coefficients if form == "cn" else c.set_density)(0, 0, (gs["C"] if form == "cn" else gs["D"])[0])
        for i, t in enumerate(which):
            c.set_field(i, fields[t])
        c.propagate(n)
        return c

    with run(range(n_traj)) as many:
        for t in (0, n_traj - 3, n_traj - 1):
            with run([t]) as one:
                for a, b in zip(many.observables(t), one.observables(0)):
                    assert np.array_equal(a, b)
                assert np.array_equal(many.get_density(t, 0), one.get_density(0, 0))


def test_group_sums_fit_at_the_largest_size():
    """k = 8192, the most that 32-bit group sums hold, with digits -128 wherever the row's scale allows it (the
    first one -125): every sum has one sign, and 2 k x^2 comes out to its last bit but one."""
    from fractions import Fraction
    x = sum(d * 2.0 ** (-8 * (s + 1)) for s, d in enumerate([-125] + [-128] * 6))
    a = np.full((3, 8192), x * (1 + 1j))
    want = float(2 * 8192 * Fraction(x) ** 2)
    for planes in (8, 19):
        c = vgtb.diag_slice_product(a, a, planes=planes)
        assert np.all(np.abs(c.real - want) <= 2.0 ** -52 * want) and not np.any(c.imag)
