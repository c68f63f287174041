"""The FP64 form's 64-bit block fixed-point sine transform (csl_fix.cuh)
through P^{-1}: every line length (rows and columns), lines whose entries
differ by hundreds of orders of magnitude, spikes, zero lines, scaling by
powers of two, infinities and NaN.

Tolerance of a transform of N points against the dense oracle, relative to the
result's norm: the odd modes are prefix sums of N/2 terms, each rounded to 53
bits of the line's norm in FP64 arithmetic, so N 2^-53 bounds both; P^{-1}
applies two per axis, and the shift below makes its scale nearly constant
(|e + i beta| varies by less than 2), so errors are not amplified."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

LENGTHS = [4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096]


@pytest.fixture(scope="module")
def csl():
    import __graft_entry__ as g
    g.build()
    import paper_2408_00488_gb300 as csl
    return csl


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def plan(csl, ns, beta, lines=0):
    faces = W.sample_faces(2, ns, W.coef_const(1.0))
    return csl.Plan([dev(f) for f in faces], 1j * beta, autotune=False, lines_per_cta=lines)


def inputs(kind, shape, axis, rng):
    v = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    if kind == "spike":
        v[:] = 0
        v[shape[0] // 3, shape[1] // 2] = 1.25 - 3j
    elif kind == "lines":  # every line of the tested axis at a scale of its own, one of them zero
        n = shape[1 - axis]
        sc = 2.0 ** rng.integers(-20, 20, n)
        sc[n // 2] = 0.0
        v *= sc[None, :] if axis == 0 else sc[:, None]
    elif kind == "within":  # neighbours in a line 300 orders of magnitude apart
        v *= np.where(rng.random(shape) < 0.5, 1e-300, 1.0)
    return v


@pytest.mark.parametrize("N", LENGTHS)
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("kind", ["normal", "spike", "lines", "within"])
def test_line_lengths(csl, N, axis, kind):
    other = 15 if N <= 1024 else 3
    ns = (N - 1, other) if axis == 1 else (other, N - 1)
    beta = 4.0 * (4.0 * N * N + 4.0 * 256)  # above every eigenvalue of L
    v = inputs(kind, (ns[1], ns[0]), axis, np.random.default_rng(N + axis))
    r1, r2 = O.precond_apply(v.real.copy(), v.imag.copy(), 1.0, 0.0, beta)
    ref = r1 + 1j * r2
    with plan(csl, ns, beta) as p:
        out = p.precondition(dev(v)).cpu().numpy()
        assert np.linalg.norm(out - ref) <= 4 * 2 * N * 2.0**-53 * np.linalg.norm(ref)
        # a power of two goes through exactly
        up = p.precondition(dev(v * 2.0**500)).cpu().numpy()
        down = p.precondition(dev(v * 2.0**-500 if kind != "within" else v * 2.0**-10)).cpu().numpy()
        assert np.array_equal(up, out * 2.0**500)
        if kind != "within":
            assert np.array_equal(down, out * 2.0**-500)
        assert not p.precondition(dev(np.zeros_like(v))).any().item()


@pytest.mark.parametrize("lines", [1, 2, 4])
def test_tile_widths(csl, lines):
    """Columns past a tile's edge, and the variant with 128 lanes per line through its tile."""
    ns = (127, 511)
    beta = 1e7
    v = W.rhs_normal((ns[1], ns[0]), 7)
    r1, r2 = O.precond_apply(v.real.copy(), v.imag.copy(), 1.0, 0.0, beta)
    with plan(csl, ns, beta, lines) as p:
        out = p.precondition(dev(v)).cpu().numpy()
    assert np.linalg.norm(out - r1 - 1j * r2) <= 8 * 512 * 2.0**-53 * np.linalg.norm(r1 + 1j * r2)


@pytest.mark.parametrize("N,variant", [(128, 0), (128, 1), (256, 0), (256, 1), (512, 1), (512, 2), (1024, 1), (1024, 2)])
def test_variants(csl, tmp_path, N, variant):
    """Every number of lanes per line, chosen through the tuner's cache."""
    n = N - 1
    v = W.rhs_normal((n, n), 10)
    beta = 4.0 * 8.0 * N * N
    r1, r2 = O.precond_apply(v.real.copy(), v.imag.copy(), 1.0, 0.0, beta)
    ref = r1 + 1j * r2
    faces = [dev(f) for f in W.sample_faces(2, (n, n), W.coef_const(1.0))]
    path = tmp_path / "tune.txt"
    path.write_text(f"csl-tune-cache 1\n8 0 {N} {n} {n} {variant} 2\n8 2 {N} {n} 1 {variant} 2\n")
    csl.tune_cache_load(str(path))
    with csl.Plan(faces, 1j * beta) as p:
        assert p.config.count("lines=2 ") == 2
        out = p.precondition(dev(v)).cpu().numpy()
    assert np.linalg.norm(out - ref) <= 8 * N * 2.0**-53 * np.linalg.norm(ref)


@pytest.mark.parametrize("ns", [(15, 63), (127, 31), (511, 63), (1023, 15)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_spreads(csl, ns, bad):
    v = W.rhs_normal((ns[1], ns[0]), 8)
    v[3, 5] = bad
    with plan(csl, ns, 1e6) as p:
        out = p.precondition(dev(v)).cpu().numpy()
    assert not np.isfinite(out).any()


def test_range_ends(csl):
    """Results that leave the double range, and lines near its lower end."""
    ns = (63, 31)
    v = W.rhs_uniform((ns[1], ns[0]), 9)
    with plan(csl, ns, 1.0) as p:
        out = p.precondition(dev(v)).cpu().numpy()
        # every intermediate stays normal (the modes shrink by about 2^-13): still an exact scaling,
        # now through exponents at which the conversions take their far case
        assert np.array_equal(p.precondition(dev(v * 2.0**-960)).cpu().numpy(), out * 2.0**-960)
        # x pass: sums of 63 entries near the largest double overflow; no NaN-free garbage may come back
        big = np.full((ns[1], ns[0]), 1.7e308 + 1.7e308j)
        assert not np.isfinite(p.precondition(dev(big)).cpu().numpy()).all()
