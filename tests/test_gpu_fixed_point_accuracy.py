"""Accuracy of the FP64 form's P^{-1} on lines whose norm is little more than
their largest entry (a point source over a small background), rows and columns of
every length: against extended precision, its root mean square error may not be
larger than that of FP64 butterflies with the same split of the modes and prefix
sum, which the fixed-point form replaced (here in NumPy).  test_gpu_fixed_point.py
checks the other properties, fixed_point_host.cu single transforms."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def csl():
    import __graft_entry__ as g
    g.build()
    import paper_2408_00488_gb300 as csl
    return csl


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


PI = np.longdouble("3.14159265358979323846264338327950288")


def sines(n, den, real):
    """sin(pi k / den), k = 0 .. n-1, in the type `real`, from the extended one."""
    return np.sin(PI * np.arange(n, dtype=np.longdouble) / den).astype(real)


def fft(x):
    """FFT of the last axis (a power of two) by radix-2 Stockham passes in x's type."""
    rows, n = x.shape
    real = x.real.dtype
    half = n // 2
    m = 1
    while half >= 1:
        w = np.empty(half, x.dtype)
        w.real = np.cos(PI * np.arange(half, dtype=np.longdouble) / half).astype(real)
        w.imag = -sines(half, half, real)
        x = x.reshape(rows, 2, half, m)
        a, b = x[:, 0], x[:, 1]
        x = np.stack([a + b, (a - b) * w[None, :, None]], axis=2).reshape(rows, n)
        half //= 2
        m *= 2
    return x


def dst(z, exact):
    """DST-I of the last axis (n = N - 1 entries): an FFT of the odd extension in the
    extended type, or the split and prefix sum of the kernels in FP64."""
    rows, n = z.shape
    N = n + 1
    if exact:
        e = np.zeros((rows, 2 * N), np.clongdouble)
        e[:, 1:N] = z
        e[:, N + 1:] = -z[:, ::-1]
        f = fft(e)[:, 1:N]
        return f * np.clongdouble(0.5j)
    y = np.zeros((rows, N), np.complex128)
    j = np.minimum(np.arange(1, N), N - np.arange(1, N))
    h = 0.5 * sines(N, N, np.float64)[j]
    y[:, 1:] = h * (z + z[:, ::-1]) + 0.25 * (z - z[:, ::-1])
    Y = fft(y)
    k = np.arange(1, N // 2)
    c = np.empty((rows, N // 2), np.complex128)
    c[:, 0] = Y[:, 0]
    c[:, 1:] = Y[:, k] + Y[:, N - k]
    chunk = min(8, N // 2)
    c = np.cumsum(c.reshape(rows, -1, chunk), axis=2)  # per lane, then over the lanes
    c[:, 1:] += np.cumsum(c[:, :-1, -1], axis=1)[:, :, None]
    out = np.empty((rows, n), np.complex128)
    out[:, 0::2] = c.reshape(rows, -1)
    d = Y[:, N - k] - Y[:, k]
    out[:, 1::2] = d.imag - 1j * d.real
    return out


def precondition(v, beta, exact):
    real = np.longdouble if exact else np.float64
    ny, nx = v.shape
    mu = [4 * np.longdouble(n + 1) ** 2 * sines(n + 1, 2 * (n + 1), np.longdouble)[1:] ** 2 for n in (nx, ny)]
    e = mu[0][None, :] + mu[1][:, None]
    s = (np.longdouble(4) / ((nx + 1) * (ny + 1)) / np.sqrt(e * e + np.longdouble(beta) ** 2)).astype(real)
    t = v.astype(np.clongdouble if exact else np.complex128)
    t = dst(dst(t, exact).T, exact).T * s
    return dst(dst(t.T, exact).T, exact)


@pytest.mark.parametrize("N", [16, 128, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("kind,background", [("constant", 1e-3), ("random", 1e-3), ("random", 1e-8), ("middle", 1e-3)])
def test_point_sources(csl, N, axis, kind, background):
    other = 15
    ns = (N - 1, other) if axis == 1 else (other, N - 1)  # (nx, ny); axis 1: rows of N points
    beta = 4.0 * (4.0 * N * N + 4.0 * 256)  # above every eigenvalue of L: a scale that is nearly constant
    rng = np.random.default_rng(10 * N + axis)
    lines = rng.uniform(0.5, 1.5, (other, 1)) + 1j * rng.uniform(0.5, 1.5, (other, 1))
    v = np.repeat(background * lines, N - 1, axis=1)
    if kind == "random":
        v = background * (rng.uniform(-1, 1, v.shape) + 1j * rng.uniform(-1, 1, v.shape))
    at = np.full(other, N // 2 - 1) if kind == "middle" else rng.integers(0, N - 1, other)
    v[np.arange(other), at] += rng.uniform(0.5, 1.5, other) - 1j * rng.uniform(0.5, 1.5, other)
    v = np.ascontiguousarray(v if axis == 1 else v.T)
    ref = precondition(v, beta, True)
    faces = W.sample_faces(2, ns, W.coef_const(1.0))
    with csl.Plan([dev(f) for f in faces], 1j * beta, autotune=False) as p:
        out = p.precondition(dev(v)).cpu().numpy()
    err, err64 = (np.sqrt(float((np.abs(x.astype(np.clongdouble) - ref) ** 2).sum())) for x in
                  (out, precondition(v, beta, False)))
    assert err <= err64, (err, err64, err / err64)


@pytest.mark.parametrize("N", [64, 1024, 4096])
def test_neighbours_far_apart_scale_down(csl, N):
    """Entries 300 orders of magnitude apart, scaled down by a power of two."""
    rng = np.random.default_rng(N)
    ns = (N - 1, 15)
    v = W.rhs_normal((15, N - 1), N) * np.where(rng.random((15, N - 1)) < 0.5, 1e-300, 1.0)
    faces = W.sample_faces(2, ns, W.coef_const(1.0))
    with csl.Plan([dev(f) for f in faces], 1j * 4.0 * (4.0 * N * N + 1024.0), autotune=False) as p:
        out = p.precondition(dev(v)).cpu().numpy()
        assert np.array_equal(p.precondition(dev(v * 2.0**-10)).cpu().numpy(), out * 2.0**-10)
