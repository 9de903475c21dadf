"""The general lattice walk (any replicas, widths and alignments, FP32 and FP64) against the
oracle, at shapes where its windows, replica groups and halos can go wrong: lattices narrower
and wider than one window, 2-wide sides, replica counts that take 16-, 8- and 4-byte values and
every kind of replica group, one and several strips.

FP32: the vector bound of the lattice tests (1e-5 per replica). FP64: 1e-10 (order of the sums
only). Elements: within the bound of a cancelling sum, see _close. Steps grouped three, two or one to a
pass are bit-identical: every level computes a value with the same operations.
"""
import numpy as np
import pytest

import oracle as O
from paper_2509_01928_gb300 import _native as N
from paper_2509_01928_gb300 import build as B
from paper_2509_01928_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build_library()
    return N.load()


def _run(t, x0, alpha, beta, iters, flags=0, skip=0):
    h = N.ising_create(N.Problem(t), flags)
    try:
        src = torch.from_numpy(x0)
        buf = torch.empty(src.numel() + skip, dtype=src.dtype, device="cuda")
        x = buf[skip:].reshape(src.shape)
        x.copy_(src)
        N.ising_iterate(h, x, alpha, [beta], iters)
        return x.cpu().numpy()
    finally:
        N.ising_destroy(h)


def _close(x, ref, tol):
    x, ref = x.astype(np.float64).reshape(ref.shape), ref
    rel = np.linalg.norm(x - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert rel.max() <= tol, f"relative error {rel.max():.3e}"
    # an element: its sum of five products carries at most five roundings of relative size eps of the
    # largest terms, whose cube root is at most the largest |x|; where the sum cancels, the cube root
    # of that error remains (a wrong neighbour or window seam is an error of order 1)
    eps = 2.0 ** -24 if tol > 1e-8 else 2.0 ** -53
    assert np.abs(x - ref).max() <= (5 * eps) ** (1 / 3) * np.abs(ref).max()


@pytest.mark.parametrize("shape", [(2, 2), (2, 3), (5, 61), (3, 300), (70, 7), (41, 129)])
@pytest.mark.parametrize("R", [1, 2, 3, 4, 7, 10, 16, 17, 20, 23, 100])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_walk_matches_the_oracle(shape, R, dtype, monkeypatch):
    t = I.torus_pm1(*shape, seed=11)
    t.right[::2] *= 3
    x0 = I.x0_uniform(t.n, R, seed=12, dtype=dtype)
    alpha, beta = O.alpha_beta(t, eta=1.0, method="wigner")
    iters = 8  # two passes of three and one of two
    ref = O.doch(O.Problem(t), x0, alpha, beta, iters)
    x = _run(t, x0, [alpha], beta, iters)
    _close(x, ref.reshape(x.shape), 1e-5 if dtype == np.float32 else 1e-10)
    if dtype == np.float32 and shape[1] % 4:
        assert np.array_equal(x, _run(t, x0, [alpha], beta, iters, flags=N.FLAG_SINGLE_STEP))
        monkeypatch.setenv("ISING_LATTICE_PASS", "2")
        assert np.array_equal(x, _run(t, x0, [alpha], beta, iters))


@pytest.mark.parametrize("R", [4, 8])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_walk_unaligned_arrays_and_schedule(R, dtype):
    t = I.torus_pm1(9, 14, seed=13)
    x0 = I.x0_uniform(t.n, R, seed=14, dtype=dtype)
    alpha, beta = O.alpha_beta(t, eta=1.0, method="wigner")
    sched = alpha * (1.0 + 0.2 * np.cos(np.arange(7)))
    ref = O.doch(O.Problem(t), x0, sched, beta, 7)
    outs = [_run(t, x0, sched, beta, 7, skip=skip) for skip in (0, 1, 2)]
    _close(outs[0], ref, 1e-5 if dtype == np.float32 else 1e-10)
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_update_of_extreme_values(dtype):
    """Zeros, subnormal and huge values, infinities and NaN: the update's cube root keeps signs,
    zeros and non-finite values where CUDA's cbrt has them."""
    t = I.torus_pm1(6, 10, seed=15)
    big = 1e30 if dtype == np.float32 else 1e200
    x0 = I.x0_uniform(t.n, 2, seed=16, dtype=dtype)
    x0[0], x0[7], x0[20], x0[33], x0[45] = 0.0, big, -big, np.inf, np.nan
    x0[50:56] = 0.0
    x = _run(t, x0, [1.0], 2.0, 1)
    with np.errstate(all="ignore"):
        z = x0.astype(np.float64).reshape(6, 10, 2)
        r, d = t.right.astype(float)[..., None], t.down.astype(float)[..., None]
        u = (r * np.roll(z, -1, 1) + np.roll(r, 1, 1) * np.roll(z, 1, 1) + d * np.roll(z, -1, 0)
             + np.roll(d, 1, 0) * np.roll(z, 1, 0) + z)
        ref = np.cbrt(u / 2.0).reshape(x.shape)
    assert np.array_equal(np.isnan(x), np.isnan(ref)) and np.array_equal(np.isinf(x), np.isinf(ref))
    ok = np.isfinite(ref)
    np.testing.assert_allclose(x[ok], ref[ok], rtol=1e-6 if dtype == np.float32 else 1e-14, atol=1e-6)
    assert np.all(x[ref == 0] == 0)


@pytest.mark.parametrize("form", ["lattice", "csr"])
@pytest.mark.parametrize("lo, hi, beta", [(-149, -100, 2.0 ** -6), (-125, -118, 1.0), (119, 124, 1.0), (-149, 124, 1.0),
                                          (-10, 10, 2.0)])
def test_fp32_roots_of_any_size(form, lo, hi, beta):
    """FP32 updates whose root lies outside 2^-40 .. 2^40, subnormal sums among them, are as exact as the
    rest. All terms are positive: the five-term sum (six roundings with the division) and the cube root give
    a relative error of at most (6 / 3 + 1) 2^-24, or half the spacing of subnormal quotients in z."""
    t = I.torus_pm1(30, 42, seed=17)
    t.right[:], t.down[:] = 1, 1
    rng = np.random.default_rng(18)
    x0 = (np.exp2(rng.uniform(lo, hi, (t.n, 4)))).astype(np.float32)
    x0[5] = 0.0
    x = _run(t if form == "lattice" else t.to_csr(), x0, [1.0], beta, 1)
    z = x0.astype(np.float64).reshape(30, 42, 4)
    u = sum(np.roll(z, s, a) for s in (1, -1) for a in (0, 1)) + z
    a = (u / beta).reshape(x.shape)
    room = np.maximum(np.cbrt(a + 2.0 ** -149) - np.cbrt(a), np.cbrt(a) * 3 * 2.0 ** -24)
    assert np.all(np.abs(x.astype(np.float64) - np.cbrt(a)) <= room)


def test_zero_replica_beside_others():
    """A replica at zero (a fixed point) leaves the near range in every block; the others keep their values."""
    t = I.torus_pm1(20, 37, seed=19)
    x0 = I.x0_uniform(t.n, 4, seed=20)
    alpha, beta = O.alpha_beta(t, eta=1.0, method="wigner")
    whole = _run(t, x0, [alpha], beta, 7)
    x0[:, 2] = 0.0
    x = _run(t, x0, [alpha], beta, 7)
    assert np.all(x[:, 2] == 0.0) and np.array_equal(x[:, [0, 1, 3]], whole[:, [0, 1, 3]])
