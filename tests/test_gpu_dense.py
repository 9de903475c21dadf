"""Dense couplings on the tcgen05 tensor cores against the FP64 oracle.

Iterates are BF16 (the dense path's storage type). The oracle starts from the
same BF16-rounded x0.
  * One step: every element within one BF16 ulp of the oracle's x^(1) rounded
    to BF16 (the GEMM accumulates in FP32 and the result is rounded once).
  * N = 10 steps: the BF16 bar, ||x_gpu - x_ref|| / ||x_ref|| <= 2e-2 for the
    median replica and for at least 85 % of the replicas. Replicas near
    weakly stable fixed points amplify the per-step BF16 rounding of the
    state (2^-9) and some leave for another basin; which ones depends on the
    rounding sequence, so per-replica parity is not pinned beyond a few steps.
  * N = 50 steps: the median replica within 2e-2, and the mean Ising energy
    of the final spins within 2 % of the oracle's (each side computing its
    own energies).
  * Energies and cuts of a given spin vector are exact integers (J S
    accumulates exactly in FP32 for integer J with |J| <= 256): bit for bit.
Couplings in {-1, 0, +1} take the packed ternary storage (expanded on chip);
other integer couplings the BF16 storage; both are tested.
"""
import numpy as np
import pytest

import oracle as O
from paper_2509_01928_gb300 import _native as N
from paper_2509_01928_gb300 import build as B
from paper_2509_01928_gb300 import inputs as I
from fp32_bounds import close32_conditioned, fp32_drift

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_BF16 = 2e-2


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available()
    B.build_library()
    return N.load()


def _jmat(kind, n, seed):
    """Symmetric integer couplings with zero diagonal: "pm1" (dense +-1, held as packed
    ternary codes), "pm1_sparse" (+-1 with about half the pairs zero, ternary) or "int"
    (|J| in 1..3, held as BF16)."""
    J = I.dense_pm1(n, seed=seed).astype(np.int64)
    if kind == "pm1":
        return J.astype(np.int8)
    u = np.triu(I.x0_uniform(n, n, seed=seed + 1), 1)
    u = u + u.T
    if kind == "pm1_sparse":
        return (J * (np.abs(u) >= 0.5)).astype(np.int8)
    return (J * (1 + np.floor(3 * np.abs(u)).clip(0, 2))).astype(np.int8)


def _bf16(x):
    t = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).to(torch.bfloat16)
    return t, t.float().numpy().astype(np.float64)


def _rel(a, b):
    return np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)


def _bf16_ulp(v):
    """Spacing of BF16 numbers at |v| (8 significant bits)."""
    e = np.floor(np.log2(np.maximum(np.abs(v), 1e-38)))
    return 2.0 ** (e - 7)


@pytest.mark.parametrize("n, R, kind", [(256, 32, "pm1"), (200, 20, "pm1"), (130, 5, "pm1"), (384, 256, "pm1"),
                                        (256, 32, "int"), (200, 20, "int"), (384, 256, "int"),
                                        (200, 20, "pm1_sparse"), (384, 48, "pm1_sparse")])
def test_dense_iterates_bf16(n, R, kind):
    J = _jmat(kind, n, 91)
    P = O.Problem(J)
    alpha, beta = O.alpha_beta(J, eta=1.0, method="eig")
    xt, x0 = _bf16(I.x0_uniform(n, R, seed=92))
    h = N.ising_create(N.Problem(J))
    try:
        x = xt.cuda()
        N.ising_iterate(h, x, [alpha], [beta], 1)
        ref1 = O.doch(P, x0, alpha, beta, 1)
        ref1_bf = torch.from_numpy(ref1.astype(np.float32)).to(torch.bfloat16).float().numpy()
        got = x.float().cpu().numpy()
        assert np.all(np.abs(got - ref1_bf) <= _bf16_ulp(ref1) * 1.0001)
        N.ising_iterate(h, x, [alpha], [beta], 9)
        ref = O.doch(P, x0, alpha, beta, 10)
        rel = _rel(x.float().cpu().numpy().astype(np.float64), ref)
        assert np.median(rel) <= TOL_BF16
        assert np.mean(rel <= TOL_BF16) >= 0.85, f"N=10: {np.mean(rel <= TOL_BF16):.2f} within 2e-2"
        N.ising_iterate(h, x, [alpha], [beta], 40)
        ref = O.doch(P, x0, alpha, beta, 50)
        rel = _rel(x.float().cpu().numpy().astype(np.float64), ref)
        assert np.median(rel) <= TOL_BF16
        E = np.zeros(R, np.int64)
        N.ising_energy(h, x, E_int=E)
        Er, _ = O.energy_int(P, O.sign(ref))
        assert abs(E.mean() - Er.mean()) <= 0.02 * abs(Er.mean())
    finally:
        N.ising_destroy(h)


@pytest.mark.parametrize("n, R, kind", [(65, 3, "pm1"), (1000, 256, "int"), (1100, 300, "pm1"), (2300, 100, "pm1"),
                                        (2440, 33, "pm1_sparse"), (4100, 16, "pm1"), (4100, 5, "int")])
def test_dense_narrow_replica_tiles(n, R, kind):
    """Instances whose row tiles leave SMs idle: the replicas are taken in tiles of 16 to 256 (counts that
    do not divide the replicas). One step within one BF16 ulp, energies exact."""
    J = _jmat(kind, n, 96)
    P = O.Problem(J)
    alpha, beta = O.alpha_beta(J, eta=1.0, method="wigner")
    xt, x0 = _bf16(I.x0_uniform(n, R, seed=97))
    h = N.ising_create(N.Problem(J))
    try:
        x = xt.cuda()
        N.ising_iterate(h, x, [alpha], [beta], 1)
        ref = O.doch(P, x0, alpha, beta, 1)
        ref_bf = torch.from_numpy(ref.astype(np.float32)).to(torch.bfloat16).float().numpy()
        # z = (J x + alpha x)_i is an FP32 sum of n terms |J x| with partial sums of order sqrt(n): its rounding
        # stays below n 2^-24 max|J|, which the root of a z near zero amplifies
        z, dz = beta * ref ** 3, n * 2.0 ** -24 * np.abs(J).max()
        amplified = np.maximum(np.abs(np.cbrt((z + dz) / beta) - ref), np.abs(np.cbrt((z - dz) / beta) - ref))
        err = np.abs(x.float().cpu().numpy() - ref_bf)
        assert np.all(err <= _bf16_ulp(ref) * 1.0001 + amplified)
        assert np.mean(err <= _bf16_ulp(ref) * 1.0001) >= 0.9999  # such z are rare
        E = np.zeros(R, np.int64)
        N.ising_energy(h, xt.cuda(), E_int=E)
        s = O.sign(x0).astype(np.int64)
        assert np.array_equal(E, -((s * (J.astype(np.int64) @ s)).sum(0) // 2))
    finally:
        N.ising_destroy(h)


@pytest.mark.parametrize("n, R, kind", [(300, 40, "pm1"), (128, 1, "pm1"), (520, 257, "pm1"),
                                        (300, 40, "int"), (520, 257, "int"), (300, 40, "pm1_sparse")])
def test_dense_energy_exact(n, R, kind):
    J = _jmat(kind, n, 93)
    hf = (np.round(3 * I.field_gauss(n, 1.0, seed=94))).astype(np.int8)
    x = I.x0_uniform(n, R, seed=95)
    x[::7] = 0.0
    s = O.sign(x.astype(np.float64))
    Er, cr = O.energy_int(O.Problem(J, hf), s)
    h = N.ising_create(N.Problem(J, hf))
    try:
        for xin in (torch.from_numpy(x).cuda(), torch.from_numpy(s).cuda(), torch.from_numpy(x).to(torch.bfloat16).cuda()):
            E = np.zeros(R, np.int64)
            cut = np.zeros(R, np.int64)
            best = np.zeros(1, np.int32)
            N.ising_energy(h, xin, E_int=E, cut_int=cut, best=best)
            assert np.array_equal(E, Er)
            assert np.array_equal(cut, cr)
            assert best[0] == int(np.argmin(Er))
    finally:
        N.ising_destroy(h)


@pytest.mark.parametrize("n, R, alone", [(2000, 400, 100), (6000, 300, 64), (1000, 256, 1)])
def test_dense_replicas_do_not_depend_on_each_other(n, R, alone):
    """A replica's iterates are the same, bit by bit, however many run beside it: every product adds its K
    blocks in one order, whatever the tiles."""
    h = N.ising_create(N.Problem(_jmat("pm1", n, 98)), N.FLAG_SKIP_VALIDATION)
    try:
        x0 = torch.from_numpy(I.x0_uniform(n, R, seed=99)).to(torch.bfloat16).cuda()
        x, y = x0.clone(), x0[:, :alone].contiguous()
        for v in (x, y):
            N.ising_iterate(h, v, [2.0 * n ** 0.5], [n ** 1.5 * (2.0 * n ** 0.5 + n)], 6)
        assert torch.equal(x[:, :alone], y)
    finally:
        N.ising_destroy(h)


def test_dense_energy_terms_add_in_64_bits():
    """The 128 terms s_i (J s)_i of a row tile reach 2^31 past n = 65536 at |J| = 256 (a matrix too large
    for a test): the warp sum of its lanes' terms (four rows each, up to 2^26 and beyond) on its own."""
    rng = np.random.default_rng(5)
    t = rng.integers(-2 ** 31, 2 ** 31, (200, 32))
    t[0], t[1], t[2] = 4 * 256 * 70000, -4 * 256 * 70000, 2 ** 31 - 1
    t[3], t[4], t[5] = -2 ** 31, 0, -1
    td = torch.from_numpy(t.astype(np.int32)).cuda()
    out = torch.empty(len(t), dtype=torch.int64, device="cuda")
    assert N.load().ising_selftest_warp_sum(N._ptr(td), N._ptr(out), len(t), None) == 0
    assert np.array_equal(out.cpu().numpy(), t.sum(1))


def test_dense_full_size_16384x256_sampled():
    """n = 16384 dense +-1, R = 256 BF16 replicas: all replicas run on the GPU,
    two sampled replicas are recomputed by the oracle (iterates after 1 and 5
    steps within the BF16 bar; energies of the seeded start exact)."""
    n, R = 16384, 256
    J = I.dense_pm1(n, seed=3)
    alpha, beta = O.alpha_beta(J, eta=1.0, method="wigner")
    xt, x0 = _bf16(I.x0_uniform(n, R, seed=3))
    sample = [0, 201]
    P = O.Problem(J)
    h = N.ising_create(N.Problem(J))
    try:
        E = torch.zeros(R, dtype=torch.int64, device="cuda")
        x = xt.cuda()
        N.ising_energy(h, x, E_int=E)
        Er, _ = O.energy_int(P, O.sign(x0[:, sample]))
        assert np.array_equal(E.cpu().numpy()[sample], Er)
        N.ising_iterate(h, x, [alpha], [beta], 1)
        ref1 = O.doch(P, x0[:, sample], alpha, beta, 1)
        assert _rel(x.float().cpu().numpy()[:, sample].astype(np.float64), ref1).max() <= TOL_BF16
        N.ising_iterate(h, x, [alpha], [beta], 4)
        ref5 = O.doch(P, x0[:, sample], alpha, beta, 5)
        assert _rel(x.float().cpu().numpy()[:, sample].astype(np.float64), ref5).max() <= TOL_BF16
    finally:
        N.ising_destroy(h)


def test_dense_fp8_input_is_the_int8_problem():
    """J given as FP8 E4M3 bytes (+1 = 0x38, -1 = 0xB8, 0 = 0x00, 2 = 0x40, 3 = 0x44) creates the
    same device problem as the int8 matrix: identical iterates and exact energies."""
    n, R = 200, 20
    for kind in ("pm1", "int"):
        J = _jmat(kind, n, 97)
        codes = {1: 0x38, -1: 0xB8, 0: 0x00, 2: 0x40, -2: 0xC0, 3: 0x44, -3: 0xC4}
        J8 = np.vectorize(lambda v: codes[int(v)])(J).astype(np.uint8)
        alpha, beta = O.alpha_beta(J, eta=1.0, method="eig")
        xt, _ = _bf16(I.x0_uniform(n, R, seed=98))
        outs = []
        for prob in (N.Problem(J), N.Problem(J8, jtype=N.FP8E4M3)):
            h = N.ising_create(prob)
            try:
                x = xt.cuda()
                N.ising_iterate(h, x, [alpha], [beta], 12)
                E = np.zeros(R, np.int64)
                N.ising_energy(h, x, E_int=E)
                outs.append((x.float().cpu().numpy(), E))
            finally:
                N.ising_destroy(h)
        assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


# ---------------------------------------------------------------------------
# plain FP32 form (F32 iterates: FP32 products and accumulation on the CUDA cores)
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("n, R, kind", [(256, 32, "pm1"), (200, 5, "pm1"), (1500, 8, "pm1"), (384, 130, "pm1"),
                                        (200, 20, "int"), (1500, 8, "int"), (384, 48, "pm1_sparse")])
@pytest.mark.parametrize("iters", [1, 10])
def test_dense_iterates_f32(n, R, kind, iters):
    """FP32 iterates against the FP64 oracle: one step within the FP32 bar (1e-5 relative per
    replica, every element within 1e-4 of the largest); ten steps under the conditioned FP32
    bound with the dense step's rounding sqrt(n) 2^-24 (weakly stable replicas amplify it, see
    fp32_bounds). Ragged n (not a
    multiple of the 128-row tile or the 64-column stage), ragged R (scalar loads) and two
    replica tiles (R = 130)."""
    J = _jmat(kind, n, 93)
    alpha, beta = O.alpha_beta(J, eta=1.0, method="eig")
    x0 = I.x0_uniform(n, R, seed=94)
    ref, drift = fp32_drift(O.Problem(J), x0, alpha, beta, iters, eps_step=np.sqrt(n) * 2.0 ** -24)
    h = N.ising_create(N.Problem(J))
    try:
        x = torch.from_numpy(x0.copy()).cuda()
        N.ising_iterate(h, x, [alpha], [beta], iters)
        got = x.cpu().numpy().astype(np.float64)
    finally:
        N.ising_destroy(h)
    if iters == 1:
        assert _rel(got, ref).max() <= 1e-5, _rel(got, ref).max()
        assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()
    else:
        close32_conditioned(got, ref, drift)


def test_dense_f32_full_size_16384x256_sampled():
    """n = 16384 dense +-1, R = 256 FP32 replicas: two sampled replicas recomputed by the
    oracle, after 1 step within 1e-5, after 5 steps under the conditioned FP32 bound; the exact
    energy of the device's own spins."""
    n, R = 16384, 256
    J = I.dense_pm1(n, seed=3)
    alpha, beta = O.alpha_beta(J, eta=1.0, method="wigner")
    x0 = I.x0_uniform(n, R, seed=3)
    sample = [0, 201]
    P = O.Problem(J)
    h = N.ising_create(N.Problem(J))
    try:
        x = torch.from_numpy(x0.copy()).cuda()
        N.ising_iterate(h, x, [alpha], [beta], 1)
        ref1 = O.doch(P, x0[:, sample], alpha, beta, 1)
        assert _rel(x.cpu().numpy()[:, sample].astype(np.float64), ref1).max() <= 1e-5
        N.ising_iterate(h, x, [alpha], [beta], 4)
        ref5, drift = fp32_drift(P, x0[:, sample], alpha, beta, 5, eps_step=np.sqrt(n) * 2.0 ** -24)
        close32_conditioned(x.cpu().numpy()[:, sample].astype(np.float64), ref5, drift)
        E = torch.zeros(R, dtype=torch.int64, device="cuda")
        N.ising_energy(h, x, E_int=E)
        Er, _ = O.energy_int(P, O.sign(x.cpu().numpy()[:, sample].astype(np.float64)))
        assert np.array_equal(E.cpu().numpy()[sample], Er)
    finally:
        N.ising_destroy(h)


def test_dense_bf16_and_f32_forms_reach_equal_final_energy():
    """The low-precision form (BF16 state, tensor cores) against the plain FP32 form on the
    same dense +-1 instance and the same 64 starts, 300 iterations each: per-replica basins may
    differ (BF16 rounding of the state, 2^-9), so the comparison is of the energy distributions
    over replicas -- mean within 1 %, best within 2 % -- and both forms' spins have exact
    integer energies (checked against the oracle on four replicas)."""
    n, R, iters = 2048, 64, 300
    J = I.dense_pm1(n, seed=95)
    alpha, beta = O.alpha_beta(J, eta=1.0, method="eig")
    x0 = I.x0_uniform(n, R, seed=96)
    P = O.Problem(J)
    h = N.ising_create(N.Problem(J))
    out = {}
    try:
        for name, x in (("bf16", torch.from_numpy(x0).to(torch.bfloat16).cuda()),
                        ("f32", torch.from_numpy(x0.copy()).cuda())):
            N.ising_iterate(h, x, [alpha], [beta], iters)
            E = torch.zeros(R, dtype=torch.int64, device="cuda")
            N.ising_energy(h, x, E_int=E)
            s = O.sign(x.float().cpu().numpy().astype(np.float64))
            out[name] = E.cpu().numpy()
            Er, _ = O.energy_int(P, s[:, :4])
            assert np.array_equal(out[name][:4], Er)
    finally:
        N.ising_destroy(h)
    b, f = out["bf16"].astype(np.float64), out["f32"].astype(np.float64)
    assert abs(b.mean() - f.mean()) <= 0.01 * abs(f.mean()), (b.mean(), f.mean())
    assert abs(b.min() - f.min()) <= 0.02 * abs(f.min()), (b.min(), f.min())
