"""GPU adjoint (ising_backward) against the FP64 oracle adjoint.

The oracle's adjoint is pinned on the CPU against central finite differences
and a forward-mode dense Jacobian (tests/test_oracle_pins.py). Here the GPU
adjoint must match it within 1e-3 relative (vector norms, and every entry
within 1e-3 of the largest), the loss within 1e-5 relative, and the result
must not depend on the checkpoint interval.

Two precisions: x0 in FP64 runs the forward recompute in FP64 (adjoint
recursion in FP32) and must meet 1e-3 on any start. x0 in FP32 runs the
whole unrolled iteration in FP32; there d x^(k+1)/d x^k = diag(1/(3 (x^(k+1))^2))
(J + alpha I)/beta makes the gradient sensitive to components that pass near
zero in the transient, and FP32 rounding of the trajectory alone (a numpy
FP32 emulation shows the same) moves some replicas' gradients by up to
~2e-2. The FP32 path is therefore held to 1e-3 where the trajectory has no
such crossings (a periodic lattice; a graph started at a converged state),
and from random starts on random regular graphs to the loss (1e-5) and the
direction of dL/dalpha (cosine >= 0.999).
"""
import numpy as np
import pytest

import oracle as O
from paper_2509_01928_gb300 import _native as N
from paper_2509_01928_gb300 import build as B
from paper_2509_01928_gb300 import inputs as I
from short_rows import short_rows_mixed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available()
    B.build_library()
    return N.load()


def _gpu_backward(h, x0, alpha, beta, iters, ckpt):
    R = x0.shape[1]
    ga = torch.zeros(iters, dtype=torch.float64, device="cuda")
    gx = torch.zeros(x0.shape, dtype=torch.float64 if x0.dtype == np.float64 else torch.float32,
                     device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    ze = torch.zeros(1, dtype=torch.int64, device="cuda")
    N.ising_backward(h, torch.from_numpy(x0).cuda(), alpha, beta, iters, ckpt, grad_alpha=ga, grad_x0=gx,
                     loss=loss, zero_events=ze)
    torch.cuda.synchronize()
    return ga.cpu().numpy(), gx.cpu().numpy().astype(np.float64), loss.item(), ze.item()


def _rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))


@pytest.mark.parametrize("R, iters, ckpt", [(8, 40, 7), (6, 25, 25), (1, 13, 4)])
def test_adjoint_matches_oracle(R, iters, ckpt):
    g = I.regular_pm1(3000, 3, seed=5)
    x0 = I.x0_uniform(g.n, R, seed=81, dtype=np.float64)
    a0, beta = O.alpha_beta(g, eta=1.0, method="eig")
    alpha = a0 * (1.0 + 0.1 * np.cos(np.arange(iters) / 3.0))
    ga_r, gx_r, loss_r, z_r = O.backward(O.Problem(g), x0, alpha, beta, iters)
    p = N.Problem(g)
    h = N.ising_create(p)
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, ckpt)
        ga2, gx2, loss2, _ = _gpu_backward(h, x0, alpha, beta, iters, 1)
    finally:
        N.ising_destroy(h)
    assert ze == z_r == 0
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert _rel(ga, ga_r) <= 1e-3 and np.abs(ga - ga_r).max() <= 1e-3 * np.abs(ga_r).max()
    assert _rel(gx, gx_r) <= 1e-3 and np.abs(gx - gx_r).max() <= 1e-3 * np.abs(gx_r).max()
    # checkpoint-and-recompute is exact: any interval gives the same numbers
    assert np.array_equal(ga, ga2) and np.array_equal(gx, gx2) and loss == loss2


@pytest.mark.parametrize("R", [8, 6, 3])
def test_adjoint_short_rows_mixed_degrees(R):
    """The adjoint step pipelines its loads across a thread's rows; on 40,010 spins with empty
    rows, hub rows longer than its first batch of 4 entries and a hub as the last row it
    matches the oracle adjoint (FP64 forward), for every vector width."""
    g = short_rows_mixed(40010, seed=71)
    deg = np.diff(g.row_ptr)
    assert deg.min() == 0 and deg.max() > 4 and deg[-1] > 4
    iters = 12
    x0 = I.x0_uniform(g.n, R, seed=86, dtype=np.float64)
    a0, beta = O.alpha_beta(g, eta=1.0, method="wigner")
    alpha = a0 * (1.0 + 0.1 * np.cos(np.arange(iters) / 3.0))
    ga_r, gx_r, loss_r, _ = O.backward(O.Problem(g), x0, alpha, beta, iters)
    h = N.ising_create(N.Problem(g))
    try:
        ga, gx, loss, _ = _gpu_backward(h, x0, alpha, beta, iters, 5)
    finally:
        N.ising_destroy(h)
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert _rel(ga, ga_r) <= 1e-3 and np.abs(ga - ga_r).max() <= 1e-3 * np.abs(ga_r).max()
    assert _rel(gx, gx_r) <= 1e-3 and np.abs(gx - gx_r).max() <= 1e-3 * np.abs(gx_r).max()


@pytest.mark.parametrize("n, R, iters, ckpt", [(36, 3, 5, 2), (130, 1, 9, 1), (1000, 2, 12, 50), (1003, 38, 6, 4),
                                               (1003, 39, 6, 4), (1848, 5, 7, 3), (1850, 2, 4, 3)])
def test_adjoint_of_small_instances(n, R, iters, ckpt):
    """Instances whose iterate fits in shared memory run whole segments per launch: one CTA or a
    cluster per replica, shares that do not divide n, segments of one step, more replicas than
    clusters of four fit (single steps), and both sides of 2048 spins."""
    g = short_rows_mixed(n + 200 + n % 2, seed=n)
    x0 = I.x0_uniform(g.n, R, seed=87, dtype=np.float64)
    a0, beta = O.alpha_beta(g, eta=1.0, method="wigner")
    alpha = a0 * (1.0 + 0.1 * np.cos(np.arange(iters) / 3.0))
    ga_r, gx_r, loss_r, z_r = O.backward(O.Problem(g), x0, alpha, beta, iters)
    h = N.ising_create(N.Problem(g))
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, ckpt)
    finally:
        N.ising_destroy(h)
    assert ze == z_r
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert _rel(ga, ga_r) <= 1e-3 and np.abs(ga - ga_r).max() <= 1e-3 * np.abs(ga_r).max()
    assert _rel(gx, gx_r) <= 1e-3 and np.abs(gx - gx_r).max() <= 1e-3 * np.abs(gx_r).max()


@pytest.mark.parametrize("per_row, R, iters, ckpt", [(35, 10, 65, 32), (30, 10, 65, 32), (55, 11, 42, 20), (70, 10, 33, 32),
                                                     (40, 14, 65, 32), (55, 16, 21, 20)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_adjoint_of_long_rows_with_a_short_last_segment(per_row, R, iters, ckpt, dtype):
    """Segments of different lengths need different shared memory, which decides how many CTAs a
    replica can have: every dL/dalpha_k must come from the same layout of partial sums. FP64 gradients
    are compared entry by entry, FP32 ones by norm within what the rounding of their trajectory moves
    (about 2e-2 at most, as above), both bit by bit between checkpoint intervals."""
    g = I.erdos_renyi_pm1(2000, per_row / 2000, seed=89)
    P = O.Problem(g)
    a0, beta = O.alpha_beta(g, eta=1.0, method="wigner")
    alpha = a0 * (1.0 + 0.1 * np.cos(np.arange(iters) / 3.0))
    x0 = O.doch(P, I.x0_uniform(g.n, R, seed=90, dtype=np.float64), a0, beta, 300).astype(dtype)
    ga_r, gx_r, loss_r, z_r = O.backward(P, x0, alpha, beta, iters)
    h = N.ising_create(N.Problem(g))
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, ckpt)
        ga1, gx1, loss1, _ = _gpu_backward(h, x0, alpha, beta, iters, 1)
        gan, gxn, lossn, _ = _gpu_backward(h, x0, alpha, beta, iters, iters)
    finally:
        N.ising_destroy(h)
    assert ze == z_r
    assert loss == loss1 == lossn == pytest.approx(loss_r, rel=1e-5)
    # checkpoint-and-recompute is exact: any interval gives the same numbers
    for o_ga, o_gx in ((ga1, gx1), (gan, gxn)):
        assert np.array_equal(o_ga, ga) and np.array_equal(o_gx, gx)
    if dtype == np.float32:
        assert _rel(ga, ga_r) <= 2e-2
        return
    # each entry against the size of its own step's neighbours: the gradients of early steps are small
    near = np.maximum.reduce([np.abs(np.roll(ga_r, k)) for k in (-2, -1, 0, 1, 2)])
    assert np.all(np.abs(ga - ga_r) <= 1e-3 * near)
    assert _rel(gx, gx_r) <= 1e-3


def test_adjoint_with_field_and_gaussian_couplings():
    g = I.regular_gauss(2000, 5, seed=82)
    hf = I.field_gauss(g.n, 0.1, seed=83)
    g.val = g.val.astype(np.float32)
    hf32 = hf.astype(np.float32)
    R, iters = 4, 30
    x0 = I.x0_uniform(g.n, R, seed=84, dtype=np.float64)
    a0, beta = O.alpha_beta(g, eta=1.0, method="eig")
    alpha = np.full(iters, a0)
    ga_r, gx_r, loss_r, _ = O.backward(O.Problem(g, hf32.astype(np.float64)), x0, alpha, beta, iters)
    h = N.ising_create(N.Problem(g, hf32))
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, 8)
    finally:
        N.ising_destroy(h)
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert _rel(ga, ga_r) <= 1e-3
    assert _rel(gx, gx_r) <= 1e-3


@pytest.mark.parametrize("case", ["lattice_random_start", "er_converged_start"])
def test_adjoint_fp32_matches_oracle_when_well_conditioned(case):
    """FP32 end to end where the trajectory keeps away from zero crossings:
    a periodic lattice (as CSR) from a random start, and the Erdos-Renyi
    n = 800 graph started at a converged oracle state (the alpha schedule
    then only moves the fixed point slightly)."""
    R, iters = 8, 40
    if case == "lattice_random_start":
        g = I.torus_pm1(40, 50, seed=3).to_csr()
    else:
        g = I.erdos_renyi_pm1(800, 0.06, seed=1)
    P = O.Problem(g)
    a0, beta = O.alpha_beta(g, eta=1.0, method="eig")
    alpha = a0 * (1.0 + 0.1 * np.cos(np.arange(iters) / 3.0))
    x0 = I.x0_uniform(g.n, R, seed=81, dtype=np.float64)
    if case == "er_converged_start":
        x0 = O.doch(P, x0, a0, beta, 300)
    x0 = x0.astype(np.float32)
    ga_r, gx_r, loss_r, _ = O.backward(P, x0, alpha, beta, iters)
    h = N.ising_create(N.Problem(g))
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, 6)
    finally:
        N.ising_destroy(h)
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert _rel(ga, ga_r) <= 1e-3 and np.abs(ga - ga_r).max() <= 1e-3 * np.abs(ga_r).max()
    assert _rel(gx, gx_r) <= 1e-3 and np.abs(gx - gx_r).max() <= 1e-3 * np.abs(gx_r).max()


def test_adjoint_fp32_random_start_loss_and_direction():
    g = I.regular_pm1(3000, 3, seed=5)
    R, iters = 8, 40
    x0 = I.x0_uniform(g.n, R, seed=81)
    a0, beta = O.alpha_beta(g, eta=1.0, method="eig")
    alpha = a0 * (1.0 + 0.1 * np.cos(np.arange(iters) / 3.0))
    ga_r, gx_r, loss_r, _ = O.backward(O.Problem(g), x0, alpha, beta, iters)
    h = N.ising_create(N.Problem(g))
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, 7)
    finally:
        N.ising_destroy(h)
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert ga @ ga_r / (np.linalg.norm(ga) * np.linalg.norm(ga_r)) >= 0.999


def test_autograd_function_and_schedule_descent():
    from paper_2509_01928_gb300.autograd import relaxed_energy

    g = I.regular_pm1(4000, 3, seed=85)
    R, iters = 16, 30
    x0 = torch.from_numpy(I.x0_uniform(g.n, R, seed=86)).cuda().requires_grad_(True)
    a0, beta = O.alpha_beta(g, eta=1.0, method="eig")
    alpha = torch.full((iters,), a0, dtype=torch.float64, device="cuda", requires_grad=True)
    h = N.ising_create(N.Problem(g))
    try:
        L = relaxed_energy(x0, alpha, h, beta, ckpt_every=10)
        L.backward()
        ga, gx, loss, _ = _gpu_backward(h, x0.detach().cpu().numpy(), alpha.detach().cpu().numpy(), beta, iters, 10)
        assert L.item() == loss
        assert np.array_equal(alpha.grad.cpu().numpy(), ga)
        assert np.array_equal(x0.grad.cpu().numpy().astype(np.float64), gx)
        # a small step against the gradient lowers the loss (first-order descent)
        step = 1e-3 * a0 / np.abs(ga).max()
        with torch.no_grad():
            L2 = relaxed_energy(x0, alpha - step * alpha.grad, h, beta, ckpt_every=10)
        assert L2.item() < L.item()
    finally:
        N.ising_destroy(h)


def test_backward_argument_errors():
    t = I.torus_pm1(8, 8, seed=87)
    h = N.ising_create(N.Problem(t))
    try:
        x0 = torch.zeros((t.n, 1), dtype=torch.float32, device="cuda")
        with pytest.raises(N.IsingError) as e:
            N.ising_backward(h, x0, [1.0], 1.0, 1, 1)
        assert e.value.name == "ISING_ERR_UNSUPPORTED"
    finally:
        N.ising_destroy(h)


def test_adjoint_full_size_3regular_1e5():
    """n = 1e5 random 3-regular graph, +-1 couplings, R = 64, 200 FP32 iterations,
    checkpoint every 20, against the FP64 oracle adjoint on all 64 replicas."""
    g = I.regular_pm1(100_000, 3, seed=5)
    R, iters = 64, 200
    x0 = I.x0_uniform(g.n, R, seed=5, dtype=np.float64)
    a0, beta = O.alpha_beta(g, eta=1.0, method="wigner")
    alpha = np.full(iters, a0)
    h = N.ising_create(N.Problem(g))
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, 20)
    finally:
        N.ising_destroy(h)
    ga_r, gx_r, loss_r, z_r = O.backward(O.Problem(g), x0, alpha, beta, iters)
    assert ze == z_r
    assert loss == pytest.approx(loss_r, rel=1e-5)
    assert _rel(ga, ga_r) <= 1e-3
    assert _rel(gx, gx_r) <= 1e-3


def test_adjoint_fp32_full_size_along_the_device_trajectory():
    """The stated configuration end to end in FP32: n = 1e5 random 3-regular
    graph, +-1 couplings, R = 64, 200 FP32 iterations, checkpoint every 20.
    An FP32 trajectory differs from the FP64 one where components pass near
    zero, so the FP32 adjoint is checked against the FP64 oracle adjoint
    replayed along the device's own FP32 trajectory: the trajectory comes from
    200 single-step ising_iterate calls (bit-identical to one 200-step call,
    which is the forward kernel ising_backward recomputes with), each of its
    steps is checked against T in FP64 applied to the device's previous
    iterate, and the gradients must agree within 1e-3 relative (the loss within
    1e-6, the zero-crossing count exactly)."""
    g = I.regular_pm1(100_000, 3, seed=5)
    R, iters, ckpt = 64, 200, 20
    x0 = I.x0_uniform(g.n, R, seed=5)
    a0, beta = O.alpha_beta(g, eta=1.0, method="wigner")
    alpha = np.full(iters, a0)
    P = O.Problem(g)
    h = N.ising_create(N.Problem(g))
    traj = np.empty((R, iters + 1, g.n), np.float32)   # replica-major copy of x^(0..N)
    try:
        ga, gx, loss, ze = _gpu_backward(h, x0, alpha, beta, iters, ckpt)
        x = torch.from_numpy(x0.copy()).cuda()
        traj[:, 0, :] = x0.T
        for k in range(iters):
            N.ising_iterate(h, x, [a0], [beta], 1)
            traj[:, k + 1, :] = x.cpu().numpy().T
        x_all = torch.from_numpy(x0.copy()).cuda()
        N.ising_iterate(h, x_all, [a0], [beta], iters)
        assert np.array_equal(x_all.cpu().numpy().T, traj[:, iters, :])
    finally:
        N.ising_destroy(h)
    for k in (0, 1, 50, iters - 1):                   # steps of the device trajectory are steps of T
        xk = np.ascontiguousarray(traj[:, k, :].T, dtype=np.float64)
        ref = O.doch(P, xk, a0, beta, 1)
        got = traj[:, k + 1, :].T.astype(np.float64)
        rel = np.linalg.norm(got - ref, axis=0) / np.linalg.norm(ref, axis=0)
        assert rel.max() <= 1e-6, (k, rel.max())
    ga_r = np.zeros(iters)
    gx_r = np.empty((g.n, R))
    loss_r, z_r = 0.0, 0
    for r in range(R):
        g_a, gx_r[:, r], l_r, z = O.adjoint_along_replica(P, traj[r], alpha, beta, R)
        ga_r += g_a
        loss_r += l_r
        z_r += z
    assert ze == z_r
    assert loss == pytest.approx(loss_r, rel=1e-6)
    assert _rel(ga, ga_r) <= 1e-3 and np.abs(ga - ga_r).max() <= 1e-3 * np.abs(ga_r).max()
    rel_r = np.linalg.norm(gx - gx_r, axis=0) / np.linalg.norm(gx_r, axis=0)
    assert rel_r.max() <= 1e-3, rel_r.max()
