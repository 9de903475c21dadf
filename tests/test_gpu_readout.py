"""Energy readout at the sizes where its layout can go wrong: replica counts that take the
16-byte loads and those that do not, arrays that are not 16-byte aligned, rows shorter and
longer than one batch of entries, one-row and odd lattices, batches with tiny instances.

Integer energies and cuts are exact; FP64 ones within 1e-12 relative of the oracle (a sum of
at most 2e5 terms in FP64: 2e5 * 2^-53 = 2e-11 in the worst case, its square root typically).
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
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.build_library()
    return N.load()


def _shifted(a, skip):
    """A device copy of `a` that starts `skip` elements into its allocation."""
    t = torch.from_numpy(np.ascontiguousarray(a))
    buf = torch.empty(t.numel() + skip, dtype=t.dtype, device="cuda")
    view = buf[skip:].reshape(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("R", [1, 2, 3, 4, 20, 300, 1028])
@pytest.mark.parametrize("kind", ["torus", "torus_odd", "er", "hub"])
def test_integer_energies(kind, R):
    J = {"torus": lambda: I.torus_pm1(6, 8, seed=1), "torus_odd": lambda: I.torus_pm1(2, 517, seed=2),
         "er": lambda: I.erdos_renyi_pm1(97, 0.3, seed=3), "hub": lambda: short_rows_mixed(530, seed=4)}[kind]()
    x = I.x0_uniform(J.n, R, seed=5)
    x[::31] = -0.0
    s = O.sign(x.astype(np.float64))
    Er, cr = O.energy_int(O.Problem(J), s)
    h = N.ising_create(N.Problem(J))
    try:
        for dt, skip in ((np.float32, 0), (np.float32, 1), (np.float64, 0), (np.float64, 1), (np.int8, 0), (np.int8, 1)):
            xin = _shifted(s.astype(np.int8) if dt == np.int8 else x.astype(dt), skip)
            E, cut = torch.zeros(R, dtype=torch.int64, device="cuda"), torch.zeros(R, dtype=torch.int64, device="cuda")
            N.ising_energy(h, xin, E_int=E, cut_int=cut)
            assert np.array_equal(E.cpu().numpy(), Er) and np.array_equal(cut.cpu().numpy(), cr)
    finally:
        N.ising_destroy(h)


@pytest.mark.parametrize("R", [1, 6, 16])
def test_real_energies_of_uneven_instances(R):
    sizes, degs = [6, 1000, 64, 8], [2, 12, 9, 2]
    gs = [I.regular_gauss(n, d, seed=10 + n) for n, d in zip(sizes, degs)]
    hs = [I.field_gauss(n, 0.1, seed=20 + n) for n in sizes]
    off = np.cumsum([0] + sizes).astype(np.int64)
    nz = np.cumsum([0] + [g.nnz for g in gs])
    J = I.CSR(off[-1], np.concatenate([[0]] + [g.row_ptr[1:] + z for g, z in zip(gs, nz[:-1])]),
              np.concatenate([g.col + o for g, o in zip(gs, off[:-1])]).astype(np.int32),
              np.concatenate([g.val for g in gs]).astype(np.float32))
    J.val[np.abs(J.val) < 1e-3] = 1e-40  # subnormal couplings take the conversion
    x = I.x0_uniform(int(off[-1]), R, seed=30)
    h = N.ising_create(N.Problem(J, np.concatenate(hs), off), N.FLAG_SKIP_VALIDATION)
    try:
        E, cut = np.zeros((4, R)), np.zeros((4, R))
        N.ising_energy(h, _shifted(x, 0), E_f64=E, cut_f64=cut)
    finally:
        N.ising_destroy(h)
    for b in range(4):
        g = I.CSR(sizes[b], gs[b].row_ptr, gs[b].col, J.val[nz[b]:nz[b + 1]].astype(np.float64))
        Er, cr = O.energy(O.Problem(g, hs[b]), O.sign(x[off[b]:off[b + 1]].astype(np.float64)))
        scale = np.abs(g.val).sum() + np.abs(hs[b]).sum()
        np.testing.assert_allclose(E[b], Er, rtol=0, atol=1e-12 * scale)
        np.testing.assert_allclose(cut[b], cr, rtol=0, atol=1e-12 * scale)


def test_all_satisfied_and_infinite_couplings():
    """Aligned spins on positive couplings cut nothing (exactly 0); an infinite coupling (accepted
    without validation) gives an infinite energy."""
    g = I.regular_gauss(40, 3, seed=7)
    g.val = np.abs(g.val)
    for inf in (False, True):
        if inf:
            g.val[0] = np.inf
        h = N.ising_create(N.Problem(g), N.FLAG_SKIP_VALIDATION)
        try:
            E, cut = np.zeros(4), np.zeros(4)
            N.ising_energy(h, np.ones((40, 4), np.float32), E_f64=E, cut_f64=cut)
        finally:
            N.ising_destroy(h)
        if inf:
            assert np.all(np.isneginf(E))
        else:
            assert np.all(cut == 0.0)
