"""Float64 runs at the ends of what digit planes can hold: rows that underflow
stay on the tensor cores, and a density with entries far below their rows' norms
(decaying or weakly coupled matrices) has them as precise as the FMA kernel gives
them."""
import numpy as np
import pytest

from paper_1101_0265_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    from paper_1101_0265_gb300 import build
    build.build()
    import paper_1101_0265_gb300 as P
    return P


def _fma_run(P, F, lmin, lmax, homo, lumo, scheme):
    """The same recursion through the float64 FMA kernel's own entry point."""
    s = P.schedule(scheme, lmin, lmax, 0.0, homo, lumo, 1e-12, 200)
    eye = torch.eye(F.shape[0], dtype=torch.float64, device="cuda")
    w = lmax - lmin
    X = F * (-1.0 / w) + eye * (lmax / w)
    S = torch.empty_like(X)
    for b, a in zip(s["branch"], s["alpha"]):
        c = ((1 + a) ** 2, -2 * a * (1 + a), a * a) if b else (-(1 + a) ** 2, 2 * (1 + a), 0.0)
        P.k_step_f64(X, X, X, S, *c)
        X, S = S, X
    return X


def _block_diagonal(*blocks):
    n = sum(b.shape[0] for b in blocks)
    F, at = np.zeros((n, n)), 0
    for b in blocks:
        F[at:at + b.shape[0], at:at + b.shape[0]] = b
        at += b.shape[0]
    return F


def _virtual_block(m, seed):
    r = np.random.default_rng(seed)
    Q = np.linalg.qr(r.standard_normal((m, m)))[0]
    B = (Q * np.linspace(0.6, 0.95, m)) @ Q.T
    return 0.5 * (B + B.T)


# one decoupled unoccupied orbital, and a block of them: their rows of X are
# squared at each step, in the end far below 2^-400
@pytest.mark.parametrize("block", [1, 40])
@pytest.mark.parametrize("scheme", ["TC_MONO", "TC_SF"])
def test_rows_that_underflow_stay_on_the_tensor_cores(P, block, scheme):
    h = I.dense_hamiltonian(200, 90, 0.1, config=101)
    F = torch.from_numpy(_block_diagonal(h.F, np.array([[0.8]]) if block == 1 else _virtual_block(block, 5))).cuda()
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=h.nocc, mu=0.0, lmin=-1.0, lmax=1.0, homo=h.homo, lumo=h.lumo)
        assert pur.run(scheme, 1e-12) == P.OK
        D = torch.from_numpy(pur.density()).cuda()
        st = pur.stats()
    # three launches a step and a few for the run, not the FMA kernel's run as well
    assert st["kernel_launches"] <= 3 * st["multiplications"] + 5
    ref = _fma_run(P, F, -1.0, 1.0, h.homo, h.lumo, scheme)
    assert float((D - ref).abs().max()) <= 1e-12
    assert not bool(D[:200, 200:].any())  # uncoupled stays uncoupled


def _relative(D, ref, m):
    """Largest relative deviation over the entries of the mask m."""
    return float(((D - ref).abs()[m] / ref.abs()[m]).max())


# A gapped chain of alternating bonds: the density decays by 3 every second site
# (and is zero, up to rounding, between sites an even distance apart).
# A run of the FMA kernel keeps every entry to n u per step relative to its own
# terms: 14 steps x 240 x 2^-53 = 4e-13, raised along the decay; 1e-8 is far
# above that and far below what digits of a fixed point below the row norm leave
# (2^-58 of the norm is 1e-5 of an entry of 3e-13).
@pytest.mark.parametrize("n", [240, 513])
@pytest.mark.parametrize("scheme", ["TC_SF", "TC_MONO"])
def test_decaying_density_keeps_its_small_entries(P, n, scheme):
    n -= n % 2  # strong bonds at both ends: no state in the gap
    t = np.where(np.arange(n - 1) % 2 == 0, 0.6, 0.2)
    F = torch.from_numpy(np.diag(t, 1) + np.diag(t, -1)).cuda()
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=n // 2, mu=0.0, lmin=-0.81, lmax=0.81, homo=-0.4, lumo=0.4)
        assert pur.run(scheme, 1e-12) == P.OK
        D = torch.from_numpy(pur.density()).cuda()
    ref = _fma_run(P, F, -0.81, 0.81, -0.4, 0.4, scheme)
    assert float((D - ref).abs().max()) <= 1e-12
    i = torch.arange(n, device="cuda")
    assert _relative(D, ref, ((i[:, None] - i[None, :]) % 2 != 0) & (ref.abs() > 1e-18)) <= 1e-8


# two dense parts coupled by entries of 1e-10 and 1e-20
@pytest.mark.parametrize("coupling", [1e-10, 1e-20])
def test_weak_coupling_is_kept(P, coupling):
    a, b = I.dense_hamiltonian(150, 70, 0.1, config=102), I.dense_hamiltonian(130, 60, 0.1, config=103)
    C = coupling * np.random.default_rng(6).standard_normal((150, 130))
    F = _block_diagonal(a.F, b.F)
    F[:150, 150:] = C
    F[150:, :150] = C.T
    F = torch.from_numpy(F).cuda()
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=130, mu=0.0, lmin=-1.01, lmax=1.01, homo=-0.05, lumo=0.05)
        assert pur.run("TC_SF", 1e-12) == P.OK
        D = torch.from_numpy(pur.density()).cuda()
    ref = _fma_run(P, F, -1.01, 1.01, -0.05, 0.05, "TC_SF")
    off = ref[:150, 150:]
    # (entries that cancel are left out: below a thousandth of the largest)
    assert _relative(D[:150, 150:], off, off.abs() > 1e-3 * off.abs().max()) <= 1e-8


# rotated spectra of every filling stay on the tensor cores (tile and split edges)
@pytest.mark.parametrize("n,occ", [(160, 0.25), (161, 0.7), (300, 0.5), (513, 0.7), (1025, 0.25)])
@pytest.mark.parametrize("scheme", ["TC_SF", "FIXED_MU_SF"])
def test_dense_runs_stay_on_the_tensor_cores(P, n, occ, scheme):
    F, h = I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=int(occ * n), gap=0.01, scheme=scheme, instance=n, config=104))
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
        assert pur.run(scheme, 1e-12) == P.OK
        st = pur.stats()
    assert st["kernel_launches"] <= 3 * st["multiplications"] + 5
