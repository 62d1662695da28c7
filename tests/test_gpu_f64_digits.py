"""Float64 runs whose products are exact digit products on the tensor cores,
against extended precision, the float64 FMA kernel and themselves."""
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


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _set(pur, F, h):
    pur.set_hamiltonian(F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)


# the FMA kernel's sizes and the smallest one of the digits (160), tile edges and
# remainders, the split's row boundaries (512, 1024), one wave of tiles (2176 =
# 17 x 128: 153 tiles) and beyond
@pytest.mark.parametrize("n", [3, 15, 16, 17, 128, 129, 159, 160, 161, 255, 256, 257, 512, 513, 640, 1023, 1024, 1025, 1153, 2177])
def test_one_step_against_extended_precision(P, n):
    F, h = I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=max(1, n // 3), gap=0.05, scheme="TC_MONO", instance=n, config=91))
    with P.Purifier() as pur:
        _set(pur, F, h)
        pur.run("TC_MONO", 1e-12, 0)
        X = pur.density()
        pur.run("TC_MONO", 1e-12, 1)
        Y = pur.density()
        pur.run("TC_MONO", 1e-12, 1)
        assert np.array_equal(pur.density(), Y)
    assert np.array_equal(Y, Y.T)
    # nocc < n / 2: the first branch is P_{1,0}, Y = X^2.  Rows have 2-norms
    # <= 1: digits leave out less than 2^-56, the rounding of P and of the
    # polynomial's two operations is at most 3 x 2^-53
    rows = np.unique(np.linspace(0, n - 1, 9).astype(int))
    XL = X.astype(np.longdouble)
    S = np.stack([(XL * XL[i][None, :]).sum(axis=1) for i in rows])
    b = P.schedule("TC_MONO", h.lmin, h.lmax, 0.0, h.homo, h.lumo, 1e-12, 1)["branch"][0]
    R = S if b else 2 * XL[rows] - S
    assert float(np.max(np.abs(Y[rows] - R))) <= 4 * 2.0 ** -53


def _fma_run(P, F, h, scheme, iters):
    """The same recursion through the float64 FMA kernel's own entry point."""
    s = P.schedule(scheme, h.lmin, h.lmax, 0.0, h.homo, h.lumo, 1e-12, iters)
    eye = torch.eye(h.n, dtype=torch.float64, device="cuda")
    X, S = torch.empty_like(F), torch.empty_like(F)
    if scheme.startswith("TC"):
        w = h.lmax - h.lmin
        X = F * (-1.0 / w) + eye * (h.lmax / w)
        for b, a in zip(s["branch"], s["alpha"]):
            c = ((1 + a) ** 2, -2 * a * (1 + a), a * a) if b else (-(1 + a) ** 2, 2 * (1 + a), 0.0)
            P.k_step_f64(X, X, X, S, *c)
            X, S = S, X
        return X
    g = 2.0 * max(h.lmax, -h.lmin)
    al = list(s["alpha"]) + [1.0]
    X = F * (-al[0] / g) + eye * 0.5
    Y = torch.empty_like(F)
    for k in range(s["iterations"]):
        P.k_step_f64(X, X, None, S, 1.0, 0.0, 0.0)
        P.k_step_f64(S, X, S, Y, -2.0, 3.0, 0.0, al[k + 1], 0.5 * (1.0 - al[k + 1]))
        X, Y = Y, X
    return X


@pytest.mark.parametrize("n,scheme", [(128, "TC_SF"), (300, "FIXED_MU_SF"), (1100, "FIXED_MU_SF"), (1300, "TC_SF")])
def test_run_against_the_fma_kernel(P, n, scheme):
    F, h = I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=n // 2, gap=0.02, scheme=scheme, instance=n, config=92))
    with P.Purifier() as pur:
        _set(pur, F, h)
        assert pur.run(scheme, 1e-12) == P.OK
        D = _cuda(pur.density())
    # both within float64 rounding (amplified by 1 / mapped gap) of the exact density
    assert float((D - _fma_run(P, F, h, scheme, 200)).abs().max()) <= 1e-12


def _bits(t):
    return t.contiguous().view(torch.int64)


@pytest.mark.parametrize("scheme", ["TC_MONO", "FIXED_MU_MONO"])
@pytest.mark.parametrize("what", ["nan", "inf", "diverging"])
def test_values_outside_the_digits_take_the_fma_kernel(P, scheme, what):
    # an operand that digits cannot hold: the run is the FMA kernel's
    n, iters = 200, 14
    F, h = I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=100, gap=0.2, scheme=scheme, instance=3, config=93))
    if what == "diverging":
        F *= 3.0  # the spectrum leaves [lmin, lmax]: iterates grow past 2^400, then overflow
    else:
        F[7, 11] = F[11, 7] = float(what)
    with P.Purifier() as pur:
        _set(pur, F, h)
        assert pur.run(scheme, 1e-12, iters, check=False) in (P.ERR_BOUNDS, P.ERR_NOT_CONVERGED)
        D = _cuda(pur.density())
        ref = _fma_run(P, F, h, scheme, iters)
        assert not bool(torch.isfinite(ref).all())
        assert torch.equal(torch.isnan(D), torch.isnan(ref)) and torch.equal(torch.isinf(D), torch.isinf(ref))
        # the handle goes on: a sound input on the same handle
        F2, h2 = I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=80, gap=0.2, scheme=scheme, instance=4, config=93))
        _set(pur, F2, h2)
        assert pur.run(scheme, 1e-12) == P.OK
        assert abs(pur.stats()["trace"] - 80) < 1e-9
