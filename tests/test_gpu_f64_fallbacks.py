"""Float64 products that change from digits to the FMA kernel on the way, and the
digits' largest sizes."""
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


def _ones_run(P, n, iters, refine):
    # X_0 = 0.4 J (J: all ones) with ends that do not enclose the spectrum: each
    # step about squares the one eigenvalue, 0.4 n at first
    F = torch.eye(n, dtype=torch.float64, device="cuda") - 0.8
    with P.Purifier(precision="mixed", refine_fp64=refine) as pur:
        pur.set_hamiltonian(F, nocc=n // 10, lmin=-1.0, lmax=1.0, homo=0.1, lumo=0.2)
        pur.run("TC_MONO", 1e-9, iters, check=False)
        return torch.from_numpy(pur.density()).cuda(), pur.stats()


# The two refinement steps X <- 3 X^2 - 2 X^3 take the row scale 2^100 to 2^300 and
# their second square to 2^600: the first step is made of digits, the second one
# has an operand that they cannot hold and is made again.
@pytest.mark.parametrize("n", [200, 300])
def test_refinement_goes_on_with_the_fma_kernel(P, n):
    X, st0 = _ones_run(P, n, 4, 0)
    scale = float(X.abs().max()) * n ** 0.5
    assert 2.0 ** 70 < scale < 2.0 ** 130
    D, st = _ones_run(P, n, 4, 2)
    S, Y = torch.empty_like(X), torch.empty_like(X)
    for _ in range(2):
        P.k_step_f64(X, X, X, S, 1.0, 0.0, 0.0)
        P.k_step_f64(S, X, S, Y, -2.0, 3.0, 0.0)
        X, Y = Y, X
    # entries of one sign: products are exact to n 2^-53 relative, twice cubed
    assert bool(torch.isfinite(X).all()) and float((D / X - 1.0).abs().max()) <= 20 * n * 2.0 ** -53
    assert st["refine_multiplications"] == 4
    # three of the four products were made of digits: 43 pairs each
    t = (n + 127) // 128
    assert st["tensor_flops"] - st0["tensor_flops"] == 3 * 43 * (t * (t + 1) // 2) * 2.0 * 128 * 128 * 128 * t


def test_gap_estimate_of_a_diverging_iterate(P):
    h = I.dense_hamiltonian(200, 80, 0.1, config=116)
    with P.Purifier() as pur:
        # ends that do not enclose the spectrum: the iterate leaves the digits' range
        pur.set_hamiltonian(3.0 * h.F, nocc=80, lmin=-1.0, lmax=1.0)
        with pytest.raises(P.PurifyError) as e:
            pur.estimate_gap()
        assert e.value.code == P.ERR_NOT_CONVERGED
        # the handle goes on
        pur.set_hamiltonian(h.F, nocc=80, lmin=h.lmin, lmax=h.lmax)
        ho, lu = pur.estimate_gap()
        assert h.homo <= ho < lu <= h.lumo
        assert pur.run("TC_SF", 1e-12) == P.OK


# beyond 4096 columns the split reads its rows again instead of holding them
@pytest.mark.parametrize("n", [4097, 4610])
def test_rows_longer_than_the_registers_hold(P, n):
    F, h = I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=n // 2, gap=0.1, scheme="TC_MONO", instance=n, config=117))
    s = P.schedule("TC_MONO", h.lmin, h.lmax, 0.0, h.homo, h.lumo, 1e-12, 1)
    w = h.lmax - h.lmin
    X = F * (-1.0 / w) + torch.eye(n, dtype=torch.float64, device="cuda") * (h.lmax / w)
    Y = torch.empty_like(X)
    b = s["branch"][0]
    P.k_step_f64(X, X, X, Y, 1.0 if b else -1.0, 0.0 if b else 2.0, 0.0)
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
        pur.run("TC_MONO", 1e-12, 1)
        D = torch.empty_like(X)
        pur.density(D)
        st = pur.stats()
    assert bool((D == D.T).all())
    # rows of 2-norm <= 1; the FMA chain's own bound, n 2^-53, is the larger part
    assert float((D - Y).abs().max()) <= n * 2.0 ** -53
    assert st["tensor_flops"] > 0.0
