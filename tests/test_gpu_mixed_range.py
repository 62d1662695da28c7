"""Small mixed products whose sums leave the fixed-point range: spectral ends
that do not enclose the spectrum, and a run cut short while its iterate is
still finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    from paper_1101_0265_gb300 import build
    build.build()
    import paper_1101_0265_gb300 as P
    return P


# X_0 = 0.4 J (J: all ones): X_0^2 has entries 0.16 n, from 32 (n = 200) on; whole
# tiles, split ones, one wave less and more
@pytest.mark.parametrize("n", [200, 300, 600, 1101, 1500, 2177])
@pytest.mark.parametrize("rule", ["beta", "trace"])
def test_products_out_of_range_are_carried(P, n, rule):
    F = torch.eye(n, dtype=torch.float64, device="cuda") - 0.8 * torch.ones((n, n), dtype=torch.float64, device="cuda")
    homo, lumo = 0.1, 0.2
    s = P.schedule("TC_MONO", -1.0, 1.0, None, homo, lumo, 1e-9, 1)
    with P.Purifier(precision="mixed", branch_rule=rule) as pur:
        pur.set_hamiltonian(F, nocc=n // 10, lmin=-1.0, lmax=1.0, homo=homo, lumo=lumo)
        assert pur.run("TC_MONO", 1e-9, 1, check=False) == P.ERR_NOT_CONVERGED
        D = torch.from_numpy(pur.density()).cuda()
        st = pur.stats()
        tr, idem = pur.step_history()
    br = s["branch"][0] if rule == "beta" else (1 if 0.4 * n > n // 10 else 0)
    y = 0.16 * n if br else 0.8 - 0.16 * n
    # digits of 0.4 carry 36 bits or more: relative error n 2^-36 at most
    assert float((D / y - 1.0).abs().max()) <= n * 2.0 ** -36
    assert st["iterations"] == 1 and len(tr) == len(idem) == 1 and st["product_launches"] == 1
    assert tr[0] == pytest.approx(n * y, rel=1e-6) and idem[0] == pytest.approx(n * abs(0.4 - 0.16 * n), rel=1e-5)


def test_the_handle_goes_on(P):
    from paper_1101_0265_gb300 import inputs as I
    h = I.dense_hamiltonian(600, 250, 0.05, config=108)
    with P.Purifier(precision="mixed") as pur:
        pur.set_hamiltonian(h.F, nocc=250, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
        pur.run("TC_SF", 1e-9)
        ref = pur.density()
        F = torch.eye(600, dtype=torch.float64, device="cuda") - 0.8
        pur.set_hamiltonian(F, nocc=60, lmin=-1.0, lmax=1.0, homo=0.1, lumo=0.2)
        assert pur.run("TC_MONO", 1e-9, 1, check=False) == P.ERR_NOT_CONVERGED
        pur.set_hamiltonian(h.F, nocc=250, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
        pur.run("TC_SF", 1e-9)
        assert np.array_equal(pur.density(), ref)
