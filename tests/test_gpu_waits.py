"""Bounded device waits outside the mixed products: the float64 products'
report a time-out and leave the handle usable, the grid barriers' lead to the
step-by-step launches with the same coefficients."""
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


def _set(pur, h):
    pur.set_hamiltonian(h.F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)


# 1000 cycles are far below one stage's copies and MMAs: the first wait gives up
@pytest.mark.parametrize("scheme,n", [("TC_SF", 256), ("FIXED_MU_SF", 600), ("TC_SF", 1300)])
def test_short_waits_in_a_float64_run(P, scheme, n):
    h = I.dense_hamiltonian(n, n // 2, 0.05, config=105)
    with P.Purifier() as pur:
        _set(pur, h)
        assert pur.run(scheme, 1e-12) == P.OK
        ref = pur.density()
        pur.set_options(wait_kcycles=1)
        assert pur.run(scheme, 1e-12, check=False) == P.ERR_DEVICE_TIMEOUT
        assert pur.stats()["device_flag"] == 32
        with pytest.raises(P.PurifyError) as e:
            pur.estimate_gap()
        assert e.value.code == P.ERR_DEVICE_TIMEOUT
        torch.cuda.synchronize()  # the context is intact
        # sums that were left behind are gone: the same density as before
        pur.set_options(wait_kcycles=0)
        assert pur.run(scheme, 1e-12) == P.OK
        assert pur.stats()["device_flag"] == 0
        assert np.array_equal(pur.density(), ref)


# a barrier that gives up (blocks of another stream's kernel may hold SMs for
# long) costs time, not the call
@pytest.mark.parametrize("n", [130, 1000, 2500])
def test_bounds_when_the_barrier_gives_up(P, n):
    F, h = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=n // 2, gap=0.1, scheme="TC_SF", instance=n, config=106))
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=h.nocc)
        a = pur.stats()
        pur.set_options(wait_kcycles=1)
        pur.set_hamiltonian(F, nocc=h.nocc)
        b = pur.stats()
    assert (a["lmin"], a["lmax"]) == (b["lmin"], b["lmax"])
    assert b["kernel_launches"] > a["kernel_launches"]  # step by step


# below n = 160 the float64 steps wait for nothing: only the filters' barrier does
@pytest.mark.parametrize("n", [60, 150])
def test_gap_when_the_barrier_gives_up(P, n):
    F, h = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=2 * n // 5, gap=0.06, scheme="TC_SF", instance=n, config=107))
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=h.nocc, lmin=h.lmin, lmax=h.lmax)
        ref = pur.estimate_gap()
        pur.set_options(wait_kcycles=1)
        assert pur.estimate_gap() == ref
        assert h.homo <= ref[0] < ref[1] <= h.lumo
