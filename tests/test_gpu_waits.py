"""Bounded device waits outside the mixed products: a wait of a float64 product
that runs out is reported and leaves the handle usable."""
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
