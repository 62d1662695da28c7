"""Trace-rule runs that max_iter ends: the density is the last iterate."""
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


@pytest.mark.parametrize("iters", [1, 3, 16, 17])
@pytest.mark.parametrize("n", [200, 3200])
@pytest.mark.parametrize("host_schedule", [0, 1])
def test_density_of_a_run_cut_short(P, iters, n, host_schedule):
    F, h = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=n // 3, gap=1e-3, scheme="TC_MONO", instance=n, config=115))
    out = []
    for kw in ({"precision": "fp64"}, {"precision": "mixed", "host_schedule": host_schedule}):
        with P.Purifier(branch_rule="trace", **kw) as pur:
            # a density of the same handle before it
            pur.set_hamiltonian(F, nocc=h.nocc, lmin=-1.5, lmax=1.5, homo=h.homo, lumo=h.lumo)
            pur.run("TC_MONO", 1e-9, 2, check=False)
            pur.set_hamiltonian(F, nocc=h.nocc, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
            assert pur.run("TC_MONO", 1e-9, iters, check=False) == P.ERR_NOT_CONVERGED
            assert pur.stats()["iterations"] == iters
            out.append(pur.density())
    # the mixed path's bound
    assert np.max(np.abs(out[0] - out[1])) <= 1e-6
