"""Lanczos kernels that run all steps in one launch, at the edges of their ranges."""
import numpy as np
import pytest

from oracle import purify_oracle as O
from paper_1101_0265_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    from paper_1101_0265_gb300 import build
    build.build()
    import paper_1101_0265_gb300 as P
    return P


# fewer rows than a block's warps, partial groups of rows and columns, one row per
# block more than a round of warps takes (152 x 32 = 4864), the largest
# one-launch size and the first beyond it (one launch per step)
@pytest.mark.parametrize("n,k", [(2, 2), (5, 5), (31, 8), (127, 16), (129, 16), (257, 24), (1025, 16), (4900, 8),
                                 (8192, 4), (8193, 4)])
def test_bound_steps_against_the_oracle(P, n, k):
    F, _ = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=max(1, n // 2) if n < 4 else n // 2, gap=0.1,
                                                         scheme="TC_SF", instance=n, config=98))
    a, b = P.k_lanczos_f64(F, k)
    ao, bo = O.lanczos(F.cpu().numpy(), k, O.lanczos_start(n))
    # (n = k: the last residual is rounding)
    m = k if n > k else k - 1
    assert np.max(np.abs(a - ao)) < 1e-9 and np.max(np.abs(b[:m] - bo[:m]), initial=0.0) < 1e-9
    a2, b2 = P.k_lanczos_f64(F, k)
    assert np.array_equal(a, a2) and np.array_equal(b, b2)


# rows of X in shared memory (up to about 1850 on 152 SMs) and not
@pytest.mark.parametrize("n", [40, 153, 1840, 1900, 2500])
def test_gap_edges(P, n):
    F, h = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=2 * n // 5, gap=0.06, scheme="TC_SF", instance=n,
                                                         config=99))
    with P.Purifier(precision="mixed") as pur:
        pur.set_hamiltonian(F, nocc=h.nocc)
        ho, lu = pur.estimate_gap()
        # inner estimates (how tight they are is the 40 steps' residuals)
        assert h.homo <= ho < lu <= h.lumo
        assert pur.estimate_gap() == (ho, lu)
        assert pur.run("TC_SF", 1e-9) == P.OK  # (checks the trace against nocc)
