"""A batch's instances share a memory pool: freed memory serves the next ones."""
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


def test_memory_of_released_instances_is_used_again(P):
    hs = [I.dense_hamiltonian(n, n // 2, 0.05, config=97, instance=n) for n in (64, 129, 300, 511)]
    kinds = ("TC_SF", "FIXED_MU_SF", "TC_SF", "FIXED_MU_SF")

    def add(B, k):
        h = hs[k]
        return B.add(h.F, h.nocc, h.lmin, h.lmax, h.homo, h.lumo, scheme=kinds[k], tol=1e-9, mu=0.0)

    ref = []
    for k in range(len(hs)):  # each in a batch of its own
        B = P.Batch()
        i = add(B, k)
        B.run()
        ref.append(B.density(i))
        B.close()
    B = P.Batch()
    for order in ((0, 1, 2, 3), (3, 1, 0, 2), (2, 2, 0, 3, 1)):
        ids = [(add(B, k), k) for k in order]
        B.run()
        for i, k in ids:
            assert np.array_equal(B.density(i), ref[k])
            B.release(i)
        assert B.bytes_in_use() == 0
    # an instance released while it runs, its memory taken by the next one
    a, b = add(B, 3), add(B, 1)
    B.advance(1)
    B.release(a)
    c = add(B, 3)
    while not (B.done(b) and B.done(c)):
        B.advance(2)
    assert np.array_equal(B.density(b), ref[1]) and np.array_equal(B.density(c), ref[3])
    B.close()
