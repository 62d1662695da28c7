"""Statistics that tell which kernels a run took."""
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


def test_launches_of_a_replayed_trace_run(P):
    h = I.dense_hamiltonian(300, 120, 0.1, config=114)
    with P.Purifier(precision="mixed", branch_rule="trace") as pur:
        pur.set_hamiltonian(h.F, nocc=h.nocc, lmin=h.lmin, lmax=h.lmax)
        pur.run("TC_MONO", 1e-4)
        first = pur.stats()
        pur.run("TC_MONO", 1e-4)  # the graph again
        second = pur.stats()
    # per step the schedule's kernel, a product and its finish; per block of 16 one more schedule kernel
    blocks = -(-first["iterations"] // 16)
    least = blocks * (16 * 3 + 1)
    assert least <= second["kernel_launches"] <= least + 4
    assert first["kernel_launches"] == second["kernel_launches"]
