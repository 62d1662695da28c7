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


def _set(pur, h, F=None):
    pur.set_hamiltonian(h.F if F is None else F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)


@pytest.mark.parametrize("n", [100, 159, 160, 300])
@pytest.mark.parametrize("scheme", ["TC_SF", "FIXED_MU_SF"])
def test_tensor_flops_of_float64_runs(P, n, scheme):
    h = I.dense_hamiltonian(n, n // 2, 0.1, config=113)
    with P.Purifier() as pur:
        _set(pur, h)
        assert pur.run(scheme, 1e-12) == P.OK
        st = pur.stats()
        t = (n + 127) // 128
        pairs = st["multiplications"] * (t * (t + 1) // 2) * 2.0 * 128 * 128 * 128 * t
        assert st["tensor_flops"] == (43 * pairs if n >= 160 else 0.0)
        F = h.F.copy()
        F[3, 4] = F[4, 3] = float("nan")  # the FMA kernel's run
        _set(pur, h, F)
        pur.run(scheme, 1e-12, check=False)
        assert pur.stats()["tensor_flops"] == 0.0


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
