"""Device memory that handles and batches hold between calls."""
import pytest

from paper_1101_0265_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MiB = 1 << 20


@pytest.fixture(scope="module")
def P():
    from paper_1101_0265_gb300 import build
    build.build()
    import paper_1101_0265_gb300 as P
    return P


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _mixed_run(P, n):
    h = I.dense_hamiltonian(n, n // 2, 0.05, config=109)
    pur = P.Purifier(precision="mixed")
    pur.set_hamiltonian(h.F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
    pur.run("TC_SF", 1e-9)
    return pur


def test_a_small_mixed_handle_holds_sums_of_its_own_size(P):
    _mixed_run(P, 64).close()  # what the process allocates once
    before = _free()
    pur = _mixed_run(P, 64)
    held = before - _free()
    pur.close()
    # 60 MB of product scratch for every SM, the matrices and planes of one tile
    assert held <= 80 * MiB, held / MiB


def test_growing_sizes_on_one_handle(P):
    # the sums grow with the handle's largest size; every size gives its own density
    ref = {}
    for n in (64, 300, 900, 2000):
        pur = _mixed_run(P, n)
        ref[n] = pur.density()
        pur.close()
    with P.Purifier(precision="mixed") as pur:
        for n in (300, 64, 900, 300, 2000, 64):
            h = I.dense_hamiltonian(n, n // 2, 0.05, config=109)
            pur.set_hamiltonian(h.F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
            pur.run("TC_SF", 1e-9)
            assert (pur.density() == ref[n]).all()


def test_trace_rule_graphs_follow_grown_sums(P):
    with P.Purifier(precision="mixed", branch_rule="trace") as pur:
        out = []
        for n in (300, 900, 300):
            h = I.dense_hamiltonian(n, n // 2, 0.05, config=110)
            pur.set_hamiltonian(h.F, nocc=h.nocc, lmin=h.lmin, lmax=h.lmax)
            pur.run("TC_MONO", 1e-4)
            out.append(pur.density())
        assert (out[0] == out[2]).all()


def test_large_float64_workspaces_are_given_back(P):
    n = 8192
    F, h = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=n // 2, gap=0.1, scheme="TC_SF", instance=1, config=111))
    before = _free()
    with P.Purifier() as pur:
        pur.set_hamiltonian(F, nocc=h.nocc, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)
        pur.run("TC_SF", 1e-12, 2)
        held = before - _free()
    # F, two iterates and the product buffer; digits and sums of this size (1.3 GiB) are given back
    assert held <= 4 * 8 * n * n + 64 * MiB, held / MiB


def test_rounds_of_a_batch_do_not_add_up(P):
    n = 8192
    F, h = I.reflected_hamiltonian_device(I.InstanceSpec(n=n, nocc=n // 2, gap=0.1, scheme="TC_SF", instance=1, config=112))
    B = P.Batch()
    before = _free()

    def add():
        return [B.add(F, h.nocc, h.lmin, h.lmax, h.homo, h.lumo, scheme="TC_SF", tol=1e-9, mu=0.0) for _ in range(2)]

    ids = add()
    most = before - _free()
    assert most >= B.bytes_in_use()
    for _ in range(3):
        for i in ids:
            B.release(i)
        assert B.bytes_in_use() == 0 and before - _free() <= most
        ids = add()
        assert before - _free() <= most + 64 * MiB
    B.close()
    assert before - _free() <= 64 * MiB
