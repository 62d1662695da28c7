"""Small mixed products (sums to memory, separate finish pass): the same
densities as the persistent kernel's, at the edges of tiles and waves."""
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


def _input(n, scheme, config):
    return I.dense_hamiltonian_device(I.InstanceSpec(n=n, nocc=max(1, n // 3), gap=0.02, scheme=scheme, instance=n,
                                                     config=config), keep_q=True)


def _set(pur, F, h):
    pur.set_hamiltonian(F, nocc=h.nocc, mu=0.0, lmin=h.lmin, lmax=h.lmax, homo=h.homo, lumo=h.lumo)


# one tile, tile edges, a part of a block, 12 tile columns (one band) and one
# more, one wave of tiles less and more (17 x 18 / 2 = 153), nearly two waves
@pytest.mark.parametrize("n,digits", [(n, 0) for n in (3, 127, 128, 129, 300, 1536, 1537, 2048, 2049, 2177, 2944)]
                         + [(n, d) for n in (3, 129, 300) for d in (2, 3, 4)])
def test_whole_tiles_equal_the_queue_kernel(P, n, digits):
    # a batch runs on the persistent queue kernel: the same bits
    for scheme in ("TC_SF", "FIXED_MU_SF"):
        F, h = _input(n, scheme, 94)
        B = P.Batch(digits=digits)
        i = B.add(F, h.nocc, h.lmin, h.lmax, h.homo, h.lumo, scheme=scheme, tol=1e-9, mu=0.0)
        B.run(use_graph=False)
        ref = B.density(i)
        B.close()
        with P.Purifier(precision="mixed", split_k=False, digits=digits) as pur:
            _set(pur, F, h)
            pur.run(scheme, 1e-9)
            assert np.array_equal(pur.density(), ref)
            pur.run(scheme, 1e-9)  # the buffers of the first run again
            assert np.array_equal(pur.density(), ref)


# parts of the last wave: 4 ways (n = 1000), 2 and 3 ways, one split tile after a full wave
@pytest.mark.parametrize("n", [200, 600, 1000, 1101, 1300, 2177])
def test_split_tiles(P, n):
    F, h = _input(n, "TC_SF", 95)
    D = h.Q[:, :h.nocc] @ h.Q[:, :h.nocc].T
    with P.Purifier(precision="mixed") as pur:
        _set(pur, F, h)
        pur.run("TC_SF", 1e-9)
        X = torch.from_numpy(pur.density()).cuda()
        assert float((X - D).abs().max()) <= 1e-6  # the mixed path's bound
        assert bool((X == X.T).all())
        tr, idem = pur.step_history()
        assert abs(tr[-1] - h.nocc) <= 1e-5
        # other sizes between: tiles that were split are whole now, and back
        F2, h2 = _input(n + 700, "TC_SF", 95)
        _set(pur, F2, h2)
        pur.run("TC_SF", 1e-9)
        _set(pur, F, h)
        pur.run("TC_SF", 1e-9)
        assert torch.equal(torch.from_numpy(pur.density()).cuda(), X)


@pytest.mark.parametrize("scheme", ["TC_SF", "FIXED_MU_SF"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_not_finite_input_gives_no_density(P, scheme, value):
    F, h = _input(300, scheme, 96)
    Fb = F.clone()
    Fb[5, 9] = Fb[9, 5] = value
    with P.Purifier(precision="mixed") as pur:
        _set(pur, Fb, h)
        assert pur.run(scheme, 1e-9, check=False) == P.ERR_BOUNDS
        assert np.isnan(pur.density()).all()
        _set(pur, F, h)
        assert pur.run(scheme, 1e-9) == P.OK
        assert abs(pur.stats()["trace"] - h.nocc) <= 1e-5
