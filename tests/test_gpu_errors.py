"""Error paths that are tested without faulting the GPU: a bounded device wait that runs out
(the wait-gate hook: a flag that nothing clears) and device allocations that fail (the
allocation-budget hook).  Each returns its status code and leaves the library usable."""
import gc

import numpy as np
import pytest

import oracle
import qed_workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
qed = pytest.importorskip("paper_2403_07042_gb300")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07042_gb300 import build
    build.build()
    yield
    qed.set_alloc_budget(-1)


def _rho0(m, b):
    return torch.from_numpy(oracle.initial_density(m, b)).cuda()


@pytest.mark.parametrize("make", [lambda: W.jch_two_cavities(), lambda: W.hb_shaped()])
def test_wait_gate_times_out_then_model_recovers(make):
    m = make()
    b = oracle.enumerate_basis(m)
    gm = qed.Model(m, precision="split_fp16x2")
    gm.set_wait_gate(True, budget_cycles=20000)
    rho = _rho0(m, b)
    gm.evolve(rho, 6)
    with pytest.raises(qed.QedError) as ei:
        gm.sync()
    assert ei.value.status == qed.QED_ETIMEOUT
    # the flag stays reported once: the next check is clean
    gm.sync()
    gm.set_wait_gate(False)
    rho = _rho0(m, b)
    rec = gm.evolve(rho, 200, record_every=50, obs_ids=list(range(b.dim)))
    gm.sync()
    rho_ref, rec_ref = oracle.evolve(m, n_steps=200, record_every=50, basis=b, obs_ids=list(range(b.dim)))
    assert np.abs(rho.cpu().numpy() - rho_ref).max() <= 1e-5
    assert np.abs(rec.cpu().numpy() - rec_ref).max() <= 1e-6


def test_wait_gate_rejected_on_fp64():
    gm = qed.Model(W.jch_two_cavities(), precision="fp64")
    with pytest.raises(qed.QedError) as ei:
        gm.set_wait_gate(True)
    assert ei.value.status == qed.QED_EUNSUPPORTED


@pytest.mark.parametrize("precision", ["fp64", "split_fp16x2"])
def test_alloc_budget_gives_enomem_and_frees(precision):
    m = W.hb_shaped()
    qed.Model(m, precision=precision).close()  # warm-up: modules loaded, pools settled
    gc.collect()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for budget in (0, 1 << 20, 8 << 20):
        qed.set_alloc_budget(budget)
        with pytest.raises(qed.QedError) as ei:
            qed.Model(m, precision=precision)
        assert ei.value.status == qed.QED_ENOMEM
    qed.set_alloc_budget(-1)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free0  # the failed builds freed what they had
    gm = qed.Model(m, precision=precision)
    b = oracle.enumerate_basis(m)
    rho = _rho0(m, b)
    gm.evolve(rho, 20)
    gm.sync()
    rho_ref = oracle.evolve(m, n_steps=20, basis=b, return_records=False)
    assert np.abs(rho.cpu().numpy() - rho_ref).max() <= (1e-12 if precision == "fp64" else 1e-5)


def test_alloc_budget_in_the_adjoint():
    m = W.jc_single(n_max=3, g=0.02, dt=0.1, n_steps=40)
    gm = qed.Model(m, precision="split_fp16x2")
    b = oracle.enumerate_basis(m)
    w = torch.ones(b.dim, dtype=torch.float64, device="cuda")
    qed.set_alloc_budget(0)
    with pytest.raises(qed.QedError) as ei:
        gm.adjoint(_rho0(m, b), 40, w, checkpoint_every=10)
    assert ei.value.status == qed.QED_ENOMEM
    qed.set_alloc_budget(-1)
    loss, *_ = gm.adjoint(_rho0(m, b), 40, w, checkpoint_every=10)
    assert abs(float(loss) - 1.0) <= 1e-6  # the trace of a closed unit-trace evolution


def _same(model, rho0, rho_ref, u_ref):
    rho = rho0.clone()
    model.evolve(rho, 20)
    model.sync()
    return torch.equal(rho, rho_ref) and torch.equal(model.get_U(), u_ref)


@pytest.mark.parametrize("precision,dim", [("fp64", 8), ("fp64", 36), ("fp64", 70), ("fp64", 130),
                                           ("split_fp16x2", 130)])
@pytest.mark.parametrize("change", ["effective", "lie", "U"])
def test_failed_propagator_change_leaves_the_model_as_it_was(precision, dim, change):
    """set_scheme and set_U that run out of memory at any of their allocations: the model steps on
    with its old scheme and propagator, equal to the bit, and the repeated call takes effect."""
    m = {8: lambda: W.jc_single(n_max=3, g=0.02, dt=0.1, gamma=1e-3), 36: W.jch_two_cavities}.get(
        dim, lambda: W.chain_instance(np.random.default_rng(dim), dim, dim))()
    before, after = ("effective", "lie") if change == "lie" else ("lie", change)
    gm, ref = (qed.Model(m, precision=precision, scheme=before) for _ in range(2))
    rho0 = torch.from_numpy(W.random_density(dim, seed=3)).cuda()
    other = torch.diag(torch.exp(1j * torch.arange(dim, device="cuda", dtype=torch.float64)))

    def do(model):
        if after == "U":
            model.set_U(other)
        else:
            model.set_scheme(after)

    def run(model):
        rho = rho0.clone()
        model.evolve(rho, 20)
        model.sync()
        return rho, model.get_U()

    expected = run(ref)
    do(ref)
    changed = run(ref)
    failed, budget = 0, 0
    while True:
        qed.set_alloc_budget(budget)
        try:
            do(gm)
            break
        except qed.QedError as e:
            assert e.status == qed.QED_ENOMEM
            failed += 1
        finally:
            qed.set_alloc_budget(-1)
        assert _same(gm, rho0, *expected), budget
        budget = max(8 * dim, budget + budget // 2)
        assert budget < 1 << 30
    assert _same(gm, rho0, *changed)
    # (a given U needs tables of its own in a cluster run and in split precision)
    assert failed > 0 or (precision == "fp64" and after == "U" and dim > 8)


@pytest.mark.parametrize("precision", ["fp64", "split_fp16x2"])
@pytest.mark.parametrize("change", [dict(extra_tunnel=[float("nan")]), dict(extra_tunnel=[float("-inf")]),
                                    dict(omega_c=1e308), dict(extra_tunnel=[1e300], dt=1e10),
                                    dict(g=[1e308] * 4)])
def test_hamiltonian_that_is_not_finite_is_refused(precision, change):
    """A tunnelling amplitude that is not a number, or entries, row sums or dt H that overflow: no
    propagator exists, in the series or in the Pade approximant."""
    m = W.hb_shaped()
    m.update(change)
    with pytest.raises(qed.QedError) as ei:
        qed.Model(m, precision=precision)
    assert ei.value.status == qed.QED_ENUMERIC


def test_alloc_budget_in_tc_gemm():
    A = torch.zeros((2, 128, 64), dtype=torch.float16, device="cuda")
    qed.set_alloc_budget(0)
    with pytest.raises(qed.QedError) as ei:
        qed.tc_gemm(A, A)
    assert ei.value.status == qed.QED_ENOMEM
    qed.set_alloc_budget(-1)
    assert float(qed.tc_gemm(A, A).abs().max()) == 0.0
