"""The unitary step through the sparse Hamiltonian (the Taylor series of exp applied to every
column) against the general path, the dense products with U: a model whose own U is put
back with set_U takes that path.  At the edges of the kernels' blocks (32-row warps, 256 and
512 threads, one and two columns a block), with detuned cavities (a diagonal left in the
series), complex ones (the effective step), norms that need substeps, and every scheme."""
import numpy as np
import pytest

import qed_workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
qed = pytest.importorskip("paper_2403_07042_gb300")

U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_07042_gb300 import build
    build.build()


def chain(D, detuned=False, dt=0.1):
    """D states of a chain (the first by excitations): two atoms and up to three photons a cavity."""
    rng = np.random.default_rng(D)
    L = 5
    m = W.chain_instance(rng, 64, 64)
    m.update(n_cavities=L, atoms_per_cavity=[2] * L, n_max=[3] * L, dim_cap=D, dt=dt,
             g=[float(x) for x in rng.uniform(0.005, 0.02, size=2 * L)], bonds=[(c, c + 1) for c in range(L - 1)],
             zeta=[float(x) for x in rng.uniform(0.002, 0.01, size=L - 1)],
             jumps=[(0, c, 1e-3) for c in range(L)], omega_a=1.3 if detuned else 1.0)
    return m


def state(D, hermitian=True):
    gen = torch.Generator(device="cuda").manual_seed(D)
    w = torch.randn((D, 3), dtype=torch.complex128, device="cuda", generator=gen)
    v = w if hermitian else torch.randn((D, 3), dtype=torch.complex128, device="cuda", generator=gen)
    r = w @ v.mH
    if hermitian:
        r = 0.5 * (r + r.mH)
        return (r / torch.trace(r).real).contiguous()
    return (r / r.norm()).contiguous()


@pytest.mark.parametrize("D,detuned,dt,scheme", [
    (1, False, 0.1, "lie"), (2, False, 0.1, "lie"), (31, False, 0.1, "strang"), (32, True, 0.1, "lie"),
    (33, False, 0.1, "effective"), (255, True, 0.1, "effective"), (256, False, 0.1, "lie"),
    (257, False, 2.0, "lie"), (512, True, 0.1, "strang"), (513, False, 0.1, "lie"), (1024, False, 0.1, "lie"),
    (1025, True, 0.1, "lie"),
])
def test_fp64_matches_dense_products(D, detuned, dt, scheme):
    """n steps differ by the dense side's rounding, 2 n D u for a matrix of norm <= 1 (sums of D
    terms whose magnitudes add to at most 1, twice a step), and the series', whose terms and
    couplings add to far fewer roundings than 2 D + 64 a step."""
    n = 5
    m = chain(D, detuned, dt)
    a, b = (qed.Model(m, scheme=scheme) for _ in range(2))
    b.set_U(a.get_U())
    for hermitian in (True, False):
        rho = state(D, hermitian)
        ra, rb = rho.clone(), rho.clone()
        a.evolve(ra, n)
        b.evolve(rb, n)
        a.sync()
        b.sync()
        err = (ra - rb).abs().max().item()
        assert err <= n * (4 * D + 64) * U, (D, hermitian, err)


def test_fp64_injected_and_restored_propagator():
    """set_U takes over from the series, after steps as well; leaving the scheme and coming back
    restores the model's own propagator."""
    m = chain(200)
    gm = qed.Model(m)
    own = gm.get_U()
    rho0 = state(200)
    ref = rho0.clone()
    gm.evolve(ref, 20)
    gm.set_U(torch.eye(200, dtype=torch.complex128, device="cuda"))
    assert torch.equal(gm.get_U(), torch.eye(200, dtype=torch.complex128, device="cuda"))
    moved = rho0.clone()
    gm.evolve(moved, 20)
    gm.sync()
    assert (moved - ref).abs().max().item() > 1e-3  # the identity leaves the phases out
    gm.set_scheme("effective")
    gm.set_scheme("lie")
    assert torch.equal(gm.get_U(), own)
    again = rho0.clone()
    gm.evolve(again, 20)
    gm.sync()
    assert torch.equal(again, ref)


@pytest.mark.parametrize("precision,D,detuned,scheme,tol", [
    ("fp64", 33, True, "lie", 1e-9), ("fp64", 95, False, "strang", 1e-9), ("fp64", 96, True, "strang", 1e-9),
    ("fp64", 257, False, "lie", 1e-9), ("split_fp16x2", 130, True, "lie", 2.4e-5),
])
def test_sparse_gradients_match_dense(precision, D, detuned, scheme, tol):
    """The gradients through the sparse Frechet series against the dense one (an injected U: the
    products with U and the Pade approximant), to the FP64 and the split adjoint's accuracy
    relative to the largest gradient; a coupling of strength zero keeps its gradient."""
    m = chain(D, detuned)
    m["g"][1] = 0.0
    m["zeta"][2] = 0.0
    a, b = (qed.Model(m, precision=precision, scheme=scheme) for _ in range(2))
    b.set_U(a.get_U())
    rho, o = state(D), torch.linspace(-1.0, 1.0, D, dtype=torch.float64, device="cuda")
    ga, gb = (x.adjoint(rho, 9, o, checkpoint_every=4) for x in (a, b))
    for x, y in zip(ga, gb):
        assert (x - y).abs().max().item() <= tol * max(1e-12, y.abs().max().item())
    assert ga[1][1].abs().item() > 0.0


@pytest.mark.parametrize("scale", [1e-300, 1e-160, 1e-30, 1e30, 1e250])
def test_fp64_step_is_linear_in_the_magnitude(scale):
    """The double-float increments follow each column's exponent, and columns beyond its range
    take the FP64 loop: a step of s rho is s times the step of rho (powers of two and the loop's
    own rounding, 64 u), also with columns of very different magnitude, zero and denormal ones."""
    D = 130
    gm = qed.Model(chain(D, True))
    rho = state(D, hermitian=False)
    col = torch.ones(D, dtype=torch.float64, device="cuda")
    col[3], col[4], col[5] = 0.0, 2.0 ** -90, 2.0 ** 40
    base = rho * col[None, :]
    s = 2.0 ** round(np.log2(scale))
    one, many = base.clone(), (base * s).contiguous()
    gm.evolve(one, 1)
    gm.evolve(many, 1)
    gm.sync()
    top = one.abs().max().item()
    assert ((many / s) - one).abs().max().item() <= 64 * U * top


def test_fp64_non_finite_elements_stay_where_couplings_take_them():
    D = 130
    gm = qed.Model(chain(D))
    rho = state(D)
    bad = rho.clone()
    bad[7, 9] = float("nan")
    good = rho.clone()
    gm.evolve(bad, 1)
    gm.evolve(good, 1)
    assert torch.isnan(bad[7, 9].real)
    same = torch.isfinite(bad.real) & torch.isfinite(bad.imag)
    assert same.any() and (bad[same] - good[same]).abs().max().item() <= 64 * U


@pytest.mark.parametrize("D,scheme", [(1, "lie"), (2, "effective"), (9, "lie"), (10, "lie"), (13, "effective"),
                                      (17, "lie"), (36, "lie"), (63, "effective"), (64, "lie"), (65, "lie")])
@pytest.mark.parametrize("injected", [False, True])
def test_fp64_cluster_steps_match_kernel_steps(D, scheme, injected):
    """Many steps in one cluster launch (up to 64 states; one to sixteen CTAs, rows that do not
    divide, five jumps into the vacuum) against the same steps kernel by kernel (qed_profile runs
    them so): two dense products a step on either side, 4 D u a step for a matrix of norm <= 1."""
    n = 7
    gm = qed.Model(chain(D, True), scheme=scheme)
    if injected:
        gm.set_U(gm.get_U())
    ids = [0, D - 1, D, gm.n_observables - 1]
    for hermitian in (True, False):
        a = state(D, hermitian)
        b = a.clone()
        got = gm.evolve(a, n, record_every=2, obs_ids=ids, step_offset=3)
        rows = []
        for i in range(n + 1):
            if (3 + i) % 2 == 0:
                rows.append(gm.observables(b, ids))
            if i < n:
                gm.profile(b, 1)
        gm.sync()
        assert (a - b).abs().max().item() <= n * (4 * D + 64) * U
        # a recorded sum of D populations of magnitude at most one, each weighed up to 3
        assert (got - torch.stack(rows)).abs().max().item() <= 3 * D * n * (4 * D + 64) * U


@pytest.mark.parametrize("D", [96, 257, 1025])
def test_captured_get_U_leaves_the_late_U_to_be_formed(D):
    """An FP64 model forms its U on first use: a captured read of it runs only with the graph, so
    reads outside (on another stream too) must neither miss nor wait for it.  The same kernel
    forms all of them: equal to the bit."""
    gm, ref = qed.Model(chain(D), precision="fp64"), qed.Model(chain(D), precision="fp64")
    expected = ref.get_U()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        captured = gm.get_U(stream=torch.cuda.current_stream())
    with torch.cuda.stream(side):
        outside = gm.get_U(stream=side)
    assert torch.equal(outside, expected) and torch.equal(gm.get_U(), expected)
    captured.zero_()
    graph.replay()
    assert torch.equal(captured, expected)


@pytest.mark.parametrize("D,detuned", [(33, False), (96, True)])
def test_fp64_propagator_is_exact_in_its_small_elements(D, detuned):
    """Elements of U that couplings make, up to second neighbours: each level adds a rounding of its
    coupling, of 1/n, of the sum and one for each of up to 8 couplings (11 u), the two factors of
    the phase and their product 7 u: below 32 u of the element itself."""
    m = chain(D, detuned)
    H = np.asarray(qed.spec_hamiltonian(m)).real
    X = H.astype(np.longdouble) * np.longdouble(m["dt"])
    re, im, term = np.eye(D, dtype=np.longdouble), np.zeros((D, D), np.longdouble), np.eye(D, dtype=np.longdouble)
    for n in range(1, 40):  # (-i X)^n / n!, X real
        term = X @ term / n
        if n % 2:
            im += (-1) ** ((n + 1) // 2) * term
        else:
            re += (-1) ** (n // 2) * term
    near = (H != 0) | (np.eye(D) > 0)
    second = (near.astype(int) @ near.astype(int) > 0) & ~np.eye(D, dtype=bool)
    got = qed.Model(m).get_U().cpu().numpy()
    err = np.hypot((got.real - re).astype(float), (got.imag - im).astype(float))[second]
    size = np.hypot(re.astype(float), im.astype(float))[second]
    assert size.min() > 0
    assert (err / size).max() <= 32 * U


@pytest.mark.parametrize("D", [2, 36, 64, 65, 130])
def test_fp64_rho_need_not_start_on_a_16_byte_boundary(D):
    """A complex array of a C program starts where a double may: every FP64 size takes it, and the
    steps and records are those of an aligned copy, to the bit."""
    import ctypes
    gm = qed.Model(chain(D))
    rho = state(D)
    at = torch.zeros(2 * D * D + 3, dtype=torch.float64, device="cuda")
    odd = at[1:1 + 2 * D * D]
    assert odd.data_ptr() % 16 == 8
    odd.copy_(torch.view_as_real(rho).reshape(-1))
    ids = np.arange(D + 1, dtype=np.int32)
    rec = torch.zeros((4, D + 1), dtype=torch.float64, device="cuda")
    expected = gm.evolve(rho, 6, record_every=2, obs_ids=ids)
    status = qed.lib().qed_evolve(gm._h, ctypes.c_void_p(odd.data_ptr()), 6, 0, 2, D + 1,
                                  ids.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)),
                                  ctypes.c_void_p(rec.data_ptr()),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert status == 0
    gm.sync()
    assert torch.equal(odd, torch.view_as_real(rho).reshape(-1)) and torch.equal(rec, expected)
    assert at[0].item() == 0.0 and at[1 + 2 * D * D:].abs().max().item() == 0.0


def test_captured_get_U_into_an_array_of_doubles():
    """The same for a captured read of the late U."""
    import ctypes
    D = 130
    gm, expected = qed.Model(chain(D)), qed.Model(chain(D)).get_U()
    odd = torch.zeros(2 * D * D + 1, dtype=torch.float64, device="cuda")[1:]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        status = qed.lib().qed_get_U(gm._h, ctypes.c_void_p(odd.data_ptr()),
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert status == 0
    graph.replay()
    assert torch.equal(odd, torch.view_as_real(expected).reshape(-1))


def _long_double_steps(m, n, k):
    """(exp(-i H dt))^n e_k in long double, by the series of the whole H."""
    H = np.asarray(qed.spec_hamiltonian(m)).real
    X = H.astype(np.longdouble) * np.longdouble(m["dt"])
    re, im = np.zeros(len(H), np.longdouble), np.zeros(len(H), np.longdouble)
    re[k] = 1
    for _ in range(n):
        a, b = re.copy(), im.copy()
        for j in range(1, 40):  # (-i X)^j / j! applied to a + i b
            a, b = X @ b / j, -(X @ a) / j
            re, im = re + a, im + b
    return re, im


@pytest.mark.parametrize("D,detuned", [(8, False), (33, False), (64, True), (70, False), (96, True), (130, False),
                                       (257, True)])
@pytest.mark.parametrize("n", [1, 4])
def test_fp64_evolve_is_exact_in_its_small_elements(D, detuned, n):
    """What couplings make out of a pure state, and out of a far smaller one in another component of
    H, has the accuracy of its own size: U's elements up to second neighbours are within 32 u (the
    test above), each side adds the roundings of a sum of up to 9 terms of one phase and of its
    phases, so that a step takes 96 u of the element itself."""
    m = chain(D, detuned)
    m["jumps"] = []
    H = np.asarray(qed.spec_hamiltonian(m)).real
    near = ((H != 0) | (np.eye(D) > 0)).astype(int)
    reach = near @ near > 0
    joined = reach
    for _ in range(10):
        joined = joined @ joined
    k = 1
    far = np.flatnonzero(~joined[k])[-1]
    small = 2.0 ** -100
    rho = torch.zeros((D, D), dtype=torch.complex128, device="cuda")
    rho[k, k], rho[far, far] = 1.0, small
    gm = qed.Model(m)
    gm.evolve(rho, n)
    gm.sync()
    got = rho.cpu().numpy()
    for at, size in ((k, 1.0), (far, small)):
        re, im = _long_double_steps(m, n, at)
        of = np.flatnonzero(reach[at])
        re, im = re[of], im[of]
        ref_re, ref_im = np.outer(re, re) + np.outer(im, im), np.outer(im, re) - np.outer(re, im)
        block = got[np.ix_(of, of)] / size
        err = np.hypot((block.real - ref_re).astype(float), (block.imag - ref_im).astype(float))
        ref = np.hypot(ref_re.astype(float), ref_im.astype(float))
        assert ref.min() > 0
        assert (err / ref).max() <= 96 * n * U, (at, (err / ref).max() / U)


@pytest.mark.parametrize("dt", [1.0, 0.1, 1e-2, 1e-4, 1e-6])
def test_hopping_gradients_keep_their_accuracy_at_small_steps(dt):
    """The gradient of a hopping that the excitation reaches after two couplings is of the order
    dt^4: the series of the derivative must reach it at every dt.  Against long double, relative to
    the largest: the states and co-states of four steps carry 96 u a step each (test above), their
    products and the two series' sums 64 u more: 900 u."""
    D, n = 129, 4
    m = chain(D)
    m["jumps"], m["dt"] = [], dt
    H = np.asarray(qed.spec_hamiltonian(m)).real
    gm = qed.Model(m)
    L, nc = gm.labels(), m["n_cavities"]
    atom = [3 * c + 1 for c in range(nc)]
    k = next(i for i in range(D) if L[i].sum() == 1 and L[i][atom[-1]] == 1)  # an atom of the last cavity
    rho = torch.zeros((D, D), dtype=torch.complex128, device="cuda")
    rho[k, k] = 1.0
    o = torch.zeros(D, dtype=torch.float64, device="cuda")
    o[k] = 1.0
    got = gm.adjoint(rho, n, o, checkpoint_every=n)[2].cpu().numpy()
    # in long double: psi_j forwards, chi_j backwards from e_k, and dL/dzeta =
    # 2 Re [<chi_n | psi_n>^* sum_j <chi_n | U^(n-1-j) dU psi_j>], dU by its series
    X = H.astype(np.longdouble) * np.longdouble(dt)
    grad = []
    for b in range(len(m["zeta"])):
        one = dict(m, g=[0.0] * len(m["g"]), zeta=[float(i == b) for i in range(len(m["zeta"]))], omega_c=0.0,
                   omega_a=0.0)
        E = np.asarray(qed.spec_hamiltonian(one)).real.astype(np.longdouble) * np.longdouble(dt)
        # the pair (psi, dpsi) under exp(-i [[X, 0], [E, X]])
        p = [np.zeros(D, np.longdouble) for _ in range(4)]
        p[0][k] = 1
        for _ in range(n):
            t = [x.copy() for x in p]
            for j in range(1, 40):
                re, im, dre, dim = t
                t = [X @ im / j, -(X @ re) / j, (X @ dim + E @ im) / j, -(X @ dre + E @ re) / j]
                p = [x + y for x, y in zip(p, t)]
        grad.append(2 * (p[0][k] * p[2][k] + p[1][k] * p[3][k]))
    ref = np.array(grad)
    size = float(np.abs(ref).max())
    assert size > 0
    assert float(np.abs(got - ref).max()) <= 900 * U * size, float(np.abs(got - ref).max()) / size / U


@pytest.mark.parametrize("D,injected,in_cluster", [(8, False, True), (8, True, True), (36, False, True),
                                                   (36, True, False), (49, False, False), (64, True, False)])
def test_fp64_runs_in_a_cluster_where_that_is_faster(D, injected, in_cluster):
    """One launch a run, or three a step (long components of H, an injected U); the same results."""
    gm = qed.Model(chain(D))
    if injected:
        gm.set_U(gm.get_U())
    rho = state(D)
    ref = rho.clone()
    before = qed.launch_count()
    gm.evolve(rho, 6)
    assert qed.launch_count() - before == (1 if in_cluster else 18)
    gm.profile(ref, 6)  # kernel by kernel
    assert (rho - ref).abs().max().item() <= 6 * (4 * D + 64) * U


@pytest.mark.parametrize("shape", [(3, 5), (4, 4), (17, 1), (5, 5), (8, 4), (11, 3)])
@pytest.mark.parametrize("scheme", ["lie", "strang"])
def test_fp64_jumps_into_one_state(shape, scheme):
    """15 to 33 leaks into the vacuum, about the number that masks of the jumps take, against the
    oracle with its own U."""
    import oracle
    m = W.lattice(*shape, gamma=0.02, seed=1)
    b = oracle.enumerate_basis(m)
    gm = qed.Model(m, scheme=scheme)
    propagator = oracle.propagator(oracle.hamiltonian(m, b), m["dt"])
    gm.set_U(torch.from_numpy(propagator).cuda())
    rho0 = W.random_density(b.dim, seed=2)
    rho = torch.from_numpy(rho0).cuda()
    gm.evolve(rho, 30)
    gm.sync()
    ref = oracle.evolve(m, rho0=rho0, n_steps=30, U=propagator, basis=b, return_records=False, scheme=scheme)
    assert np.abs(rho.cpu().numpy() - ref).max() <= 1e-12


def strong(D, norm):
    """A chain whose couplings take the infinity norm of dt H without its diagonal to `norm`."""
    m = chain(D)
    for _ in range(2):
        H = np.asarray(qed.spec_hamiltonian(m)).real * m["dt"]
        now = np.abs(H - np.diag(np.diag(H))).sum(1).max()
        m["g"], m["zeta"] = [x * norm / now for x in m["g"]], [x * norm / now for x in m["zeta"]]
    assert abs(now - norm) <= 1e-12 * norm
    return m


@pytest.mark.parametrize("D,norm,scheme,passes", [
    (33, 1.5, "lie", False), (33, 7.9, "effective", False), (64, 4.0, "lie", False), (130, 0.9, "lie", False),
    (130, 1.5, "strang", False), (160, 0.9, "lie", True), (257, 1.5, "effective", True), (257, 4.0, "lie", False),
    (350, 4.0, "strang", True), (512, 7.9, "lie", True), (33, 9.5, "lie", False), (130, 9.5, "effective", False),
    (130, 40.0, "lie", False)])
def test_fp64_strong_couplings_match_oracle(D, norm, scheme, passes):
    """Norms of one to eight substeps and beyond the series (the Pade approximant, with squarings at
    40), through passes or dense products as passes_pay has it, against the oracle with its own
    propagator (an eigendecomposition; scipy's expm for the effective step).  U: a substep's sums are
    within 30 u of the column (e times 11 roundings a term), eight of them 240 u, squarings double
    what Pade and its elimination leave (D u); either reference is within 16 D u.  A step adds 4 D + 64."""
    import oracle
    m = strong(D, norm)
    b = oracle.enumerate_basis(m)
    H, jumps = oracle.hamiltonian(m, b), oracle.jump_operators(m, b)
    ref_U = oracle.effective_propagator(H, jumps, m["dt"]) if scheme == "effective" else oracle.propagator(H, m["dt"])
    gm = qed.Model(m, scheme=scheme)
    bound = (256 + 16 * D * max(1.0, norm / 8)) * U
    assert np.abs(gm.get_U().cpu().numpy() - ref_U).max() <= bound
    n = 3
    rho0 = W.random_density(D, seed=D)
    ref = oracle.evolve(m, rho0=rho0, n_steps=n, U=ref_U, basis=b, return_records=False, scheme=scheme)
    rho = torch.from_numpy(rho0).cuda()
    gm.evolve(rho, n)
    gm.sync()
    assert np.abs(rho.cpu().numpy() - ref).max() <= n * (2 * bound + (4 * D + 64) * U)
    assert ("strip_f64_1" in gm.profile(rho, 1)) == passes


@pytest.mark.parametrize("D,norm,scheme", [(33, 1.5, "lie"), (33, 9.5, "strang"), (130, 1.5, "lie"), (130, 4.0, "strang"),
                                           (257, 1.5, "lie")])
def test_gradients_of_strong_couplings_match_oracle(D, norm, scheme):
    """Beyond the first substep the derivative is the dense one, the co-state by passes (dim 257) or
    products; to the FP64 adjoint's accuracy."""
    import oracle
    m = strong(D, norm)
    b = oracle.enumerate_basis(m)
    o = np.linspace(-1.0, 1.0, D)
    rho0 = W.random_density(D, seed=D + 1)
    ref = oracle.adjoint_gradients(m, o, n_steps=4, rho0=rho0, basis=b, scheme=scheme)
    gm = qed.Model(m, scheme=scheme)
    got = gm.adjoint(torch.from_numpy(rho0).cuda(), 4, torch.from_numpy(o).cuda(), checkpoint_every=3)
    for x, y in zip(got[1:], ref[1:]):
        y = np.asarray(y, float)
        assert np.abs(x.cpu().numpy() - y).max() <= 1e-9 * np.abs(y).max()


@pytest.mark.parametrize("shape", [(43, 43), (44, 54)])
def test_fp64_passes_of_the_largest_dimensions(shape):
    """3699 and 4753 states (the largest take 4800): a pure state's step, to the bound of 96 u of the
    unit vector's projector."""
    m = W.lattice(*shape, seed=5, gamma=0.0)
    gm = qed.Model(m)
    D = gm.dim
    H = np.asarray(qed.spec_hamiltonian(m)).real * m["dt"]
    k = D // 2
    re, im = np.zeros(D), np.zeros(D)
    re[k] = 1.0
    a, b = re.copy(), im.copy()
    for j in range(1, 25):
        a, b = H @ b / j, -(H @ a) / j
        re, im = re + a, im + b
    psi = torch.from_numpy(re + 1j * im).cuda()
    rho = torch.zeros((D, D), dtype=torch.complex128, device="cuda")
    rho[k, k] = 1.0
    gm.evolve(rho, 1)
    gm.sync()
    assert (rho - torch.outer(psi, psi.conj())).abs().max().item() <= 96 * U
    assert "strip_f64_1" in gm.profile(rho, 1)


@pytest.mark.parametrize("D,precision", [(64, "fp64"), (129, "fp64"), (129, "split_fp16x2")])
@pytest.mark.parametrize("detuned", [False, True])
@pytest.mark.parametrize("dt", [0.1, 1e-3])
def test_propagator_is_exact_many_couplings_away(D, precision, detuned, dt):
    """Elements up to eight couplings away, as the Pade approximant has them: 11 u a level and the
    phases' 7 u (as for second neighbours above), the series' tail far below: 11 h + 16 u."""
    m = chain(D, detuned, dt)
    H = np.asarray(qed.spec_hamiltonian(m)).real
    X = H.astype(np.longdouble) * np.longdouble(dt)
    re, im, term = np.eye(D, dtype=np.longdouble), np.zeros((D, D), np.longdouble), np.eye(D, dtype=np.longdouble)
    for n in range(1, 40):
        term = X @ term / n
        if n % 2:
            im += (-1) ** ((n + 1) // 2) * term
        else:
            re += (-1) ** (n // 2) * term
    near = ((H != 0) | (np.eye(D) > 0)).astype(int)
    got = qed.Model(m, precision=precision).get_U().cpu().numpy()
    err = np.hypot((got.real - re).astype(float), (got.imag - im).astype(float))
    size = np.hypot(re.astype(float), im.astype(float))
    reach, before = near > 0, np.eye(D) > 0
    for h in range(1, 9):
        at = reach & ~before
        if at.any():
            assert (err[at] / size[at]).max() <= (11 * h + 16) * U, (h, (err[at] / size[at]).max() / U)
        before, reach = reach, reach.astype(int) @ near > 0
    assert at.any()
