"""Device memory of the digit products: what an earlier FP64 product keeps for speed never makes a
later call fail that fits without it, and what a limit leaves no room for runs another way."""
import numpy as np
import pytest

from synthetic import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from conftest import build_library
    build_library()
    import paper_2511_21640_gb300 as m
    return m


def _vectors(n, k, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((k, n)) + 1j * rng.standard_normal((k, n))


@pytest.mark.parametrize("precision", ["sliced", "sliced24"])
@pytest.mark.parametrize("kind,nocc,nvir", [("EA", 12, 40), ("IP", 36, 20)])
def test_sliced_product_after_kept_fp64_digits(gpu, kind, nocc, nvir, precision):
    """A limit that a block of sliced products just fits in: it also fits after an FP64 product has
    kept its operators' longer digits. Both results carry the product's 40 (24) bits, so they agree
    to 1e-11 (1e-6) of the largest output."""
    p = make_problem(nocc=nocc, nvir=nvir, naux=60, seed=5)

    def context(limit):
        return gpu.Context(p.B, p.eps_occ, p.eps_vir, kind=kind, order=3, x=0.5, mem_limit=limit)

    with context(0) as c:
        setup_peak = c.memory()["peak"]
        X = _vectors(c.N, 1500, 6)
        want = c.sigma(X, precision)
        peak = c.memory()["peak"]
    assert peak > setup_peak
    limit = peak + (1 << 20)
    with context(limit) as c:
        held = c.memory()["in_use"]
        c.sigma(X[:32], "fp64")
        assert c.memory()["in_use"] > held + (8 << 20)
        got = c.sigma(X, precision)
        assert c.memory()["peak"] <= limit
    assert np.abs(got - want).max() < (1e-11 if precision == "sliced" else 1e-6) * np.abs(want).max()


def _problem():
    return make_problem(nocc=12, nvir=40, naux=60, seed=5)


def test_kept_digits_take_a_quarter_together(gpu):
    """All operators' digits together stay within a quarter of what a limit leaves, also when each
    alone would fit."""
    p = _problem()
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        held, setup_peak = c.memory()["in_use"], c.memory()["peak"]
        X = _vectors(c.N, 32, 7)
        want = c.sigma(X, "fp64")
        every = c.kept_digits()["own"]
        assert every > 0
    left = int(3.6 * every)
    assert held + left > setup_peak
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5, mem_limit=held + left) as c:
        for _ in range(3):
            got = c.sigma(X, "fp64")
            assert c.kept_digits()["own"] <= left // 4
        assert np.abs(got - want).max() < 1e-13 * np.abs(want).max()


def test_a_failed_build_is_not_charged_and_not_final(gpu):
    """Digits whose allocation fails are not counted as kept; once there is memory again, later
    products keep them; a closed context leaves nothing counted."""
    p = _problem()
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        X = torch.from_numpy(_vectors(c.N, 32, 8)).cuda()
        want = c.sigma(X, "fp64").cpu().numpy()
        every = c.kept_digits()
        assert every["own"] > 0 and every["own"] == every["device"]
        peak = c.memory()["peak"]
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        assert c.kept_digits()["device"] == 0
        # room for a product on the FP64 units (its scratch), not for the digits
        scratch = 4 * 16 * 32 * 12 * 40 * 40
        assert c.memory()["in_use"] + scratch < peak
        assert gpu.lib.adc_diag_set_alloc_limit(c.kept_digits()["total"] + scratch) == 0
        try:
            got = c.sigma(X, "fp64").cpu().numpy()
            short = c.kept_digits()
        finally:
            gpu.lib.adc_diag_set_alloc_limit(0)
        assert short["own"] == short["device"] < every["own"]
        for _ in range(40):
            again = c.sigma(X, "fp64").cpu().numpy()
        assert c.kept_digits()["own"] == every["own"]
        for s in (got, again):
            assert np.abs(s - want).max() < 1e-13 * np.abs(want).max()


@pytest.mark.parametrize("other", ["context", "batch"])
def test_kept_digits_go_back_to_other_contexts(gpu, other):
    """Device memory that suffices only with the digits another, idle context keeps: a second
    context's product, and a batch's, take them and run; the first context then works as before."""
    p = _problem()

    def context():
        return gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5)

    with context() as a, context() as b:
        small, X = _vectors(a.N, 32, 9), _vectors(a.N, 300, 10)
        Xd = torch.from_numpy(X).cuda()
        need = 16 * (2 * 300 * b.N + 2 * 300 * 12 * 40 * 40)  # host blocks copied in and out, scratch
        if other == "batch":
            for _ in range(2):  # operator copies and tile widths first, then what the batch itself holds
                with gpu.Batch([b]) as batch:
                    before = b.kept_digits()["total"]
                    batch.sigma([Xd])
                    need = b.kept_digits()["total"] - before
        want = a.sigma(small, "fp64")
        kept = a.kept_digits()
        assert kept["own"] == kept["device"] > 0 and need > kept["own"]
        batch = gpu.Batch([b])
        assert gpu.lib.adc_diag_set_alloc_limit(a.kept_digits()["total"] + need - kept["own"] // 2) == 0
        try:
            got = b.sigma(X, "fp64")[:2] if other == "context" else batch.sigma([Xd])[0][:2].cpu().numpy()
        finally:
            gpu.lib.adc_diag_set_alloc_limit(0)
            batch.close()
        assert a.kept_digits()["own"] == 0
        ref = b.sigma(X[:2], "fp64")
        assert np.abs(got - ref).max() < (1e-13 if other == "context" else 1e-3) * np.abs(ref).max()
        again = a.sigma(small, "fp64")
        assert np.abs(again - want).max() < 1e-13 * np.abs(want).max()


def test_kept_digits_do_not_shrink_the_subspace(gpu, capfd):
    """An FP64 solve under a limit that just holds its default subspace goes through the same
    subspace sizes as without a limit (as printed per iteration), and reaches the same roots."""
    p, nroots, block = _problem(), 16, 32

    def solve(limit):
        with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5, mem_limit=limit, block=block,
                         verbose=True) as c:
            held, N = c.memory()["in_use"], c.N
            om = c.davidson(nroots, tol=1e-9, precision="fp64", want_vectors=False)[0]
        lines = [ln for ln in capfd.readouterr().err.splitlines() if ln.startswith("[davidson] it")]
        return held, N, om, [int(ln.split(" m ")[1].split()[0]) for ln in lines]

    held, N, want, sizes = solve(0)
    # 256 vectors and their products, the solve's other vectors and its estimate of one product's scratch, 8% over
    vec = 16 * N
    need = (2 * 8 * block + 3 * nroots + 2 * block) * vec + 16 * (2 * block * 12 * 40 * 40 + 8 * block * N)
    _, _, got, limited = solve(held + int(need / 0.92) + (1 << 20))
    assert max(sizes) > 160 and limited == sizes
    assert np.abs(got - want).max() < 1e-9


def _limited(gpu, p, left):
    """A context with `left` bytes to allocate after its setup."""
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        held = c.memory()["in_use"]
        assert held + left > c.memory()["peak"]
    return gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5, mem_limit=held + left, profile=True)


def test_per_call_planes_leave_kept_digits(gpu):
    """Digit planes that one product slices and frees never push out those kept for every product."""
    p = _problem()
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        X = _vectors(c.N, 32, 7)
        want = c.sigma(X, "fp64")
        left = int(2.5 * c.kept_digits()["own"])
    with _limited(gpu, p, left) as c:
        for _ in range(2):
            got = c.sigma(X, "fp64")
            assert 0 < c.kept_digits()["own"] <= left // 4
    assert np.abs(got - want).max() < 1e-13 * np.abs(want).max()


def test_a_limit_chunks_the_digits(gpu):
    """A limit without room for a term's whole digit planes (149 MB for the ladder of 200 vectors):
    the term runs from digits all the same, in chunks."""
    p = _problem()
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        X = _vectors(c.N, 200, 11)
        want = c.sigma(X, "fp64")
    blocks = 16 * (2 * 200 * c.N + 2 * 200 * 12 * 40 * 40)
    with _limited(gpu, p, blocks + (30 << 20)) as c:
        c.profile(True)
        got = c.sigma(X, "fp64")
        ran = c.profile_read()
        c.profile(False)
    assert "tc_digits_fp64/ladder" in ran and "zgemm_fp64/ladder" not in ran, ran
    assert np.abs(got - want).max() < 1e-13 * np.abs(want).max()


def test_batch_solve_stays_within_its_plan(gpu):
    """Two problems in a wave whose budget is just the plan's estimate, set up one after the other
    (the estimate does not count the intermediates of setups at the same time): the digit planes
    of their FP64 setup and products, which it does not count either, stay out of it. The roots are those
    of the problems solved alone, to the solves' tolerance."""
    probs = []
    for i in range(2):
        p = make_problem(nocc=18, nvir=90, naux=60, seed=12 + i)
        p.kind, p.order, p.x = "EA", 3, 0.5
        probs.append(p)
    sizes = [dict(nocc=18, nvir=90, naux=60, kind="EA", order=3, x=0.5)] * 2
    budget = int(gpu.batch_plan(sizes, 2, 1 << 60)[3].sum())
    gpu.lib.adc_diag_alloc_peak()
    before = gpu.lib.adc_diag_alloc_peak()  # the record starts at the total now
    om, _, status, info, rc = gpu.batch_solve(probs, 2, tol=1e-6, precision="fp64", mem_budget=budget,
                                              init_lanes=1)
    peak = gpu.lib.adc_diag_alloc_peak() - before
    assert rc == 0 and info["waves"] == 1
    assert peak <= budget, (peak, budget)
    for p, w in zip(probs, om):
        with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
            assert np.abs(c.davidson(2, tol=1e-6, precision="fp64", want_vectors=False)[0] - w).max() < 1e-8


@pytest.mark.parametrize("M,N,K", [(1300, 1300, 2000), (300, 36, 12600), (700, 650, 3000)])
def test_fp64_units_without_room_for_partial_sums(gpu, M, N, K):
    """A product on the FP64 units with memory for its operands alone runs with whole inner sums.
    Reference and product are the same computation there: equal."""
    with gpu.Context(*(lambda p: (p.B, p.eps_occ, p.eps_vir))(make_problem(4, 6, 8, seed=1)), kind="IP") as c:
        operands = 16 * (M * K + N * K + 2 * M * N)
        assert gpu.lib.adc_diag_set_alloc_limit(c.kept_digits()["total"] + operands + 65536) == 0
        try:
            err, _ = gpu.diag_gemm(0, M, N, K, seed=3, reps=1)
        finally:
            gpu.lib.adc_diag_set_alloc_limit(0)
    assert err == 0.0


def test_a_limit_equal_to_what_a_context_holds(gpu):
    """Nothing is held for speed alone under a limit: a product of device operands too small for
    digits needs no more than its scratch."""
    p = make_problem(4, 10, 12, seed=2)
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        peak = c.memory()["peak"]
    free = peak - (4 << 20) - (16 << 10)  # what the partial sums' buffers of an unlimited context take
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5, mem_limit=free + (1 << 18)) as c:
        X = torch.from_numpy(_vectors(c.N, 2, 3)).cuda()
        got = c.sigma(X, "fp64").cpu().numpy()
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5) as c:
        want = c.sigma(X, "fp64").cpu().numpy()
    assert np.abs(got - want).max() < 1e-13 * np.abs(want).max()


@pytest.mark.parametrize("precision", ["sliced", "sliced24"])
@pytest.mark.parametrize("kind,nocc,nvir", [("EA", 12, 40), ("IP", 36, 20)])
def test_sliced_product_does_not_depend_on_earlier_calls(gpu, kind, nocc, nvir, precision):
    """The same sliced product before and after an FP64 product of the context: the same bits."""
    p = make_problem(nocc=nocc, nvir=nvir, naux=60, seed=13)
    with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind=kind, order=3, x=0.5) as c:
        X = _vectors(c.N, 32, 14)
        first = c.sigma(X, precision)
        c.sigma(X, "fp64")
        assert c.kept_digits()["own"] > 0
        assert np.array_equal(c.sigma(X, precision), first)


def test_memory_comes_back_beside_running_products(gpu):
    """The same while the other context, in a thread of its own, runs FP64 products all the time: its
    digits are in use and its products' planes come and go, and the second context's products all
    find their memory."""
    import threading
    p = _problem()

    def context():
        return gpu.Context(p.B, p.eps_occ, p.eps_vir, kind="EA", order=3, x=0.5)

    with context() as a, context() as b:
        small, X = _vectors(a.N, 32, 9), _vectors(a.N, 300, 10)
        Xa = torch.from_numpy(small).cuda()
        Sa = torch.empty_like(Xa)
        torch.cuda.synchronize()
        want, ref = a.sigma(small, "fp64"), b.sigma(X, "sliced")[:2]
        need = 16 * 2 * 300 * b.N
        stop, failed = threading.Event(), []

        def products():
            while not stop.is_set():
                rc = [gpu.lib.adc_sigma(a._h, Xa.data_ptr(), Sa.data_ptr(), 32, 0) for _ in range(50)]
                rc.append(gpu.lib.adc_sync(a._h))
                if any(rc):
                    failed.append(rc)
                    return

        own = a.kept_digits()["own"]
        assert gpu.lib.adc_diag_set_alloc_limit(a.kept_digits()["total"] + need - own // 2) == 0
        t = threading.Thread(target=products)
        t.start()
        try:
            for _ in range(100):
                got = b.sigma(X, "sliced")[:2]
        finally:
            stop.set()
            t.join()
            gpu.lib.adc_diag_set_alloc_limit(0)
        assert not failed
        assert np.abs(got - ref).max() < 1e-11 * np.abs(ref).max()
        assert np.abs(a.sigma(small, "fp64") - want).max() < 1e-13 * np.abs(want).max()
