"""The factor tree with its minors by shared Laplace steps and by LU (explicit terms whose minors
share much, little, or nothing between the two flavours) against the direct sweep, which factorises
every term's minors; site counts around the warp of 32 sites (needs a GB300; marked gpu)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04269_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


def terms(rng, n_u, n_d, n_sets, n_terms):
    """Explicit terms drawn from n_sets index tuples per flavour and side (few sets: many shared
    minors), real weights."""
    def sets(n):
        return [rng.choice(12, size=n, replace=False) for _ in range(n_sets)]
    su, sd, ru, rd = sets(n_u), sets(n_d), sets(n_u), sets(n_d)
    snk = np.array([np.concatenate((su[a], sd[b])) for a, b in rng.integers(0, n_sets, (n_terms, 2))], dtype=np.int8)
    src = np.array([np.concatenate((ru[a], rd[b])) for a, b in rng.integers(0, n_sets, (n_terms, 2))], dtype=np.int8)
    return snk, src, rng.integers(1, 5, n_terms).astype(np.complex128)


@pytest.mark.parametrize("n_u,n_d,n_sets,n_terms,complex_w", [
    (2, 1, 12, 200, False),          # one flavour of single entries
    (3, 2, 30, 400, True),           # complex coefficients
    (5, 4, 40, 2000, False),         # levels on both flavours
    (6, 6, 3, 4, False),             # a few scattered minors: LU
    (6, 0, 60, 2000, False),         # one flavour empty
])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-9)])
def test_tree_levels_match_direct(ctx, n_u, n_d, n_sets, n_terms, complex_w, prec, tol):
    rng = np.random.default_rng(100 * n_u + n_d)
    snk, src, w = terms(rng, n_u, n_d, n_sets, n_terms)
    if complex_w:
        w = w + 1j * rng.standard_normal(n_terms)
    for sites in (1, 31, 33):
        f = rng.standard_normal((2, 1, 1, sites, 12, 12, 2)).view(np.complex128)[..., 0]
        U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f)
        got = {}
        for algo, p in (("tree", prec), ("direct", "fp64")):
            plan = ctx.plan_terms(n_u, n_d, snk, src, w, algo=algo, prec=p)
            C = torch.zeros(1, 1, dtype=torch.complex128, device="cuda")
            S = torch.zeros(1, 1, sites, dtype=torch.complex128, device="cuda")
            plan.correlator(U, D, C, S)
            torch.cuda.synchronize()
            got[algo] = S.cpu().numpy().ravel()
            plan.destroy()
        # the sums of n_terms products cancel to about sqrt(n_terms) of them: compare to the
        # largest site value
        assert np.max(np.abs(got["tree"] - got["direct"])) <= tol * np.max(np.abs(got["direct"]))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_tree_of_more_sites_than_one_wave(ctx, prec):
    """The tables of 3He I take 4 MB a site, so that 1500 sites run in three waves of at most 2 GB
    with a shorter last one: the same site values, bit for bit, as in calls of one wave each."""
    rng = np.random.default_rng(8)
    plan = ctx.plan_operator("he3_I", "tree", prec)
    wave = (2 << 30) // plan.info["scratch_bytes_per_site"] // 32 * 32
    n = 1500
    assert 2 * wave < n < 3 * wave
    f = rng.standard_normal((2, 1, 1, n, 12, 12, 2)).view(np.complex128)[..., 0]
    U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f)

    def sites(a, b):
        C = torch.zeros(1, 1, dtype=torch.complex128, device="cuda")
        S = torch.zeros(1, 1, b - a, dtype=torch.complex128, device="cuda")
        plan.correlator(U[:, :, a:b].contiguous(), D[:, :, a:b].contiguous(), C, S)
        torch.cuda.synchronize()
        return S.cpu().numpy().ravel()

    whole = sites(0, n)
    parts = np.concatenate([sites(a, min(a + 300, n)) for a in range(0, n, 300)])
    plan.destroy()
    assert np.all(whole != 0) and np.array_equal(whole, parts)


def test_tree_autotune_times_what_the_schedule_changes(ctx):
    """The schedule sets the block size of the tree's LU kernel: a plan without it (dinucleon I) is
    evaluated under its own schedule only, four times; one with it (the proton's down entries)
    under others too."""
    from paper_2201_04269_gb300 import abi
    for op, alone in (("dinucleon_I", True), ("proton", False)):
        plan = ctx.plan_operator(op, "tree", "mixed")
        before = abi.mbc_get_schedule(plan.handle)
        f = np.random.default_rng(9).standard_normal((2, 1, 1, 33, 12, 12, 2)).view(np.complex128)[..., 0]
        U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f)
        C = torch.zeros(1, 1, dtype=torch.complex128, device="cuda")
        plan.correlator(U, D, C)
        n0 = ctx.launches
        plan.correlator(U, D, C)
        n1 = ctx.launches
        best = plan.autotune(U, D, 33)
        evaluations = (ctx.launches - n1) / (n1 - n0)
        assert evaluations == 4 if alone else evaluations > 4
        assert not alone or best == before
        plan.destroy()
