"""Site staging by exponent field (ordinary exponents) and by value (the rest), and the FP32 slice
guard at slice sizes around its warps, blocks and shared-memory key table (needs a GB300; marked
gpu)."""
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


def sites(plan, U, D):
    n = U.shape[2]
    C = torch.zeros(1, 1, dtype=torch.complex128, device="cuda")
    S = torch.zeros(1, 1, n, dtype=torch.complex128, device="cuda")
    plan.correlator(U, D, C, S)
    torch.cuda.synchronize()
    return S.cpu().numpy().ravel()


# the largest |re|, |im| lies in [1, 2): its exponent field is 1023 + shift, and fields from 200 on
# take the path by exponent field
@pytest.mark.parametrize("shift", [-900, -824, -823, -822, 60])
@pytest.mark.parametrize("algo,prec", [("egraph", "fp32"), ("egraph", "mixed"), ("tree", "mixed"), ("direct", "mixed")])
def test_staging_scales_exactly(ctx, algo, prec, shift):
    """The proton (two up, one down) is homogeneous: fields times powers of two give the same
    values times a power of two, bit for bit, on either path."""
    rng = np.random.default_rng(3)
    f = rng.uniform(-1.0, 1.0, (2, 1, 1, 33, 12, 12, 2))
    f[..., 0, 0, 0] = 1.5
    f[0, 0, 0, :, 3] *= 2.0 ** -70               # rows far below the largest entry, and zeros
    f[1, 0, 0, :, :, 7] = 0.0
    plan = ctx.plan_operator("proton", algo, prec)
    if prec == "fp32":
        plan.set_guard(float("inf"), float("inf"))
    up = -shift                                  # keeps the product in range
    got = []
    for a, b in ((0, 0), (shift, up)):
        z = np.stack((np.ldexp(f[0], a), np.ldexp(f[1], b))).view(np.complex128)[..., 0]
        U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in z)
        got.append(sites(plan, U, D))
    plan.destroy()
    assert np.all(got[0] != 0)
    k = 2 * shift + up
    assert np.array_equal(np.ldexp(got[0].view(np.float64), k), got[1].view(np.float64))


@pytest.mark.parametrize("tiny", [-1070, -1046, -1045, -1030])
@pytest.mark.parametrize("algo,prec", [("egraph", "fp32"), ("egraph", "mixed"), ("tree", "mixed"), ("direct", "mixed")])
def test_staging_of_subnormal_blocks(ctx, algo, prec, tiny):
    """The same with a down block of subnormal numbers only: integers of up to three bits times
    2^tiny, whose high words are all zero when the largest is below 2^-1042 (tiny up to -1045), and a site of
    zeros, which stays zero."""
    rng = np.random.default_rng(6)
    f = rng.integers(-7, 8, (2, 1, 1, 33, 12, 12, 2)).astype(np.float64)
    f[..., 0, 0, 0] = 7.0
    f[1, 0, 0, 5] = 0.0
    plan = ctx.plan_operator("proton", algo, prec)
    if prec == "fp32":
        plan.set_guard(float("inf"), float("inf"))
    got = []
    for a, b in ((0, 0), (500, tiny)):
        z = np.stack((np.ldexp(f[0], a), np.ldexp(f[1], b))).view(np.complex128)[..., 0]
        U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in z)
        got.append(sites(plan, U, D))
    plan.destroy()
    live = np.arange(33) != 5
    assert np.all(got[0][live] != 0) and got[0][5] == 0
    assert np.array_equal(np.ldexp(got[0].view(np.float64), 2 * 500 + tiny), got[1].view(np.float64))


@pytest.mark.parametrize("algo,prec", [("egraph", "fp32"), ("egraph", "mixed")])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_staging_non_finite_site(ctx, algo, prec, bad):
    """A site with a non-finite propagator is not finite; its neighbours keep their bits."""
    rng = np.random.default_rng(4)
    f = rng.standard_normal((2, 1, 1, 5, 12, 12, 2)).view(np.complex128)[..., 0]
    U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f)
    plan = ctx.plan_operator("proton", algo, prec)
    if prec == "fp32":                           # (the slice guard would recompute the whole slice: C is not a number)
        plan.set_guard(float("inf"), float("inf"))
    ref = sites(plan, U, D)
    U[0, 0, 2] = bad
    got = sites(plan, U, D)
    plan.destroy()
    assert not np.isfinite(got[2])
    keep = [0, 1, 3, 4]
    assert np.array_equal(got[keep], ref[keep])


@pytest.mark.parametrize("V3", [1, 31, 33, 511, 513, 40960, 40961])
def test_slice_guard_sizes(ctx, V3):
    """+inf lists only the site of zero propagators (its estimate, 0/0, is not a number), a tighter
    tolerance never fewer, 0 every site once; C(t) is within the tolerance of the double-float plan."""
    rng = np.random.default_rng(V3)
    f = rng.standard_normal((2, 1, 2, V3, 12, 12, 2)).view(np.complex128)[..., 0]
    f[:, 0, 1, V3 // 2] = 0.0
    U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f)
    mixed = ctx.plan_operator("proton", "egraph", "mixed")
    plan = ctx.plan_operator("proton", "egraph", "fp32")

    def run(p):
        C = torch.zeros(1, 2, dtype=torch.complex128, device="cuda")
        p.correlator(U, D, C)
        torch.cuda.synchronize()
        return C.cpu().numpy().ravel()

    ref = run(mixed)
    last = 0
    for tol in (float("inf"), 1e-6, 3e-7, 1e-7, 1e-8, 0.0):
        plan.set_guard(float("inf"), tol)
        C = run(plan)
        n = ctx.fp32_recomputed
        assert n >= last, (tol, n, last)
        last = n
        if tol == float("inf"):
            assert n == 1
        else:
            # double-float sites agree with the other plan's to its own rounding, 1e-10 of the
            # sum's condition here (sites add up as a random walk)
            assert np.all(np.abs(C - ref) <= (tol + 1e-10) * np.abs(ref)), (tol, C, ref)
    assert last == 2 * V3
    mixed.destroy()
    plan.destroy()


def test_batched_slice_guard_of_mixed_slice_sizes(ctx):
    """Items of one batch whose slices lie on both sides of the guard's block and key-table sizes are
    guarded as in separate calls: the same C(t), bit for bit, and as many sites recomputed.  A
    tolerance per size at which some slices are listed and some are not."""
    from paper_2201_04269_gb300 import abi
    items, plans, single, listed = [], [], [], 0
    for V3, T in ((33, 40), (64, 40), (513, 20), (2048, 8), (40960, 3), (40961, 3)):
        rng = np.random.default_rng(V3)
        f = rng.standard_normal((2, 1, T, V3, 12, 12, 2)).view(np.complex128)[..., 0]
        U, D = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f)
        plan = ctx.plan_operator("proton", "egraph", "fp32")
        C = torch.zeros(1, T, dtype=torch.complex128, device="cuda")
        n = 0
        for tol in (2e-7, 3e-7, 5e-7, 8e-7, 1.2e-6):          # (the first at which not every slice is listed)
            plan.set_guard(float("inf"), tol)
            plan.correlator(U, D, C)
            n = ctx.fp32_recomputed
            if n < T * V3 // 4:
                break
        listed += n
        single.append(C.cpu().numpy().copy())
        items.append(dict(plan=plan.handle, U=U, D=D, n_sets=1, T=T, V3=V3, C=C))
        plans.append(plan)
    assert listed > 0
    abi.mbc_batch(ctx.handle, items)
    torch.cuda.synchronize()
    assert ctx.fp32_recomputed == listed
    for it, C in zip(items, single):
        assert np.array_equal(it["C"].cpu().numpy(), C), it["V3"]
    for plan in plans:
        plan.destroy()
