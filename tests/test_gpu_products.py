"""Products with the mobility at the sizes where their kernels change shape.

Tolerances: FP64 1e-12 relative L2 (a sum of n terms of about a hundred
roundings each, n eps ~ 1e-12 at the sizes here); FP32 1e-5 of the largest
velocity, the bar of the FP32 products, unless a test derives its own."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1602_02170_gb300 import inputs as I
from tests.gpu_common import ctx, dev, host, rel_l2  # noqa: F401

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}


def _cloud(seed, n):
    return I.blob_cloud(seed, n, 0.5, 2.0 * max(1.0, n ** 0.5), 0.5, 1.5)


@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 2209, 3140, 4420])
def test_fp64_items_of_every_size(ctx, n, wall):
    """The FP64 kernel's items hold 4, 8, 16 or 32 sources (the last three
    from about 2,200, 3,140 and 4,420 blobs); ragged and full blocks."""
    r, f = _cloud(n, n)
    got = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, wall, "fp64"))
    assert rel_l2(got, O.matvec(r, f, 0.5, 1.0, wall)) <= TOL["fp64"]


def test_fp64_length_scale_outside_fp32_range(ctx):
    """Lengths of 1e-25 put r^2 outside the FP32 range, where the FP64
    reciprocal square root takes its general form: M scales as 1 / length."""
    r, f = _cloud(5, 200)
    ref = O.matvec(r, f, 0.5, 1.0, True)
    got = host(ctx.mobility_matvec(dev(r * 1e-25), dev(f), 0.5e-25, 1.0, True, "fp64"))
    assert rel_l2(got * 1e-25, ref) <= TOL["fp64"]


def test_fp64_sums_of_many_blobs(ctx):
    """65,536 blobs without the wall, a few targets in extended precision.  A
    target takes 4,096 additions of items' sums, spread over 16 arrays: 256
    roundings of 0.29 ulp (rms) each at half of the array's final size, 2.5e-16
    of the whole, beside about 4e-16 of the pairs' and the items' own: 9e-16
    (in one array the additions alone are four times as much)."""
    n, a = 65536, 0.5
    r, f = I.blob_cloud(9, n, a, 400.0, a, 3 * a)
    got = host(ctx.mobility_matvec(dev(r), dev(f), a, 1.0, False, "fp64"))
    X = np.longdouble
    R, F, a = r.astype(X), f.astype(X), X(a)
    at = np.random.default_rng(9).permutation(n)[:24]
    ref = np.empty((len(at), 3), X)
    for k, i in enumerate(at):
        d = R[i] - R
        r2 = np.maximum((d * d).sum(1), X(1e-30))
        q = np.sqrt(r2)
        near = r2 < 4 * a * a
        C = np.where(near, 1 - 9 * q / (32 * a), 3 * a / (4 * q) + a ** 3 / (2 * q * r2))
        D = np.where(near, 3 / (32 * a * q), (3 * a / 4 - 3 * a ** 3 / (2 * r2)) / (q * r2))
        ref[k] = (C[:, None] * F + (D * (d * F).sum(1))[:, None] * d).sum(0)
    ref /= 6 * X("3.14159265358979323846264338327950288") * a
    err = np.sqrt((((got[at] - ref) ** 2).sum() / (ref ** 2).sum()).astype(np.float64))
    assert err <= 9e-16


@pytest.mark.parametrize("n", [3000, 9000])
def test_fp64_product_in_a_graph(n):
    """A captured FP64 product, on a new context or after a first call, and (from
    8,192 blobs on, whose graphs hold no workspace) after a larger product has
    moved the context's.  1e-14: the last FP64 bits of sums of n terms."""
    import torch

    import paper_1602_02170_gb300 as mb

    r, f = _cloud(n, n)
    R, F = dev(r), dev(f)
    for warm in (False, True):
        with mb.Context(0) as c:
            with mb.Context(0) as other:
                want = host(other.mobility_matvec(R, F, 0.5, 1.0, True, "fp64"))
            if warm:
                c.mobility_matvec(R, F, 0.5, 1.0, True, "fp64")
            out = torch.zeros_like(R)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                c.mobility_matvec(R, F, 0.5, 1.0, True, "fp64", out=out)
            if n >= 8192:
                R2, F2 = (dev(v) for v in _cloud(1, 2 * n))
                c.mobility_matvec(R2, F2, 0.5, 1.0, True, "fp64")
            for _ in range(2):
                out.zero_()
                g.replay()
                assert rel_l2(host(out), want) <= 1e-14


@pytest.mark.parametrize("target", ["f", "r"])
def test_fp64_product_in_place(ctx, target):
    """The velocities may overwrite the forces or the positions."""
    r, f = _cloud(6, 700)
    R, F = dev(r), dev(f)
    want = host(ctx.mobility_matvec(R, F, 0.5, 1.0, True, "fp64"))
    out = F if target == "f" else R
    ctx.mobility_matvec(R, F, 0.5, 1.0, True, "fp64", out=out)
    assert rel_l2(host(out), want) <= 1e-14


@pytest.mark.parametrize("gap", [90.0, 95.9, 96.1, 400.0])
def test_fp32_far_and_very_far_blocks(ctx, gap):
    """Two clusters of blobs a = 0.5 high above the wall, forces on one of
    them only: the other's velocities come from block pairs around the
    distance of 192 a = 96 from which the FP32 kernel leaves out the terms in
    (a / rho)^4.  Expected: some twenty roundings of 2^-24 a pair, separations
    from hi parts (2^-24 of coordinates up to 420 against 90 and more) and
    dropped terms below 2^-26, so 4e-6 of the FP64 product."""
    rng = np.random.default_rng(int(gap))
    n = 9216  # 18 blocks of 512 in each cluster
    r = rng.uniform([0, 0, 40], [10, 10, 50], (2 * n, 3))
    r[n:, 0] += 10.0 + gap
    f = rng.standard_normal((2 * n, 3))
    f[n:] = 0.0
    ctx.set_pair_variant(3)
    try:
        got = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, True, "fp32"))
    finally:
        ctx.set_pair_variant(-1)
    ref = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, True, "fp64"))
    assert rel_l2(got[n:], ref[n:]) <= 4e-6


@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("n", [1, 63, 65, 599, 600, 2999, 3001, 11999, 12003])
def test_fp32_symmetric_blocks_of_every_size(ctx, n, wall):
    """The symmetric FP32 kernel's blocks hold 64, 128 (from 3,000 blobs) or
    256 blobs (from 12,000); ragged and nearly empty last blocks, against the
    FP64 product."""
    r, f = _cloud(n, n)
    ctx.set_pair_variant(3)
    try:
        got = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, wall, "fp32"))
    finally:
        ctx.set_pair_variant(-1)
    ref = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, wall, "fp64"))
    assert np.abs(got - ref).max() <= TOL["fp32"] * np.abs(ref).max()


@pytest.mark.parametrize("wall,bar", [(True, 2.1e-7), (False, 1.7e-7)])
def test_fp32_sums_of_the_middle_sizes(ctx, wall, bar):
    """40 shells of 162 blobs (blocks of 128 blobs): pair terms good to about
    1.1e-7, or 1.5e-7 where the wall's parts nearly cancel, in FP32 sums of 16
    terms (0.4 x 2^-24 sqrt(16 / 2) = 0.7e-7 for one rounding a term, 1e-7 for
    two): 1.3e-7 and 1.8e-7, a sixth more allowed.  Sums over 64 terms have
    twice the rounding, 1.8e-7 and 2.5e-7."""
    rng = np.random.default_rng(11)
    nb, a = 40, 0.12
    p = np.arange(nb)
    q = np.stack([p % 7 * 3.125, p // 7 * 3.125, rng.uniform(1.05 + a, 1.45 + a, nb)], axis=1)
    th = I.random_unit_quaternions(rng, nb)
    start = 162 * np.arange(nb + 1)
    r = O.blob_positions(q, th, start, np.tile(I.shell(162), (nb, 1)))
    f = rng.standard_normal(r.shape)
    got = host(ctx.mobility_matvec(dev(r), dev(f), a, 1.0, wall, "fp32"))
    ref = host(ctx.mobility_matvec(dev(r), dev(f), a, 1.0, wall, "fp64"))
    assert rel_l2(got, ref) <= bar


def test_fp32_product_in_place_and_variant_by_size(ctx):
    for n, variant in ((400, 4), (700, 3)):
        r, f = _cloud(n, n)
        R, F = dev(r), dev(f)
        want = host(ctx.mobility_matvec(R, F, 0.5, 1.0, True, "fp32"))
        assert ctx.pair_variant(n, True) == variant
        ctx.mobility_matvec(R, F, 0.5, 1.0, True, "fp32", out=F)
        assert rel_l2(host(F), want) <= 1e-14


@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("n", [1, 15, 33, 1100, 1101, 1153, 23999, 24001])
def test_df64_blocks_of_every_size(ctx, n, wall):
    """Double-float: forward only up to 1,100 blobs, blocks of 64 blobs above
    and of 256 from 24,000, ragged and nearly empty last blocks, in a narrow
    strip (so that the largest sizes have far and near block pairs), against
    the FP64 product.  Positions are carried to 2^-49 of coordinates up to 30
    at separations of 0.1 and more, the arithmetic to about 2^-45: 1e-12."""
    r, f = I.blob_cloud(n, n, 0.1, 30.0, 0.1, 0.5)
    r[:, 1] *= 0.2
    got = host(ctx.mobility_matvec(dev(r), dev(f), 0.1, 1.0, wall, "df64"))
    ref = host(ctx.mobility_matvec(dev(r), dev(f), 0.1, 1.0, wall, "fp64"))
    assert rel_l2(got, ref) <= 1e-12


def test_df64_overlaps_in_both_halves(ctx):
    """Coincident, overlapping and touching blobs 32 and 64 places apart, the
    halves of one packed pair and its neighbours, above the forward-only
    size."""
    rng = np.random.default_rng(3)
    r = np.stack([np.arange(1300) * 3.0, np.full(1300, 1.0), rng.uniform(0.5, 2.0, 1300)], axis=1)
    for p in range(0, 1200, 97):
        r[p + 1] = r[p]
        r[p + 32] = r[p] + [0.3, 0.0, 0.0]
        r[p + 64] = r[p] + [0.0, 1.0, 0.0]
    f = rng.standard_normal(r.shape)
    ref = O.matvec(r, f, 0.5, 1.0, True)
    got = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, True, "df64"))
    # coordinates up to 3,900 carried to 2^-49, separations from 0.3 on: 1e-10
    assert np.isfinite(got).all()
    assert rel_l2(got, ref) <= 1e-10


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nt,ns", [(1, 1), (31, 3), (63, 15), (65, 17), (257, 129), (20000, 50), (70, 6000), (3000, 2500)])
def test_eval_splits(ctx, prec, nt, ns):
    """Flow evaluation from one item to chunks of every length, against the
    oracle's matvec over blobs and force-free points (FP32: of the unbounded
    flow's norm, as its terms nearly cancel near the wall)."""
    r, f = _cloud(nt + ns, ns)
    x, _ = _cloud(nt, nt)
    got = host(ctx.mobility_eval(dev(x), dev(r), dev(f), 0.5, 1.0, True, prec))
    ref = O.eval_points(x, r, f, 0.5, 1.0, True)
    free = O.eval_points(x, r, f, 0.5, 1.0, False)
    assert np.linalg.norm(got - ref) <= TOL[prec] * np.linalg.norm(free)


def test_eval_within_a_small_budget():
    """A context whose budget holds no partial sums evaluates in one chunk."""
    import paper_1602_02170_gb300 as mb

    r, f = _cloud(1, 3000)
    x, _ = _cloud(2, 2000)
    with mb.Context(0) as big, mb.Context(0, 200_000) as small:
        want = host(big.mobility_eval(dev(x), dev(r), dev(f), 0.5, 1.0, True, "fp32"))
        got = host(small.mobility_eval(dev(x), dev(r), dev(f), 0.5, 1.0, True, "fp32"))
        assert small.workspace_bytes() <= 200_000 < big.workspace_bytes()
    assert rel_l2(got, want) <= TOL["fp32"]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("chunks", [0.9, 1.0, 1.2, 2.0, 3.5, 6.8, 9.0, 10.1, 16.0, 40.0])
def test_eval_at_every_budget(ctx, prec, chunks):
    """Whatever the budget beyond the packed positions, the evaluation takes the
    chunks whose partial sums it holds, headroom of the allocation included."""
    import paper_1602_02170_gb300 as mb

    nt, ns = 2000, 3000
    r, f = _cloud(1, ns)
    x, _ = _cloud(2, nt)
    packed = 2 * 18 * (ns + nt) if prec == "fp32" else 0  # 16 bytes and an eighth
    want = host(ctx.mobility_eval(dev(x), dev(r), dev(f), 0.5, 1.0, True, prec))
    budget = packed + int(24 * nt * chunks)
    with mb.Context(0, max(1, budget)) as c:
        got = host(c.mobility_eval(dev(x), dev(r), dev(f), 0.5, 1.0, True, prec))
        assert c.workspace_bytes() <= budget
    assert rel_l2(got, want) <= TOL[prec]


@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("n", [1, 33, 599, 600, 3001, 16383, 16384, 20011])
def test_noalloc_every_size_and_in_place(ctx, n, wall):
    """The allocation-free product takes the one-warp kernel below 600 blobs,
    the symmetric one above and the spatial order from 16,384 on, and may
    overwrite its forces; against the FP64 product."""
    import paper_1602_02170_gb300 as mb

    r, f = _cloud(n, n)
    R, F = dev(r), dev(f)
    ref = host(ctx.mobility_matvec(R, F, 0.5, 1.0, wall, "fp64"))
    got = host(mb.mobility_matvec_noalloc(R, F, 0.5, 1.0, wall))
    assert np.abs(got - ref).max() <= TOL["fp32"] * np.abs(ref).max()
    mb.mobility_matvec_noalloc(R, F, 0.5, 1.0, wall, out=F)
    assert np.abs(host(F) - got).max() <= 1e-14 * np.abs(ref).max()


@pytest.mark.parametrize("wall", [True, False])
@pytest.mark.parametrize("n", [4095, 4096, 4097])
def test_fp32_symmetric_blocks_where_they_grow(ctx, n, wall):
    """Blocks of 64 blobs below 4,096 blobs, of 128 from there on; the last one
    is nearly empty at 4,097."""
    r, f = _cloud(n, n)
    got = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, wall, "fp32"))
    assert ctx.pair_variant(n, wall) == 3
    ref = host(ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, wall, "fp64"))
    assert np.abs(got - ref).max() <= TOL["fp32"] * np.abs(ref).max()


def test_fp32_variant_of_large_products(ctx):
    r, f = _cloud(20000, 20000)
    ctx.mobility_matvec(dev(r), dev(f), 0.5, 1.0, True, "fp32")
    assert ctx.pair_variant(20000, True) == 3


def test_fp64_reciprocal_square_root_to_the_last_bits(ctx):
    """One blob far smaller than every distance, points beside it: u = 3a/4 / r (and
    (a / r)^2 of it) in units of 1 / (6 pi eta a).  Distances of 26 bits have exact
    squares, so u carries the reciprocal square root's rounding (one ulp allowed)
    and those of two products: 2 ulp.  r^2 runs over the FP32 exponents, where the
    estimate is an FP32 one, and beyond both ends of them."""
    rng = np.random.default_rng(2)
    a = 2.0 ** -80
    e = np.concatenate([rng.integers(-72, 73, 6000), np.tile([-64, -63, 62, 63, 64], 800)])
    y = np.ldexp(rng.integers(2 ** 25, 2 ** 26, len(e)).astype(np.float64), e - 25)
    y[-10:] = np.ldexp(1.0, [-64, -63, -62, 62, 63, 64, -1, 0, 1, 2])
    x = np.zeros((len(y), 3))
    x[:, 1] = y
    got = host(ctx.mobility_eval(dev(x), dev(np.zeros((1, 3))), dev([[1.0, 0.0, 0.0]]), a, 1.0, False, "fp64"))
    L = np.longdouble
    ref = L(1.0 / (6.0 * np.pi * 1.0 * a)) * (L(0.75 * a) / L(1) / y.astype(L) + L(0.5) * L(a) ** 3 / y.astype(L) ** 3)
    assert np.abs(got[:, 0] / ref - 1).max() <= 2 * 2.0 ** -52
    assert np.all(got[:, 1:] == 0)
