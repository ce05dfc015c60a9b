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


def test_fp32_product_in_place_and_variant_by_size(ctx):
    for n, variant in ((400, 4), (700, 3)):
        r, f = _cloud(n, n)
        R, F = dev(r), dev(f)
        want = host(ctx.mobility_matvec(R, F, 0.5, 1.0, True, "fp32"))
        assert ctx.pair_variant(n, True) == variant
        ctx.mobility_matvec(R, F, 0.5, 1.0, True, "fp32", out=F)
        assert rel_l2(host(F), want) <= 1e-14
