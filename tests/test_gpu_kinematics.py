"""Blob build, K and K^T where their tiles and lane groups change: bodies of
one blob, empty bodies, more bodies in a tile of 256 blobs than it keeps in
shared memory (64), and enough bodies for half a warp each (2,048).

Sums of up to 700 terms of size 1 with coordinates up to 60: 1e-12."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from tests.gpu_common import ctx, dev, host  # noqa: F401

pytestmark = pytest.mark.gpu


def _case(counts, seed):
    rng = np.random.default_rng(seed)
    counts = np.asarray(counts)
    start = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    nb, n = len(counts), int(start[-1])
    return (rng.uniform(0, 60, (nb, 3)), rng.standard_normal((nb, 4)), start,
            rng.standard_normal((n, 3)), rng)


COUNTS = {
    "one blob": [1],
    "ones": [1] * 700,
    "ragged": [255, 1, 257, 0, 3, 700, 42],
    "empty": [5] + [0] * 90 + [7] + [0] * 90 + [300],
    "many": [3, 15, 42] * 700,
    "tiles of two rounds": [162] * 1650,
}


@pytest.mark.parametrize("name", COUNTS)
def test_kinematics_by_body_sizes(ctx, name):
    q, theta, start, rho, rng = _case(COUNTS[name], len(name))
    nb, n = len(q), len(rho)
    S = torch.as_tensor(start, device="cuda")
    r = host(ctx.blob_positions(dev(q), dev(theta), S, dev(rho)))
    unit = theta / np.linalg.norm(theta, axis=1, keepdims=True)
    assert np.abs(r - O.blob_positions(q, unit, start, rho)).max() <= 1e-12
    UO, lam = rng.standard_normal((nb, 6)), rng.standard_normal((n, 3))
    v = host(ctx.K_apply(dev(r), dev(q), S, dev(UO)))
    assert np.abs(v - O.K_apply(UO[:, :3], UO[:, 3:], r, q, start)).max() <= 1e-12
    FT = host(ctx.KT_apply(dev(r), dev(q), S, dev(lam)))
    F, T = O.KT_apply(lam, r, q, start)
    assert np.abs(FT - np.concatenate([F, T], 1)).max() <= 1e-11


@pytest.mark.parametrize("scale", [1e-155, 1e-100, 1e-16, 1e-14, 1e14, 1e16, 1e100, 1e153])
def test_blob_build_from_quaternions_of_any_length(ctx, scale):
    """Quaternions are normalised whatever their length.  At 1e-155 the squares
    are denormal, good to 5e-14 of their sum: 1e-12 for offsets of a few units."""
    q, theta, start, rho, _ = _case([7] * 50, 3)
    S = torch.as_tensor(start, device="cuda")
    r = host(ctx.blob_positions(dev(q), dev(theta * scale), S, dev(rho)))
    unit = theta / np.linalg.norm(theta, axis=1, keepdims=True)
    assert np.abs(r - O.blob_positions(q, unit, start, rho)).max() <= 1e-12


def test_rotation_matrices_to_the_last_bits(ctx):
    """The frame of a body from the rows of the identity: 2 / |theta|^2 to two ulp,
    two more products and a sum at size 1 or 2, so 8 x 2^-53 an entry."""
    rng = np.random.default_rng(4)
    nb = 4000
    theta = rng.standard_normal((nb, 4)) * 10.0 ** rng.uniform(-20, 20, (nb, 1))
    S = torch.as_tensor(3 * np.arange(nb + 1), device="cuda")
    r = host(ctx.blob_positions(dev(np.zeros((nb, 3))), dev(theta), S, dev(np.tile(np.eye(3), (nb, 1)))))
    L = np.longdouble
    s, x, y, z = (theta.astype(L) / np.sqrt((theta.astype(L) ** 2).sum(1, keepdims=True))).T
    R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y + s * z), 2 * (x * z - s * y),
                  2 * (x * y - s * z), 1 - 2 * (x * x + z * z), 2 * (y * z + s * x),
                  2 * (x * z + s * y), 2 * (y * z - s * x), 1 - 2 * (x * x + y * y)], axis=1)
    assert np.abs(r.reshape(nb, 9) - R).max() <= 8 * 2.0 ** -53
