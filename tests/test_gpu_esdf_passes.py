"""The distance transform's passes against a plain minimum in integers: the grid sizes lie on both sides
of the rule between scanning whole lines and searching by levels, with lines that fill no warp, runs of
every length, grids that are mostly free and mostly occupied, and rows of up to 1024 voxels.

Squared distances are integers on both sides and the field is voxel * sqrt(q) with one rounding each, so
the fields are equal bit for bit."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P

pytestmark = pytest.mark.gpu

FAR = 1 << 40


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2503_06757_gb300 import build
    build.build()


def nearest_sq(sites):
    """Squared distance of every voxel to the nearest site: one minimum per axis."""
    f = np.where(sites, 0, FAR).astype(np.int64)
    for axis in range(3):
        i = np.arange(f.shape[axis])
        shape = [1, 1, 1]
        shape[axis] = -1
        best = np.full_like(f, FAR)
        for t in i:
            best = np.minimum(best, f.take([t], axis) + ((i - t) ** 2).reshape(shape))
        f = best
    return f


def runs(rng, shape, mean, start):
    """Alternating runs of about `mean` voxels along x, some rows without any change."""
    occ = (np.cumsum(rng.random(shape) < 1.0 / mean, axis=2) + start) % 2
    occ[rng.random(shape[:2]) < 0.2] = start
    return occ.astype(np.uint8)


@pytest.mark.parametrize("dims", [
    (31, 33, 40), (64, 64, 64), (65, 66, 67),             # cubes around the rule's line
    (67, 68, 69), (40, 101, 90), (36, 103, 100),          # ... and every remainder of the levels' last step
    (1024, 5, 7), (3, 1024, 24), (37, 3, 1024),           # the longest line along each axis: scanned
    (2, 1024, 40), (40, 2, 1024),                         # ... and searched by levels
    (130, 131, 25), (129, 24, 120), (33, 250, 96), (2, 2, 2),
])
@pytest.mark.parametrize("kind", ["free", "occupied", "mixed", "sparse"])
def test_transform_equals_plain_minimum(dims, kind):
    rng = np.random.default_rng(sum(dims))
    shape = dims[::-1]
    if kind == "sparse":
        occ = np.zeros(shape, np.uint8)
        occ.reshape(-1)[rng.integers(0, occ.size, 3)] = 1
    else:
        occ = runs(rng, shape, {"free": 30, "occupied": 30, "mixed": 2}[kind], 1 if kind == "occupied" else 0)
        if kind != "mixed":  # thin walls of the other kind
            keep = rng.random(shape) < 0.1
            occ = np.where(keep, occ, 1 if kind == "occupied" else 0).astype(np.uint8)
    voxel = np.float32(0.03)
    got = P.Env.from_occupancy(occ, (0.0, 0.0, 0.0), float(voxel)).esdf()
    o = occ != 0
    q = np.where(o, nearest_sq(~o), nearest_sq(o))
    mag = voxel * np.sqrt(q.astype(np.float32))
    diag = voxel * np.sqrt(np.float32(sum(np.float32(d) * np.float32(d) for d in dims)))
    mag = np.where(q >= FAR // 2, diag, mag).astype(np.float32)
    np.testing.assert_array_equal(got, np.where(o, -mag, mag))
