"""The direction between two points from their positions split into two floats
each, as the adaptive ray set's screen forms it (k_rays.cu, split_direction),
restated in NumPy float32: wherever it is accepted, its z and azimuth lie within
what the screen's bounds take for the inputs (z: 10u |z| + 0.1u less the 3.5u |z|
of the operations; azimuth: 3.3u), near and far from the coordinate origin, for
neighbouring points, and coincident points are never accepted.  Without the
limit on the smallest direction the bounds fail.  CPU only."""
import numpy as np

f32 = np.float32
U = 2.0 ** -24


def split(x):
    hi = x.astype(f32)
    return hi, (x - hi.astype(np.float64)).astype(f32)


def direction(x, o, X, limit=2.0 ** -17):
    (h, l), (oh, ol) = split(x), split(o)
    d = ((h - oh).astype(f32) + (l - ol).astype(f32)).astype(f32)
    hor = np.abs(d[:, :2]).max(1)
    M = np.abs(d).max(1)
    return d, (M >= f32(limit) * X) & (hor >= f32(0.0625) * M) & (M > 1e-15) & (M < 1e15)


def errors(d, x, o):
    e = x - o  # the definition's double differences
    d = d.astype(np.float64)
    z = lambda v: v[:, 2] / np.sqrt((v * v).sum(1))
    dphi = np.arctan2(d[:, 1], d[:, 0]) - np.arctan2(e[:, 1], e[:, 0])
    dphi = np.abs((dphi + np.pi) % (2 * np.pi) - np.pi)
    return np.abs(z(d) - z(e)), np.abs(z(e)), dphi


def pairs(rng, n, scale):
    o = rng.normal(size=(n, 3)) * scale + rng.choice([0.0, 1e3, -1e6]) * scale
    step = scale * 10.0 ** rng.uniform(-7, 0.5, (n, 1))
    x = o + rng.normal(size=(n, 3)) * step * 10.0 ** rng.uniform(-4, 0, (n, 3))
    x[: n // 50] = o[: n // 50]
    return x, o


def test_split_directions_lie_within_the_bounds():
    rng = np.random.default_rng(8)
    taken = 0
    for scale in (1.0, 1e-6, 1e9):
        for _ in range(4):
            x, o = pairs(rng, 40000, scale)
            X = f32(max(np.abs(x).sum(1).max(), np.abs(o).sum(1).max()))
            d, ok = direction(x, o, X)
            same = (x == o).all(1)
            assert not ok[same].any()
            ez, z, ephi = errors(d[ok], x[ok], o[ok])
            taken += int(ok.sum())
            assert (ez <= 6.5 * U * z + 0.1 * U).all()
            assert (ephi <= 3.3 * U).all()
    assert taken > 20000


def test_without_the_limit_the_bounds_fail():
    rng = np.random.default_rng(9)
    x, o = pairs(rng, 40000, 1.0)
    X = f32(max(np.abs(x).sum(1).max(), np.abs(o).sum(1).max()))
    d, ok = direction(x, o, X, limit=0.0)
    ok &= ~(x == o).all(1)
    _, _, ephi = errors(d[ok], x[ok], o[ok])
    assert (ephi > 3.3 * U).any()


def scaled(x, o):
    """Positions times the power of two that brings the largest |x|_1 to [1, 2), and that largest value."""
    X = max(np.abs(x).sum(1).max(), np.abs(o).sum(1).max())
    s = 2.0 ** -np.floor(np.log2(float(f32(X))))
    return x * s, o * s, f32(X * s)


def scaled_direction(e):
    """From the double differences, by the largest component's power of two (components below 2^-100 of it 0)."""
    top = np.frexp(np.abs(e).max(1))[1][:, None]
    d = np.ldexp(e, 1 - top)
    return np.where(np.abs(d) < 2.0 ** -99, 0.0, d).astype(f32)


def test_any_unit_of_length():
    """Scaled positions: as many directions as in plain units, within the same bounds, whatever the unit."""
    counts = set()
    x, o = pairs(np.random.default_rng(21), 40000, 1.0)
    for k in (-97, -53, -20, 0, 20, 53, 90):
        xs, os_, X = scaled(x * 2.0 ** k, o * 2.0 ** k)
        d, ok = direction(xs, os_, X)
        assert not ok[(x == o).all(1)].any()
        ez, z, ephi = errors(d[ok], x[ok], o[ok])
        assert (ez <= 6.5 * U * z + 0.1 * U).all() and (ephi <= 3.3 * U).all()
        counts.add(int(ok.sum()))
    X = f32(max(np.abs(x).sum(1).max(), np.abs(o).sum(1).max()))
    assert counts == {int(direction(x, o, X)[1].sum())}


def test_directions_from_double_differences():
    """Where the split positions do not carry it: within the bounds for every direction, near points of a far
    mesh and directions along the axis included."""
    rng = np.random.default_rng(22)
    for scale in (1e-28, 1.0, 1e28):
        x, o = pairs(rng, 40000, scale)
        x[:2000] = o[:2000] + np.stack([np.zeros(2000), np.zeros(2000), rng.normal(size=2000) * scale], 1)
        use = ~(x == o).all(1)
        d = scaled_direction((x - o)[use])
        ez, z, ephi = errors(d, x[use], o[use])
        assert (ez <= 6.5 * U * z + 0.1 * U).all() and (ephi <= 3.3 * U).all()
