"""The closed form of u and the rounding of its tables, on the host (no GPU).

snap_pair_host evaluates S = Re Y : conj(u) of a pair as the fused dE kernel
does.  Against the layer recursion in extended precision, over pairs spread
evenly on the sphere, its error has a random part, which averages out over an
atom's pairs, and one that is the same function of (a, b) for every atom, from
the tables.  The elements of u are orthogonal on the sphere, so the second part
is found by projecting the error on them.
"""
import numpy as np
import pytest

EPS = {0: 2.0 ** -53, 1: 2.0 ** -24}


@pytest.fixture(scope="module")
def snapmod():
    from paper_2011_12875_gb300 import build, snap
    build.build()
    snap.load()
    return snap


def layers(twojmax, a, b, da=None, db=None):
    """u_t [n][t+1][t+1] of every pair, in extended precision, and its
    derivative along (da, db)."""
    col = lambda v: None if v is None else np.conj(v)[:, None, None]  # noqa: E731
    ca, cb, cda, cdb = col(a), col(b), col(da), col(db)
    u = np.ones((len(a), 1, 1), dtype=a.dtype)
    du = np.zeros_like(u)
    out, dout = [u], [du]
    for t in range(1, twojmax + 1):
        ma, mb = np.arange(t + 1), np.arange(t)
        up = np.sqrt((t - ma[:t, None]) / (t - mb[None, :]).astype(np.longdouble))
        dn = np.sqrt(ma[1:, None] / (t - mb[None, :]).astype(np.longdouble))
        sign = np.array([(-1.0) ** (t + m) for m in range(t + 1)])

        def whole(first, second):
            full = np.zeros((len(a), t + 1, t + 1), dtype=a.dtype)
            full[:, :t, :t] += up * first
            full[:, 1:, :t] -= dn * second
            full[:, :, t] = sign * np.conj(full[:, ::-1, 0])
            return full

        if da is not None:
            du = whole(cda * u + ca * du, cdb * u + cb * du)
        u = whole(ca * u, cb * u)
        out.append(u)
        dout.append(du)
    return out, dout


def full_y(snapmod, twojmax, y):
    """Half layout -> [t][ma][mb], the other columns by the inversion symmetry."""
    out = []
    for t in range(twojmax + 1):
        m = np.zeros((t + 1, t + 1), dtype=np.clongdouble)
        for ma in range(t + 1):
            for mb in range(t + 1):
                below = 2 * mb > t or (2 * mb == t and ma > mb)
                h = y[snapmod.half_index(twojmax, t, *((t - ma, t - mb) if below else (ma, mb)))]
                v = h[0] + 1j * h[1]
                m[ma, mb] = (-1) ** (ma + mb) * np.conj(v) if below else v
        out.append(m)
    return out


def sphere(rng, n):
    v = rng.normal(size=(n, 4))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def random_y(snapmod, twojmax, rng):
    y = rng.normal(size=(snapmod.half_size(twojmax), 2))
    for t in range(0, twojmax + 1, 2):  # the centre is real or imaginary by the symmetry
        y[snapmod.half_index(twojmax, t, t // 2, t // 2), 1] = 0.0
    return y


def along(o, ab, tan):
    """The derivative along tan from snap_pair_host's sums."""
    g = o[:, 1:5].copy()
    g[:, :2] += 4 * o[:, 5:] * ab[:, :2]
    return (g * tan).sum(1)


def contract(u, yf):
    return sum((np.conj(ut) * yt).real.sum((1, 2)) for ut, yt in zip(u, yf))


# The error that all pairs share, relative to the root mean square over them: a
# scale, its product with Y and the sums of fix_class are rounded once each, by
# 0.41 EPS (EPS / sqrt 3 over the mean size of a mantissa) in the root mean square
# and independently from element to element: 0.71 EPS together.  Half as much
# again is allowed; what does not average out over 12000 pairs adds 0.1 to the
# square.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("twojmax", [3, 8, 11, 14])
def test_no_error_is_shared_by_all_pairs(snapmod, twojmax, precision):
    rng = np.random.default_rng(101 + twojmax)
    n = 12000
    ab, y = sphere(rng, n), random_y(snapmod, twojmax, rng)
    if precision == 1:
        ab, y = (x.astype(np.float32).astype(np.float64) for x in (ab, y))
    o = snapmod.pair_host(twojmax, ab, y, precision=precision)
    g = ab.astype(np.longdouble)
    # along (a, b) -> (a cos + b sin, b cos - a sin)
    tan = np.stack([ab[:, 2], ab[:, 3], -ab[:, 0], -ab[:, 1]], axis=1)
    a, b = g[:, 0] + 1j * g[:, 1], g[:, 2] + 1j * g[:, 3]
    u, du = layers(twojmax, a, b, b, -a)
    yf = full_y(snapmod, twojmax, y)
    for name, got, ref in (("value", o[:, 0], contract(u, yf)), ("derivative", along(o, ab, tan), contract(du, yf))):
        err = (got - ref).astype(np.float64)
        unit = float(np.sqrt((ref * ref).mean())) * EPS[precision]
        # the projections from each half of the pairs: their product has no noise on average
        shared = 0.0
        for t, ut in enumerate(u):
            v = ut.astype(np.complex128).reshape(n, -1)
            c = [v[h::2].conj().T @ err[h::2] / (n / 2) * (t + 1) for h in (0, 1)]
            shared += float((c[0].conj() * c[1]).real.sum()) / (t + 1)
        print(f"2J{twojmax} prec {precision} {name}: rms {np.sqrt((err * err).mean()) / unit:.2f} eps, "
              f"shared {np.sign(shared) * np.sqrt(abs(shared)) / unit:.2f} eps")
        assert shared <= (1.1 * unit) ** 2, name


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("twojmax", list(range(0, 15)))
def test_value_and_gradient(snapmod, twojmax, precision):
    """S and its derivative along a tangent of the sphere, against the recursion:
    up to about 40 roundings of the size of the largest sum for each of 2J
    steps."""
    rng = np.random.default_rng(7 + twojmax)
    n = 40
    ab, y = sphere(rng, n), random_y(snapmod, twojmax, rng)
    if precision == 1:
        ab, y = (x.astype(np.float32).astype(np.float64) for x in (ab, y))
    o = snapmod.pair_host(twojmax, ab, y, precision=precision)
    g = ab.astype(np.longdouble)
    tan = rng.normal(size=(n, 4))
    tan -= (tan * ab).sum(1, keepdims=True) * ab / (ab * ab).sum(1, keepdims=True)
    tan /= np.linalg.norm(tan, axis=1, keepdims=True)
    u, du = layers(twojmax, *(x[:, 2 * k] + 1j * x[:, 2 * k + 1] for x in (g, tan.astype(np.longdouble)) for k in (0, 1)))
    yf = full_y(snapmod, twojmax, y)
    ref, d = contract(u, yf), contract(du, yf)
    tol = 40 * (twojmax + 1) * EPS[precision]
    assert np.abs(o[:, 0] - ref).max() <= tol * np.abs(ref).max()
    assert np.abs(along(o, ab, tan) - d).max() <= tol * ((twojmax + 1) * np.abs(ref).max() + np.abs(d).max())


@pytest.mark.parametrize("precision", [0, 1])
def test_no_error_is_shared_by_all_atoms(snapmod, precision):
    """One element of Y at a time, with many values: the error of its share of S,
    projected on that share, is the same for every atom only by the tables.  In
    FP32 these have what their rounding leaves off beside them, which a kernel may
    round away again; in FP64 the scale's own rounding is left, 0.41 EPS.  3000
    pairs with rounding errors of up to 4 EPS each leave 4 / sqrt(3000) = 0.07 EPS in a
    value's projection and the value's own product, 0.41 EPS, sqrt(12) less in the
    mean of twelve, 0.14 together: twice that is allowed beside the scale's."""
    twojmax, n = 11, 3000
    rng = np.random.default_rng(1)
    ab = sphere(rng, n)
    if precision == 1:
        ab = ab.astype(np.float32).astype(np.float64)
    g = ab.astype(np.longdouble)
    u, _ = layers(twojmax, g[:, 0] + 1j * g[:, 1], g[:, 2] + 1j * g[:, 3])
    els = [(t, ma, mb) for t in range(twojmax + 1) for mb in range(t // 2 + 1) for ma in range(t + 1)
           if not (2 * mb == t and ma > mb)]
    rng.shuffle(els)
    gain = []
    for t, ma, mb in els[:40]:
        weight, got = 2 if 2 * mb < t or ma < mb else 1, []
        for _ in range(12):
            y = np.zeros((snapmod.half_size(twojmax), 2))
            val = 1.0 + rng.random()
            val = float(np.float32(val)) if precision == 1 else val
            y[snapmod.half_index(twojmax, t, ma, mb), 0] = val
            ref = weight * val * u[t][:, ma, mb].real
            err = (snapmod.pair_host(twojmax, ab, y, precision=precision)[:, 0] - ref).astype(np.float64)
            got.append((err * ref).sum() / (ref * ref).sum() / EPS[precision])
        gain.append(np.mean(got))
    assert np.sqrt(np.mean(np.square(gain))) <= (0.28 if precision == 1 else (0.41 ** 2 + 0.28 ** 2) ** 0.5)
