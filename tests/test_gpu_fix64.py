"""The FP64 operator's fixed-point hops: values out of their range (which fall
back to FP64 FMAs), zeros of both signs, exact scaling by powers of two, and
accuracy against extended precision."""

import numpy as np
import pytest

import fieldgen as fg
from parity import assert_close

pytestmark = pytest.mark.gpu

C3 = -1.0 / 24.0
DIMS = (6, 4, 8, 4)


@pytest.fixture(scope="module")
def q():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_02750_gb300 import build

    build.build()
    import paper_1612_02750_gb300 as mod

    mod.load()
    return mod


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def inputs(seed, naik):
    s = fg.rng_streams(seed)
    u = fg.random_links(DIMS, "haar", s["links"])
    w = fg.random_links(DIMS, "gauss3", s["long_links"]) if naik else None
    return u, w, fg.gaussian_field(s["source"], DIMS)


def dslash(q, u, w, psi, p):
    lat = q.Lattice(DIMS)
    fat = q.qex_pack_links(lat, "f64", dev(u))
    lng = None if w is None else q.qex_pack_links(lat, "f64", dev(w))
    x = q.qex_pack_field(lat, "f64", 1 - p, dev(psi))
    out = q.qex_unpack_field(lat, "f64", p, q.qex_dslash(lat, "f64", fat, lng, C3, p, x)).cpu().numpy()
    return out[fg.even_mask(DIMS) == (p == 0)]


@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("p", [0, 1])
# in range / at its edge / past it (the FMAs take over): links 2^a, vectors 2^b
@pytest.mark.parametrize("a,b", [(0, 300), (-400, 450), (466, -460), (0, 600), (-520, 3), (500, 500), (-700, 690)])
def test_scaling_by_powers_of_two(q, naik, p, a, b):
    """Scaling links and vectors by powers of two scales the result exactly
    inside the fixed-point range; outside, both sides round on their own (2e-16
    each norm-wise, twice the largest seen for FMAs: 1e-15 together)."""
    u, w, psi = inputs(7, naik)
    ref = dslash(q, u, w, psi, p)
    got = dslash(q, u * 2.0**a, None if w is None else w * 2.0**a, psi * 2.0**b, p)
    got = got * 2.0 ** (-a) * 2.0 ** (-b) if abs(a + b) < 1000 else got * 2.0 ** (-a / 2 - b / 2) * 2.0 ** (-a / 2 - b / 2)
    if max(abs(a), abs(b)) < 460:
        assert np.array_equal(got, ref)
    else:
        assert_close(got, ref, 1e-15, (a, b))


@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("value", [np.inf, np.nan, 1e300, 1e-300, 5e-324, -0.0])
def test_special_values_of_one_site(q, oracle_mod, naik, value):
    """One site of the field, then one link, holds a special value: the sites
    it reaches are those the oracle makes non-finite, and all others agree."""
    u, w, psi = inputs(8, naik)
    f = psi.copy()
    f[1, 2, 3, 1] = value
    v = u.copy()
    v[1, 2, 3, 1, 2, 0, 1] = value
    for uu, ff in ((u, f), (v, psi)):
        for p in (0, 1):
            with np.errstate(all="ignore"):
                ref = oracle_mod.dslash_parity(DIMS, uu, ff, p, w, C3)[fg.even_mask(DIMS) == (p == 0)]
            got = dslash(q, uu, w, ff, p)
            bad = ~np.isfinite(ref).all(-1)
            assert np.array_equal(~np.isfinite(got).all(-1), bad)
            if value != 1e300:
                assert_close(got[~bad], ref[~bad], 1e-13, p)
            else:  # sites with and without the large value, apart
                big = np.abs(ref).max(-1) > 1e200
                assert_close(got[big] * 1e-300 if big.any() else got[~big], ref[big] * 1e-300 if big.any() else ref[~big],
                             1e-13, p)
                assert_close(got[~big], ref[~big], 1e-13, p)


def test_zeros_stay_zero(q):
    """Unit links with zeros of both signs and one non-zero colour: the other
    colours come out as exact zeros."""
    u = np.zeros(fg.lattice_shape(DIMS) + (4, 3, 3), complex)
    u[...] = np.eye(3)
    u = np.where(np.arange(3)[:, None] > np.arange(3), -u, u)  # -0 below the diagonal
    psi = np.zeros(fg.lattice_shape(DIMS) + (3,), complex)
    psi[..., 1] = np.random.default_rng(3).standard_normal(psi.shape[:-1]) * (1 + 0.5j)
    for p in (0, 1):
        out = dslash(q, u, None, psi, p)
        assert not out[:, (0, 2)].any() and out[:, 1].any()


@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("links", ["haar", "unit"])
def test_no_less_accurate_than_fmas(q, oracle_mod, naik, links):
    """Norm-wise error against extended precision at most that of the oracle's
    plain FP64 sums."""
    u, w, psi = inputs(9, naik)
    if links == "unit":
        u = np.zeros_like(u)
        u[...] = np.eye(3)
    L = np.array(DIMS)
    ux, px = u.astype(np.clongdouble), psi.astype(np.clongdouble)
    axes = {0: 3, 1: 2, 2: 1, 3: 0}  # direction -> array axis (t, z, y, x)
    grid = np.indices(fg.lattice_shape(DIMS))
    xyz = [grid[3], grid[2], grid[1], grid[0]]
    acc = np.zeros_like(px)
    for mu in range(4):
        eta = (-1.0) ** sum(xyz[:mu], np.zeros(grid[0].shape, int))
        for k, l, c in ((1, ux, 1.0), (3, None if w is None else w.astype(np.clongdouble), C3)):
            if l is None:
                continue
            s = eta * np.where((mu == 3) & (xyz[3] + k >= L[3]), -1.0, 1.0) * c
            m = l[..., mu, :, :] * s[..., None, None]
            fwd = np.roll(px, -k, axis=axes[mu])
            acc += (m * fwd[..., None, :]).sum(-1)
            back = (np.conj(np.swapaxes(m, -1, -2)) * px[..., None, :]).sum(-1)
            acc -= np.roll(back, k, axis=axes[mu])
    for p in (0, 1):
        sel = fg.even_mask(DIMS) == (p == 0)
        ref = acc[sel]
        got = dslash(q, u, w, psi, p)
        plain = oracle_mod.dslash_parity(DIMS, u, psi, p, w, C3)[sel]
        norm = np.sqrt((np.abs(ref) ** 2).sum())
        err = [np.sqrt((np.abs(v - ref) ** 2).sum()) / norm for v in (got, plain)]
        assert err[0] <= 1.05 * err[1], err


@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("kind", [0, 1])
# vectors 2^b: in range, and past it (links, X or Y), where FP64 FMAs take over
@pytest.mark.parametrize("a,b,c", [(0, 0, 0), (60, -40, 35), (-500, 0, 0), (0, 480, -480), (0, -300, -300)])
def test_force_scales(q, oracle_mod, naik, kind, a, b, c):
    """Force and gradient of scaled links and vectors against the oracle's of
    the unscaled ones (FP64: 1e-13 as in the force's own tests)."""
    u, w, x = inputs(10, naik)
    y = inputs(11, naik)[2]
    lat = q.Lattice(DIMS)
    fat = q.qex_pack_links(lat, "f64", dev(u * 2.0**a))
    lng = None if w is None else q.qex_pack_links(lat, "f64", dev(w * 2.0**a))
    fx = q.qex_pack_field(lat, "f64", 0, dev(x * 2.0**b))
    fy = q.qex_pack_field(lat, "f64", 1, dev(y * 2.0**c))
    got = q.qex_force(lat, fat, lng, C3, fx, fy, kind=kind)
    even = fg.even_mask(DIMS)[..., None]
    ref = oracle_mod.force(DIMS, u, np.where(even, x, 0), np.where(even, 0, y), w, C3, kind)
    shift = -b - c - (a if kind == 0 else 0)
    for g, r in zip(got, ref):
        if r is not None and g is not None:
            v = q.qex_unpack_links(lat, "f64", g).cpu().numpy()
            assert_close(v * 2.0 ** (shift / 2) * 2.0 ** (shift / 2), r, 1e-13, (kind, a, b, c))


@pytest.mark.parametrize("value", [np.inf, np.nan, 0.0])
def test_force_special_values(q, oracle_mod, value):
    """A colour vector of one site all `value`: the links it reaches are
    non-finite (or zero), and no others."""
    u, _, x = inputs(12, False)
    y = inputs(13, False)[2]
    x[1, 2, 3, 2] = value  # an even site
    lat = q.Lattice(DIMS)
    fat = q.qex_pack_links(lat, "f64", dev(u))
    g, _ = q.qex_force(lat, fat, None, C3, q.qex_pack_field(lat, "f64", 0, dev(x)),
                       q.qex_pack_field(lat, "f64", 1, dev(y)), kind=0)
    got = q.qex_unpack_links(lat, "f64", g).cpu().numpy()
    even = fg.even_mask(DIMS)
    xe = np.where(even[..., None], x, 0)
    with np.errstate(all="ignore"):
        ref = oracle_mod.force(DIMS, u, xe, np.where(even[..., None], 0, y), None, C3, 0)[0]
    bad = ~np.isfinite(ref).all((-1, -2))
    assert np.array_equal(~np.isfinite(got).all((-1, -2)), bad)
    assert_close(got[~bad], ref[~bad], 1e-13)


@pytest.mark.parametrize("links", ["haar", "unit"])
def test_force_no_less_accurate_than_fp64(q, oracle_mod, links):
    """F = 2 TA(U G): norm-wise error against extended precision at most that
    of the oracle's plain FP64 arithmetic."""
    u, _, x = inputs(14, False)
    y = inputs(15, False)[2]
    if links == "unit":
        u = np.zeros_like(u)
        u[...] = np.eye(3)
    even = fg.even_mask(DIMS)
    x, y = np.where(even[..., None], x, 0), np.where(even[..., None], 0, y)
    plain = oracle_mod.force(DIMS, u, x, y, None, 0.0, 0)[0]
    lat = q.Lattice(DIMS)
    g, _ = q.qex_force(lat, q.qex_pack_links(lat, "f64", dev(u)), None, 0.0, q.qex_pack_field(lat, "f64", 0, dev(x)),
                       q.qex_pack_field(lat, "f64", 1, dev(y)))
    got = q.qex_unpack_links(lat, "f64", g).cpu().numpy()
    z = (x + y).astype(np.clongdouble)  # X on even, Y on odd sites
    grid = np.indices(fg.lattice_shape(DIMS))
    xyz = [grid[3], grid[2], grid[1], grid[0]]
    ref = np.empty(u.shape, np.clongdouble)
    for mu in range(4):
        s = (-1.0) ** sum(xyz[:mu], np.zeros(grid[0].shape, int)) * np.where(even, 1.0, -1.0)
        s = s * np.where((mu == 3) & (xyz[3] + 1 >= DIMS[3]), -1.0, 1.0)
        there = np.roll(z, -1, axis=3 - mu) * s[..., None]
        w = (u[..., mu, :, :].astype(np.clongdouble) * there[..., None, :]).sum(-1)
        m = w[..., :, None] * np.conj(z)[..., None, :]
        m = m - np.conj(np.swapaxes(m, -1, -2))
        tr = (m[..., 0, 0] + m[..., 1, 1] + m[..., 2, 2]) / np.longdouble(3)
        ref[..., mu, :, :] = m - tr[..., None, None] * np.eye(3)
    err = [np.sqrt((np.abs(v - ref) ** 2).sum() / (np.abs(ref) ** 2).sum()) for v in (got, plain)]
    assert err[0] <= 1.05 * err[1] and err[1] < 1e-15, err
