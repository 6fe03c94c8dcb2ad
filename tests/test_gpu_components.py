"""Every real of the FP64 operator and force keeps FP64 accuracy against its own
terms, however small it is beside the others of its site: colours and real and
imaginary parts that lie decades apart, in links that mix them and in links
that do not.

The bounds are those of FP64 arithmetic, with u = 2^-53 and S the sum of the
magnitudes of a real's terms: 48 products (96 with long links) summed one after
another round by at most 48 u S (96 u S).  A force real has 6 roundings in
w = U a, 4 in its products and 6 in the trace and its third: 16 u S.  In fixed
point w may be off by 2.75 units of 1.5 x 2^50 to its S, 15 u S, and what follows
by 6 u S: 21 u S."""

import numpy as np
import pytest

import fieldgen as fg

pytestmark = pytest.mark.gpu

C3 = -1.0 / 24.0
DIMS = (6, 4, 8, 4)
U = 2.0**-53
LD = np.longdouble


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


def links_of(kind, rng):
    shape = fg.lattice_shape(DIMS) + (4, 3, 3)
    if kind == "haar":
        return fg.random_links(DIMS, "haar", rng)
    u = np.zeros(shape, complex)
    if kind == "phases":
        u[..., range(3), range(3)] = np.exp(1j * rng.uniform(0, 2 * np.pi, shape[:-1]))
    elif kind == "real":
        u[...] = np.linalg.qr(rng.standard_normal(shape))[0]
    else:  # "tiny": one colour feeds the others by 1e-20
        u[...] = np.eye(3) - 1e-20 * (1 - np.eye(3))
    return u


def spread(v, kind, s):
    v = v.copy()
    if kind == "colours":
        v[..., 1:] *= s
    elif kind == "imaginary":
        v.imag *= s
    else:  # one colour alone
        v[..., 1:] = 0
    return v


def parts(a):
    return a.real.astype(LD), a.imag.astype(LD)


def mat_vec(m, v):
    """m v and the sums of its terms' magnitudes, real and imaginary parts."""
    (mr, mi), (vr, vi) = m, v
    vr, vi = vr[..., None, :], vi[..., None, :]
    val = (mr * vr - mi * vi).sum(-1), (mr * vi + mi * vr).sum(-1)
    mag = (abs(mr * vr) + abs(mi * vi)).sum(-1), (abs(mr * vi) + abs(mi * vr)).sum(-1)
    return val, mag


def grid():
    g = np.indices(fg.lattice_shape(DIMS))
    return [g[3], g[2], g[1], g[0]]


def signs(mu, k):
    xyz = grid()
    s = (-1.0) ** sum(xyz[:mu], np.zeros(xyz[0].shape, int))
    return s * np.where((mu == 3) & (xyz[3] + k >= DIMS[3]), -1.0, 1.0)


def exact_dslash(u, w, psi):
    val, mag = [np.zeros(psi.shape, LD) for _ in range(2)], [np.zeros(psi.shape, LD) for _ in range(2)]
    for mu in range(4):
        for k, l, c in ((1, u, LD(1)), (3, w, LD(C3))):
            if l is None:
                continue
            m = parts(l[..., mu, :, :])
            dag = tuple(np.swapaxes(x, -1, -2) * f for x, f in zip(m, (1, -1)))
            s = (signs(mu, k) * c)[..., None]
            here = parts(psi)
            fwd, fm = mat_vec(m, tuple(np.roll(x, -k, axis=3 - mu) for x in here))
            back, bm = mat_vec(dag, here)
            for r in range(2):
                val[r] += s * fwd[r] - np.roll(s * back[r], k, axis=3 - mu)
                mag[r] += abs(s) * fm[r] + np.roll(abs(s) * bm[r], k, axis=3 - mu)
    return np.stack(val, -1), np.stack(mag, -1)


def reals(a):
    return np.stack(parts(a), -1)


def compare(got, plain, val, mag, bound):
    """got and the oracle's plain FP64 against the exact values, by the terms."""
    none = mag == 0
    assert not reals(got)[none].any()
    err = [abs(reals(x) - val)[~none] / mag[~none] for x in (got, plain)]
    assert err[0].max() <= bound * U, err[0].max() / U
    rms = [np.sqrt((e.astype(float) ** 2).mean()) for e in err]
    assert rms[0] <= 1.05 * rms[1], rms


CASES = [(k, "colours", s) for k in ("haar", "phases") for s in (1e-1, 1e-2, 1e-4, 1e-8, 1e-12, 1e-16)]
CASES += [("real", "imaginary", s) for s in (1e-2, 1e-4, 1e-8, 1e-12)] + [("tiny", "one", 0.0)]


@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("links,kind,s", CASES)
def test_dslash_components(q, oracle_mod, naik, links, kind, s):
    """By a site's directions on four threads (qex_dslash at this size) and by
    one thread a site (qex_dslash_mrhs)."""
    rng = np.random.default_rng(21)
    u = links_of(links, rng)
    w = links_of(links, rng) if naik else None
    psi = spread(rng.standard_normal(fg.lattice_shape(DIMS) + (3, 2)).view(complex)[..., 0], kind, s)
    val, mag = exact_dslash(u, w, psi)
    lat = q.Lattice(DIMS)
    fat = q.qex_pack_links(lat, "f64", dev(u))
    lng = q.qex_pack_links(lat, "f64", dev(w)) if naik else None
    for p in (0, 1):
        at = fg.even_mask(DIMS) == (p == 0)
        plain = oracle_mod.dslash_parity(DIMS, u, psi, p, w, C3)[at]
        x = q.qex_pack_field(lat, "f64", 1 - p, dev(psi))
        for out in (q.qex_dslash(lat, "f64", fat, lng, C3, p, x), q.qex_dslash_mrhs(lat, "f64", fat, lng, C3, p, 1, x)):
            got = q.qex_unpack_field(lat, "f64", p, out).cpu().numpy()[at]
            compare(got, plain, val[at], mag[at], 96 if naik else 48)


@pytest.mark.parametrize("links,kind,s", CASES)
def test_force_components(q, oracle_mod, links, kind, s):
    rng = np.random.default_rng(22)
    u = links_of(links, rng)
    z = spread(rng.standard_normal(fg.lattice_shape(DIMS) + (3, 2)).view(complex)[..., 0], kind, s)
    even = fg.even_mask(DIMS)
    x, y = np.where(even[..., None], z, 0), np.where(even[..., None], 0, z)
    plain = oracle_mod.force(DIMS, u, x, y, None, 0.0, 0)[0]
    lat = q.Lattice(DIMS)
    g, _ = q.qex_force(lat, q.qex_pack_links(lat, "f64", dev(u)), None, 0.0, q.qex_pack_field(lat, "f64", 0, dev(x)),
                       q.qex_pack_field(lat, "f64", 1, dev(y)))
    got = q.qex_unpack_links(lat, "f64", g).cpu().numpy()
    here = parts(z)
    b = tuple(t[..., None, :] for t in here)
    for mu in range(4):
        s_mu = (signs(mu, 1) * np.where(even, 1.0, -1.0))[..., None]
        (wr, wi), (nr, ni) = mat_vec(parts(u[..., mu, :, :]), tuple(np.roll(t, -1, axis=3 - mu) for t in here))
        wr, wi, nr, ni = ((s_mu * t)[..., None] for t in (wr, wi, nr, ni))
        m = wr * b[0] + wi * b[1], wi * b[0] - wr * b[1]
        n = abs(nr * b[0]) + abs(ni * b[1]), abs(ni * b[0]) + abs(nr * b[1])
        val = [m[0] - np.swapaxes(m[0], -1, -2), m[1] + np.swapaxes(m[1], -1, -2)]
        mag = [n[0] + np.swapaxes(n[0], -1, -2), n[1] + np.swapaxes(n[1], -1, -2)]
        for t in (val[1], mag[1]):
            t -= (t[..., 0, 0] + t[..., 1, 1] + t[..., 2, 2])[..., None, None] / LD(3) * np.eye(3) * (
                1 if t is val[1] else -1)
        compare(got[..., mu, :, :], plain[..., mu, :, :], np.stack(val, -1), np.stack(mag, -1), 21)
