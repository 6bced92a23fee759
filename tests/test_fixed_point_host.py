"""The fixed-point and FP32-first arithmetic of the FP64 kernels on the host
(tests/fx_host.py), without a GPU."""
import ctypes

import numpy as np
import pytest

from tests import fx_host

D = ctypes.c_double


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return fx_host.load(tmp_path_factory.mktemp("fx_host"))


def truth(u, f, s, c):
    """+1 inside, -1 outside the cone, by the exact sign of c E - |F| of u + s f in 80
    bits; values scaled to E first, so that no square leaves the range."""
    u, f = u.astype(np.longdouble), f.astype(np.longdouble)
    p = u + np.longdouble(s) * f
    E, T = p[:, 0], p[:, 3]
    x, y = p[:, 1] / np.longdouble(c), p[:, 2] / np.longdouble(c)
    size = np.maximum(np.maximum(np.abs(E), np.abs(x)), np.maximum(np.abs(y), np.longdouble(1e-4000)))
    inside = (E > 0) & (T > 0) & ((x / size) ** 2 + (y / size) ** 2 <= (E / size) ** 2)
    return np.where(inside, 1, -1)


@pytest.mark.parametrize("s", [0.25, 1.0, 2e6, 2e-12, 1e-36, 1e20])
@pytest.mark.parametrize("c", [1.0, 2.99792458e10, 1e-11, 2.99792458e3, 1e-18, 1e30])
def test_sure_answers_are_right(host, c, s):
    """Whatever the units, an answer given without doubt is the exact one: states of
    E from 1e-40 to 1e40 (single sizes and spread), fluxes from deep inside the cone to ten
    times its length, right-hand sides from nothing to a thousand times the state."""
    rng = np.random.default_rng(7)
    n = 4000
    for lo, hi in ((-1, 1), (5, 12), (-16, -11), (-40, 40)):
        u, f = np.zeros((n, 4)), np.zeros((n, 4))
        E = 10.0 ** rng.uniform(lo, hi, n)
        for a, amp in ((u, 1.0), (f, 10.0 ** rng.uniform(-20, 3, n) / s)):
            a[:, 0] = E * amp * (1.0 if a is u else rng.uniform(-1, 1, n))
            a[:, 3] = E * amp * (1.0 if a is u else rng.uniform(-1, 1, n))
            phi, r = rng.uniform(0, 2 * np.pi, n), 10.0 ** rng.uniform(-2, 1, n)
            a[:, 1], a[:, 2] = (c * E * amp * r * g(phi) for g in (np.cos, np.sin))
        out = np.zeros(n, np.int32)
        host.host_admissible_sure(n, fx_host.ptr(u), fx_host.ptr(f), D(s), D(c), fx_host.ptr(out))
        t = truth(u, f, s, c)
        assert np.all((out == 0) | (out == t)), (lo, hi, np.flatnonzero((out != 0) & (out != t))[:5])
        if 1e-12 <= s <= 2e6 and 1e-11 <= c <= 1e11 and s <= 1e15 * c and lo >= -12 and hi < 15:
            assert np.mean(out == 0) < 0.01        # ... and it is given


@pytest.mark.parametrize("ratio", [0.5, 0.25, 0.75, 1 / 3, 0.9999, 0.2501])
def test_scaled_pair_product_is_the_nearest(host, ratio):
    """a b / 2^62 rounded to the nearest, ties to even (dyadic ratios tie every other time),
    odd in a, zero at zero: against exact integers."""
    rng = np.random.default_rng(3)
    b = int(ratio * 2 ** 62)
    a = np.concatenate([[0, 1, -1, 2 ** 61 - 1, 1 - 2 ** 61], rng.integers(-2 ** 61, 2 ** 61, 4000),
                        rng.integers(-64, 64, 200), rng.integers(0, 2 ** 50, 800) * 1024]).astype(np.int64)
    out = np.zeros_like(a)
    host.host_product(len(a), fx_host.ptr(a), ctypes.c_longlong(b), fx_host.ptr(out))
    for x, y in zip(a.tolist(), out.tolist()):
        q, r = divmod(abs(x) * b, 2 ** 62)
        q += r > 2 ** 61 or (r == 2 ** 61 and q & 1)
        # the product of the low halves is cut at 2^-31 of a unit
        assert y == (q if x >= 0 else -q) or abs(r - 2 ** 61) < 2 ** 31, (x, y, q)


def neighbours(n, kind, size, seed):
    """[west, east, south, north][E, Fx, Fy] of n cells.  free: four unrelated cells, the flux
    components of sizes of their own, down to `size`; ahead: E equal everywhere, the fluxes at
    `size`; along: cells south and north alike, fluxes along y at `size`."""
    rng = np.random.default_rng(seed)
    E = np.repeat(10.0 ** rng.uniform(-2, 2, (n, 1)), 4, 1)
    F = rng.uniform(-1, 1, (n, 4, 2)) / 1.5
    if kind == "free":
        E = 10.0 ** rng.uniform(-2, 2, (n, 4))
        F *= size ** rng.uniform(0, 1, (n, 4, 2))
    elif kind == "ahead":
        F *= size
    else:
        E[:, :2] = 10.0 ** rng.uniform(-2, 2, (n, 2))
        F[:, :, 1] *= size
        F[:, 3] = F[:, 2]
    return np.concatenate([E[:, :, None], F * E[:, :, None]], 2)


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-9, 1e-15, 1e-20, 1e-60, 1e-200])
@pytest.mark.parametrize("kind", ["free", "ahead", "along"])
def test_sums_keep_small_fluxes(host, kind, size, dim):
    """The sums N_E and N_F / (c b) to a few roundings (16) of their own terms: fluxes, the part
    A of the pressure that goes with them, and of the isotropic rest S / 3 what FP64 leaves.
    FP64 holds that to 2^-54 E, so a pair's difference is in error by as much where E differs;
    where E is equal it drops what is below, f^2 E at most; where the cells are alike it
    cancels.  Reference: 80 bits, with S taken apart, so that it cancels there too."""
    n = 3000
    cells = neighbours(n, kind, size, 9)
    out = np.zeros((n, 3))
    assert host.host_sums(n, dim, fx_host.ptr(cells), fx_host.ptr(out)) == n
    L = np.longdouble
    E, F = cells[:, :, 0].astype(L), [cells[:, :, 1].astype(L), cells[:, :, 2].astype(L)]
    f2 = (F[0] ** 2 + F[1] ** 2) / E ** 2
    sigma = np.sqrt(E * E - 0.75 * (F[0] ** 2 + F[1] ** 2))
    A = [[1.5 * F[a] * F[b] / (E + sigma) for b in range(2)] for a in range(2)]
    tr = A[0][0] + A[1][1]
    ref, terms = np.zeros((3, n), L), np.zeros((3, n), L)
    for a in range(dim):
        lo, hi = 2 * a, 2 * a + 1
        ref[0] += (E[:, lo] + F[a][:, lo]) + (E[:, hi] - F[a][:, hi])
        terms[0] += E[:, lo] + E[:, hi]
        for b in range(2):
            ref[1 + b] += (F[b][:, lo] + A[a][b][:, lo]) + (F[b][:, hi] - A[a][b][:, hi])
            terms[1 + b] += sum(np.abs(x[:, q]) for x in (F[b], A[a][b]) for q in (lo, hi))
        ref[1 + a] += (E[:, lo] - E[:, hi]) / 3 - (tr[:, lo] - tr[:, hi]) / 3
        rest = np.where(E[:, lo] != E[:, hi], E[:, lo] + E[:, hi],
                        E[:, lo] * np.minimum(1, 2.0 ** 53 * np.maximum(f2[:, lo], f2[:, hi])))
        terms[1 + a] += np.where(np.all(cells[:, lo] == cells[:, hi], axis=1), 0, rest) / 3
    err = np.max(np.abs(out.T.astype(L) - ref) / terms, axis=1)
    assert np.all(err <= 16 * 2.0 ** -53), err * 2.0 ** 53


def test_tail_clusters_run_at_once(host):
    """Up to 152 instances: one cluster each on the device's 152 SMs (16 blocks leave room for
    nine, not more), none smaller than that asks for."""
    for count in range(1, 153):
        blocks = host.host_tail_blocks(count)
        assert blocks in (1, 2, 4, 8, 16)
        assert count * blocks <= 152
        assert blocks == 16 or 2 * blocks * count > 128
