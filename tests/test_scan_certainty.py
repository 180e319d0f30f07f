"""The binary64 kernel's line scan in binary32, checked on the CPU.

The kernel decides the event of a flight segment (Sect. 2.6) from binary32
path lengths and optical depths wherever every sign involved lies outside an
error bound, and by binary64 frequency thresholds elsewhere.  This file
restates both sides in numpy and asserts, on random segments with near-ties
planted at a line, at the electron-scattering point and at the shell exit,
that every event the binary32 side calls certain is the binary64 scan's: the
scalar scan of a lane, the one-step scan of a 32-line window, and the lone
walk's pick of the first line that absorbs by its own depth, the last also
against the mixed-precision kernel's thresholds.  The binary32 logarithm of the
draws is checked against long double.
"""
import ctypes
import ctypes.util
import math

import numpy as np
import pytest

_libm = ctypes.CDLL(ctypes.util.find_library("m") or "libm.so.6")
_libm.fma.restype = ctypes.c_double
_libm.fma.argtypes = [ctypes.c_double] * 3
fma = _libm.fma
F = np.float32
LINE, ELECTRON, SHELL = 1, 2, 3


def _rz32(x):
    """binary64 -> binary32 toward zero; below the normal range 0, above it inf."""
    b = int(np.float64(x).view(np.uint64))
    e = ((b >> 52) & 0x7FF) - 896
    mag = 0 if e <= 0 else 0x7F800000 if e >= 255 else (e << 23) | ((b >> 29) & 0x7FFFFF)
    return np.uint32(mag | ((b >> 63) << 31)).view(F)


def _f(v):
    return F(v)


def _setup(nu_cmf, D, p, q, kap, inner, xi2, xo2, tau):
    b = int(np.float64(nu_cmf).view(np.uint64))
    mc, ec = (b & ((1 << 52) - 1)) | (1 << 52), b >> 52
    im = F(1) / F(np.uint32(mc >> 29))
    pf, qf = _rz32(p), _rz32(q)
    Df = F(F(1) - pf)
    xb2 = _rz32(xi2 if inner else xo2)
    dq = F(xb2 - qf)
    e1 = F(F(2.0 ** -22) * F(xb2 + dq))
    with np.errstate(invalid="ignore", divide="ignore"):
        r = F(1) / np.sqrt(dq)
        P = F(dq * r)
    lx = F((-P if inner else P) - pf)
    mx = F(F(2.0 ** -20) * F(P + abs(pf)) + F(e1 * r) + F(2.0 ** -44)) if dq >= F(4) * e1 else F(np.inf)
    kf = _rz32(kap)
    return dict(mc=mc, ec=ec, lf=F(F(Df * im) * F(2.0 ** -29)), tf=F(kf * Df), tau=tau, lx=lx, mx=mx)


def _delta(f, nu):
    b = int(np.float64(nu).view(np.uint64))
    sh = f["ec"] - (b >> 52)
    d = f["mc"] - (((b & ((1 << 52) - 1)) | (1 << 52)) >> min(max(sh, 0), 63))
    v = F(F(np.uint32((d >> 32) & 0xFFFFFFFF)) * F(2.0 ** 32) + F(np.uint32(d & 0xFFFFFFFF)))
    return (v if d > 0 else F(0)), sh >= 0


def _scalar(f, nu, tau, scale):
    """A lane's scan: (event or 0 for doubt, line)."""
    rem, m1, m0 = f["tau"], F(2.0 ** -19), F(f["tf"] * F(2.0 ** -44) + F(2.0 ** -100))
    j = 0
    while True:
        at_exit = j >= len(nu)
        if not at_exit:
            d, ok = _delta(f, nu[j])
            l = F(d * f["lf"])
            a = F(l * f["tf"])
            M = F(F(m1 * F(a + f["tau"])) + m0) * F(scale)
            r0 = F(rem - a)
            if not ok or not r0 > M:
                return 0, j
            xm, xM = F(f["lx"] - l), F(F(2.0 ** -19) * l + f["mx"]) * F(scale)
            if not xm > xM:
                if not xm < -xM:
                    return 0, j
                at_exit = True
            else:
                t = _rz32(tau[j])
                r1 = F(r0 - t)
                if r1 < -M:
                    return LINE, j
                if not r1 > M or t < 0:
                    return 0, j
                rem = F(rem - t)
        if at_exit:
            ax = F(f["lx"] * f["tf"])
            lim = F(m1 * F(abs(ax) + f["tau"]) + F(F(f["tf"] * f["mx"]) + m0)) * F(scale)
            return (SHELL if F(rem - ax) > lim else 0), j
        m1 = F(m1 + F(2.0 ** -23))
        m0 = F(m0 + F(f["tf"] * F(2.0 ** -51)))
        j += 1


def _window(f, nu, tau, scale):
    """The one-step scan of lines 0..31 (None: the whole window is passed)."""
    n = F(32)
    m0 = F(f["tf"] * F(n * F(2.0 ** -51) + F(2.0 ** -44)) + F(2.0 ** -100))
    m1 = F(n * F(2.0 ** -23) + F(2.0 ** -19))
    own = np.array([_rz32(tau[k]) if k < len(nu) else F(0) for k in range(32)], F)
    Px = np.concatenate([[F(0)], own[:-1]]).astype(F)
    for o in (1, 2, 4, 8, 16):
        y = np.concatenate([np.zeros(o, F), Px[:-o]])
        Px = np.where(np.arange(32) >= o, (Px + y).astype(F), Px)
    for k in range(32):
        there = k < len(nu)
        d, ok = _delta(f, nu[k]) if there else (F(0), False)
        l = F(d * f["lf"])
        a = F(l * f["tf"])
        M = F(m1 * F(a + f["tau"]) + m0) * F(scale)
        r0 = F(F(f["tau"] - Px[k]) - a)
        r1 = F(r0 - own[k])
        xm, xM = F(f["lx"] - l), F(F(2.0 ** -19) * l + f["mx"]) * F(scale)
        before, inside = there and ok and r0 > M, xm > xM
        if before and inside and r1 > M and own[k] >= 0:
            continue
        if before and inside and r1 < -M:
            return LINE, k
        ax = F(f["lx"] * f["tf"])
        lim = F(m1 * F(abs(ax) + f["tau"]) + F(F(f["tf"] * f["mx"]) + m0)) * F(scale)
        if (not there or (ok and xm < -xM)) and F(F(f["tau"] - Px[k]) - ax) > lim:
            return SHELL, k
        return 0, k
    return None


def _thick(f, nu, tau, scale, inside_first=True):
    """The lone walk's shortcut: the first line whose own depth absorbs, the
    depths before it as one integer sum (None: not settled)."""
    M_ = [None] * 32
    prior = 0
    for k in range(min(32, len(nu))):
        d, ok = _delta(f, nu[k])
        l = F(d * f["lf"])
        a = F(l * f["tf"])
        own = _rz32(tau[k])
        M = F(F(F(2.0 ** -19) + F(2.0 ** -18)) * F(a + f["tau"]) + F(F(f["tf"] * F(2.0 ** -43)) + F(2.0 ** -100)))
        M = F(M * F(scale))
        left = F(f["tau"] - a)
        if ok and F(left - own) < -M:
            rk = F(left - F(F(prior) * F(2.0 ** -21)))
            inside = F(f["lx"] - l) > F(F(2.0 ** -19) * l + f["mx"]) * F(scale)
            slack = F(2.0 ** -15) * F(scale)
            return (LINE, k) if (inside or (k == 0 and not inside_first)) and rk > M + slack and l > 2.0 ** -40 else None
        if own < 0:
            return None
        prior += int(F(min(own, F(63)) * F(2.0 ** 21)))
    return None


def _exact_mixed(nu_lab, pp, q, kap, inner, xi2, xo2, tau0, nu, tau):
    """The mixed-precision kernel's scan (binary32 geometry, depths and c_e,
    binary64 thresholds); None where its first line is placed against the exit
    by the event point instead."""
    Df = F(F(1) - pp)
    nu_cmf = nu_lab * float(Df)
    b = float(_rz32(nu_lab))
    c_e = F(F(F(b) * F(1.0 / float(kap))) * F(F(1) / Df)) if kap > 0 else F(0)
    root = np.sqrt(max(F((xi2 if inner else xo2) - q), F(0)))
    key_x = nu_lab * float(F(F(1) - (-root if inner else root)))
    thr, rem, j = nu_cmf - float(F(tau0 * c_e)), tau0, 0
    while j < len(nu):
        if (kap > 0 and nu[j] <= thr) or (j > 0 and nu[j] <= key_x):
            return SHELL, j
        if kap > 0:
            t = thr + float(F(F(tau[j]) * c_e))
            if t > nu[j]:
                return LINE, j
            thr = t
        else:
            if F(tau[j]) > rem:
                return LINE, j
            rem = F(rem - F(tau[j]))
        if nu[j] <= key_x:
            return SHELL, j
        j += 1
    return SHELL, j


def _exact(nu_cmf, D, p, q, kap, inner, xi2, xo2, tau0, nu, tau):
    """The binary64 scan: frequency thresholds."""
    nu_lab = nu_cmf * (1.0 / D)
    root = math.sqrt(max((xi2 if inner else xo2) - q, 0.0))
    key_x = nu_lab * (1.0 - (-root if inner else root))
    rem, thr = tau0, -math.inf
    if kap > 0:
        c_e = (nu_lab * (1.0 / kap)) * (1.0 / D)
        thr = fma(-tau0, c_e, nu_cmf)
    j = 0
    while j < len(nu):
        if nu[j] <= thr or nu[j] <= key_x:
            break
        if kap > 0:
            t = fma(tau[j], c_e, thr)
            if t > nu[j]:
                return LINE, j
            thr = t
        else:
            if tau[j] > rem:
                return LINE, j
            rem -= tau[j]
        j += 1
    return (ELECTRON if thr > key_x else SHELL), j


def _segments(n, seed):
    r = np.random.default_rng(seed)
    for _ in range(n):
        xi = r.uniform(0.02, 0.05)
        xo = xi * (1 + 10 ** r.uniform(-3, -0.3))
        x = r.uniform(xi, xo) if r.random() < 0.8 else (xi if r.random() < 0.5 else xo)
        mu = r.uniform(-1, 1)
        p = x * mu
        q = max(fma(-p, p, x * x), 0.0)
        inner = p < 0 and q <= xi * xi
        D = 1.0 - p
        lexit = (-1 if inner else 1) * math.sqrt(max((xi * xi if inner else xo * xo) - q, 0)) - p
        nu_cmf = 10 ** r.uniform(14, 15.5)
        nu_lab = nu_cmf / D
        m = int(r.integers(0, 40))
        span = max(lexit, 1e-9) * 10 ** r.uniform(-3, 0.5)
        ls = np.sort(r.uniform(0, span, m))
        if m and r.random() < 0.3:  # a line at the exit
            ls[int(r.integers(m))] = max(lexit, 0.0) * (1 + r.choice([-1, 1]) * 10 ** r.uniform(-16, -3))
            ls.sort()
        nu = nu_cmf - ls * nu_lab
        nu = np.array(sorted(set(float(v) for v in nu), reverse=True))
        m = len(nu)
        tau = np.exp(r.uniform(-6, 1) + 3 * r.standard_normal(m))
        kap = 0.0 if r.random() < 0.15 else 10 ** r.uniform(-4, 2.5)
        tau0 = -math.log(1.0 - r.random())
        if m and r.random() < 0.6:  # a near-tie: absorbed or not, or d_e at a line
            k = int(r.integers(m))
            at = kap * D * float(np.maximum((nu_cmf - nu[k]) / nu_lab, 0)) + math.fsum(tau[: k + int(r.integers(2))])
            if 0 < at < 36:
                tau0 = at * (1 + r.choice([-1, 1]) * 10 ** r.uniform(-16.5, -4))
        yield nu_cmf, D, p, q, kap, inner, xi * xi, xo * xo, tau0, nu, tau


@pytest.mark.parametrize("seed", range(4))
def test_certain_events_are_the_binary64_scans(seed):
    certain = doubt = wrong_small = 0
    for nu_cmf, D, p, q, kap, inner, xi2, xo2, tau0, nu, tau in _segments(1500, seed):
        f = _setup(nu_cmf, D, p, q, kap, inner, xi2, xo2, _rz32(tau0))
        want = _exact(nu_cmf, D, p, q, kap, inner, xi2, xo2, tau0, nu, tau)
        for scan in (_scalar, _window):
            got = scan(f, nu, tau, 1.0)
            if got is None:
                assert want[1] >= 32
            elif got[0]:
                certain += 1
                assert got == want
            else:
                doubt += 1
                assert want[1] >= got[1]  # the lines before the doubt are passed
            small = scan(f, nu, tau, 2.0 ** -8)
            wrong_small += small is not None and small[0] != 0 and small != want
        got = _thick(f, nu, tau, 1.0)
        assert got is None or got == want
    assert certain > 1000 and doubt > 100
    assert wrong_small > 0  # a bound 2^8 times smaller is not one


@pytest.mark.parametrize("seed", range(4))
def test_lone_pick_is_the_mixed_kernels_scan(seed):
    picked = 0
    for nu_cmf, D, p, q, kap, inner, xi2, xo2, tau0, nu, tau in _segments(1500, 100 + seed):
        pp, q32, kap32 = F(p), F(q), F(kap)
        xi2, xo2, tau0 = F(xi2), F(xo2), F(tau0)
        tau = tau.astype(F)
        inner = bool(pp < 0 and q32 <= xi2)
        Df = F(F(1) - pp)
        nu_lab = nu_cmf * (1.0 / float(Df))  # so that nu_cmf is the emitted line's frequency to rounding
        f = _setup(nu_cmf, D, float(pp), float(q32), float(kap32), inner, float(xi2), float(xo2), tau0)
        root = np.sqrt(max(F((xi2 if inner else xo2) - q32), F(0)))
        f["lx"] = F(Df - F(F(1) - (-root if inner else root)))
        f["mx"] = F(2.0 ** -43)
        f["tf"] = F(kap32 * Df)
        got = _thick(f, nu, tau, 1.0, inside_first=False)
        if got is not None:
            picked += 1
            assert got == _exact_mixed(nu_lab, pp, q32, kap32, inner, xi2, xo2, tau0, nu, tau)
    assert picked > 200


def test_binary32_logarithm_of_the_draws():
    """neg_log_u53_f within 2^-21 of -ln(u 2^-53), near 1 included."""
    r = np.random.default_rng(5)
    u = np.concatenate([[1, 2, 3, 2 ** 52 - 1, 2 ** 52, 2 ** 52 + 1, 2 ** 53 - 2, 2 ** 53 - 1, 3 * 2 ** 50, 3 * 2 ** 51],
                        r.integers(1, 2 ** 53, 200_000), 2 ** 53 - 2 ** r.integers(0, 52, 20_000),
                        2 ** r.integers(0, 53, 2000)]).astype(np.uint64)
    lz = 63 - np.floor(np.log2(u.astype(np.longdouble))).astype(np.int64)
    m = u << lz.astype(np.uint64)
    up = m >= np.uint64(0xC000000000000000)
    a = np.where(up, np.uint64(0) - m, m - np.uint64(1 << 63))
    mag = ((a >> np.uint64(32)).astype(np.uint32).astype(F) * F(2.0 ** 32) + (a & np.uint64(0xFFFFFFFF)).astype(np.uint32).astype(F))
    f = np.where(up, mag * F(-(2.0 ** -64)), mag * F(2.0 ** -63)).astype(F)
    s = f * (F(1) / (F(2) + f))
    s2 = s * s
    q = s2 * F(1 / 9) + F(1 / 7)
    q = s2 * q + F(0.2)
    q = s2 * q + F(1 / 3)
    lnm = F(2) * ((s * s2) * q + s)
    got = (lz - 10 - up).astype(F) * F(float.fromhex("0x1.62e43p-1")) - lnm
    want = -np.log(u.astype(np.longdouble) * np.longdouble(2.0) ** -53)
    assert np.all(got >= 0)
    rel = np.abs(got.astype(np.longdouble) - want) / np.where(want == 0, 1, want)
    assert rel.max() < 2.0 ** -21, float(rel.max())
