"""The device FP64 diagnostics and the collision's reciprocal, against independent sums.

tclbm_diagnostics() returns, from FP64 block reductions on the device: out[0] sum rho,
out[1..2] sum rho u, out[3] sum h_bar (total energy), out[4] the kinetic energy
sum rho |u|^2 / 2 (Section V.D), out[5] sum u_y (T - T_ref) (the Nusselt sum of
Section V.D), out[6] sum |u - u_snap|^2 and out[7] sum |u|^2 (the residual E_R of
Section V.A).  Each is checked two ways: against the same sum formed on the host from
the lattice's own FP64 moments (the reduction itself: summation order only), and
against the sum formed from the FP64 oracle's fields after the same steps (the state:
the FP32 parity of the fields carried into each sum).
"""
import numpy as np
import pytest

import oracle
from paper_1610_07114_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1610_07114_gb300 import build

    build.build()
    from paper_1610_07114_gb300 import tclbm

    return tclbm


def sums(m, h, T_ref, usnap):
    """The eight diagnostics from FP64 fields, and the sums of the magnitudes of their terms."""
    r, vx, vy, t = m["rho"], m["ux"], m["uy"], m["T"]
    terms = [r, r * vx, r * vy, None, 0.5 * r * (vx * vx + vy * vy), vy * (t - T_ref),
             (vx - usnap[0]) ** 2 + (vy - usnap[1]) ** 2, vx * vx + vy * vy]
    out = np.zeros(8)
    mag = np.zeros(8)
    for k, a in enumerate(terms):
        if k == 3:
            out[3] = float(h.sum()) if h is not None else 0.0
            mag[3] = float(np.abs(h).sum()) if h is not None else 0.0
        else:
            out[k] = float(a.sum())
            mag[k] = float(np.abs(a).sum())
    return out, mag


CASES = [
    # walls (Zou-He velocity, NEE temperature) and gravity: the bench workload's kind of lattice
    ("rb_walls_gravity", lambda: W.rayleigh_benard(96, 48, Ra=2e4, seed=31, amp=1e-2), 600, 400),
    # periodic, Taylor-Green force field on a thermal lattice
    ("tg_thermal", lambda: W.taylor_green(48, F0=2e-5, nu=0.02, thermal=True), 300, 200),
    # athermal (T = T0 everywhere: out[5] vanishes identically up to the velocity sum)
    ("random_athermal", lambda: W.random_periodic(40, 28, seed=32, force="accel", thermal=False), 150, 100),
]


@pytest.mark.parametrize("name,make,n1,n2", CASES, ids=[c[0] for c in CASES])
def test_device_diagnostics_against_host_and_oracle_sums(T, name, make, n1, n2):
    case, fields = make()
    T_ref = case.get("T_ref", case["T0"])
    lat = T.Lattice(case, fields)
    assert lat.params.T_ref == pytest.approx(T_ref)
    o = oracle.Oracle(case, fields, threads=8)
    lat.step(n1)
    o.step(n1)
    lat.snapshot_velocity()
    g1, o1 = lat.moments(), o.moments()
    # the handle keeps its velocity snapshot in FP32
    us_g = np.stack([g1["ux"].astype(np.float32), g1["uy"].astype(np.float32)]).astype(np.float64)
    us_o = np.stack([o1["ux"], o1["uy"]])
    lat.step(n2)
    o.step(n2)
    dev = lat.diagnostics()
    g2 = lat.moments()
    _, hg = lat.populations()
    lat.close()
    o2 = o.moments()
    host, mag = sums(g2, hg, T_ref, us_g)
    orc, mag_o = sums(o2, o.h if case["thermal"] else None, T_ref, us_o)
    print(name, "device", dev)
    print(name, "oracle", orc)
    for k in range(8):
        # the reduction: the same FP64 node values in another order
        assert abs(dev[k] - host[k]) <= 1e-12 * mag[k] + 1e-300, (name, k, dev[k], host[k])
    # the state: the FP32 field parity (rel-L2 <= 1e-5 on rho, u, T; velocity floored at
    # U_ref, temperature deviations at T_scale) carried into each sum
    n = case["nx"] * case["ny"]
    U, Ts = case["U_ref"], case.get("T_scale", 0.0)
    assert dev[0] == pytest.approx(orc[0], rel=1e-7), name
    if case["thermal"]:
        assert dev[3] == pytest.approx(orc[3], rel=1e-7), name
    for k, floor in ((1, n * U), (2, n * U), (5, n * U * Ts)):
        tol = 2e-5 * max(mag_o[k], floor)
        assert abs(dev[k] - orc[k]) <= tol, (name, k, dev[k], orc[k], tol)
    for k in (4, 7):
        tol = 2e-5 * max(mag_o[k], n * U * U)
        assert abs(dev[k] - orc[k]) <= tol, (name, k, dev[k], orc[k], tol)
    # the residual sum compares velocities n2 steps apart; its reference is the velocity
    # field at n1 (FP32 on the device), so its error is that of u relative to the change
    assert orc[6] > 0
    assert dev[6] == pytest.approx(orc[6], rel=1e-4), name
    # E_R itself, as the serving loop and the paper's steady-state test evaluate it
    er_dev = np.sqrt(dev[6] / dev[7])
    er_orc = np.sqrt(orc[6] / orc[7])
    assert er_dev == pytest.approx(er_orc, rel=1e-4), name


def test_rcp_error_bound(T):
    # the reciprocal the collision takes of R T (~0.1-0.3), mu/p + 1/2 and mu/(p Pr) + 1/2
    # (0.5-4): the hardware approximation refined by one Newton step.  Against the exact
    # 1/x: within 2^-22 relative over [1e-3, 1e2] and on a dense sample of [0.5, 2];
    # against the correctly rounded FP32 quotient: within one ulp.
    import torch

    rng = np.random.default_rng(3)
    x = np.concatenate([np.geomspace(1e-3, 1e2, 400001), rng.uniform(0.5, 2.0, 400000),
                        np.float32(1.0) + np.arange(-2000, 2000) * np.float32(2.0**-23)]).astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    T.tclbm_test_rcp(xd.data_ptr(), yd.data_ptr(), x.size)
    y = yd.cpu().numpy()
    exact = 1.0 / x.astype(np.float64)
    rel = np.abs(y.astype(np.float64) - exact) / exact
    ieee = (np.float32(1.0) / x).astype(np.float32)
    ulps = np.abs(y.view(np.int32).astype(np.int64) - ieee.view(np.int32).astype(np.int64))
    print("rcp: max rel %.3e, mean rel %.3e, max ulps from 1/x %d, equal %.4f" %
          (rel.max(), rel.mean(), ulps.max(), float(np.mean(ulps == 0))))
    assert rel.max() <= 2.0**-22
    assert ulps.max() <= 1
    # deterministic: the same bits on a second evaluation
    yd2 = torch.empty_like(xd)
    T.tclbm_test_rcp(xd.data_ptr(), yd2.data_ptr(), x.size)
    assert torch.equal(yd, yd2)
    with pytest.raises(T.TclbmError):
        T.tclbm_test_rcp(None, None, 5)


def test_population_transfer_rounds_like_host_arithmetic(T):
    # populations in and out: base + float32(x - base), for deviations of every magnitude a
    # float has (zeros, denormals, ties between two floats, overflow to infinity, NaN)
    case, _ = W.random_periodic(64, 9, seed=61)
    lat = T.Lattice(case)  # cleared state: every population at its rest value
    base_f, base_h = lat.populations()
    rng = np.random.default_rng(62)
    mag = 10.0 ** rng.uniform(-47, 39, size=base_f.shape) * rng.choice([-1.0, 1.0], size=base_f.shape)
    ties = (1.0 + (rng.integers(0, 1 << 23, size=base_f.shape) + 0.5) * 2.0 ** -23) * 2.0 ** -10
    d = np.where(rng.random(base_f.shape) < 0.5, mag, ties)
    d[0, 0, :4] = [0.0, -0.0, np.inf, np.nan]
    with np.errstate(over="ignore", invalid="ignore"):
        f, h = base_f + d, base_h + d[::-1]
        lat.set_populations(f, h)
        got_f, got_h = lat.populations()
        want_f = base_f + (f - base_f).astype(np.float32).astype(np.float64)
        want_h = base_h + (h - base_h).astype(np.float32).astype(np.float64)
    lat.close()
    assert np.array_equal(got_f, want_f, equal_nan=True) and np.array_equal(got_h, want_h, equal_nan=True)


@pytest.mark.parametrize("amp", [1e-1, 1e-4, 1e-9, 0.0])
@pytest.mark.parametrize("force", ["none", "accel", "taylor_green"])
def test_moments_of_given_populations_to_the_last_digits(T, force, amp):
    # rho, u and T against extended precision on the same populations: rho and T are O(1)
    # values with about three roundings, u one division of a momentum whose nine terms were
    # summed exactly: 4 and 2 units of 2^-53 of their scale
    case, _ = W.random_periodic(70, 33, seed=63, force=force)
    lat = T.Lattice(case)
    f, h = lat.populations()
    rng = np.random.default_rng(64)
    lat.set_populations(f + amp * rng.uniform(-1, 1, f.shape), h + amp * rng.uniform(-1, 1, h.shape))
    f, h = (a.astype(np.longdouble) for a in lat.populations())
    m, p = lat.moments(), lat.params
    lat.close()
    L = np.longdouble
    rho, ex, ey = f.sum(0), (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    jx, jy = sum(e * v for e, v in zip(ex, f)), sum(e * v for e, v in zip(ey, f))
    Fx = Fy = L(0)
    if force == "accel":
        Fx, Fy = rho * L(np.float32(p.ax)), rho * L(np.float32(p.ay))
    elif force == "taylor_green":
        kx, ky = 2 * np.pi * np.arange(70) / 70, 2 * np.pi * np.arange(33) / 33
        t = [g.astype(np.float32).astype(L) for g in (np.sin(kx), np.cos(kx), np.sin(ky), np.cos(ky))]
        a = L(np.float32(p.famp))
        Fx, Fy = a * t[0][None, :] * t[2][:, None], a * t[1][None, :] * t[3][:, None]
    ux, uy = (jx + Fx / 2) / rho, (jy + Fy / 2) / rho
    c = L(2.0 / (2.0 / (p.gamma - 1.0) * p.R))
    Tn = c * (h.sum(0) / rho - (ux * ux + uy * uy) / 2)
    eps = 2.0 ** -53
    assert float(np.abs(m["rho"] - rho).max()) <= 4 * eps
    assert float(np.abs(m["T"] - Tn).max()) <= 8 * eps * float(np.abs(Tn).max())
    # (the momentum's terms are populations read back in FP64: 2^-55 each for the small ones)
    scale = max(float(np.abs(ux).max()), float(np.abs(uy).max()))
    assert float(np.abs(m["ux"] - ux).max()) <= 2 * eps * scale + 12 * 2.0 ** -55 * (amp < 1e-6)
    assert float(np.abs(m["uy"] - uy).max()) <= 2 * eps * scale + 12 * 2.0 ** -55 * (amp < 1e-6)


def test_division_over_the_whole_exponent_range(T):
    # the quotient of the field conversions against IEEE division: one unit in the last place
    # (a corrected quotient misses the rounded one by at most that), equal for zeros, infinities,
    # NaN, subnormal numbers and where it overflows
    import torch

    rng = np.random.default_rng(65)
    n = 1 << 18
    sign = rng.choice([-1.0, 1.0], n)
    wide = sign * np.ldexp(1 + rng.random(n), rng.integers(-1074, 1024, n).astype(np.int32))
    near = sign * np.ldexp(1 + rng.random(n), rng.integers(-66, 66, n).astype(np.int32))
    special = np.array([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, 1.7e308, -1.7e308,
                        2.0 ** -63, 2.0 ** 64, np.nextafter(2.0 ** 64, 0), 2.0 ** -64, 1e-300, 1e300, 1 / 3, 2.0 ** -850])
    sa, sx = (g.ravel() for g in np.meshgrid(special, np.concatenate([special, near[:400], wide[:400]])))
    a = np.concatenate([wide, near, near, sa, sx])
    x = np.concatenate([near, rng.permutation(near), rng.permutation(wide), sx, sa])
    dev = [torch.as_tensor(v, device="cuda") for v in (a, x)]
    y = torch.empty_like(dev[0])
    T.tclbm_test_div(dev[0].data_ptr(), dev[1].data_ptr(), y.data_ptr(), a.size)
    got = y.cpu().numpy()
    with np.errstate(all="ignore"):
        want = a / x
    plain = ~np.isfinite(want) | (np.abs(want) < 2.0 ** -851) | (np.abs(x) < 2.0 ** -63) | (np.abs(x) >= 2.0 ** 64)
    assert np.array_equal(got[plain], want[plain], equal_nan=True)
    assert np.array_equal(np.signbit(got[want == 0]), np.signbit(want[want == 0]))
    err = np.abs(got[~plain] - want[~plain]) / np.spacing(np.abs(want[~plain]))
    assert err.max() <= 1.0, err.max()
    with pytest.raises(T.TclbmError):
        T.tclbm_test_div(None, None, None, 5)


@pytest.mark.parametrize("thermal", [True, False])
def test_moments_of_infinite_and_of_zero_density(T, thermal):
    # one infinite population, and populations whose sum is exactly zero: the quotients by the
    # density are those of plain arithmetic (0, infinite or NaN), at these nodes alone
    case, _ = W.random_periodic(40, 6, seed=66, force="none", correction=thermal)
    case = dict(case, thermal=thermal)
    lat = T.Lattice(case)
    f, h = lat.populations()
    h = np.zeros_like(f) if h is None else h
    f[:, 2, 3] = [np.inf, 0, 0, 0, 0, 0, 0, 0, 0]
    f[:, 4, 5] = [0, 2.0 ** -10, 2.0 ** -10, -2.0 ** -10, -2.0 ** -10, 0, 0, 0, 0]
    lat.set_populations(f, h if thermal else None)
    f, h2 = lat.populations()
    m = lat.moments()
    lat.close()
    assert f[0, 2, 3] == np.inf and f[:, 4, 5].sum() == 0.0
    assert m["rho"][2, 3] == np.inf and m["ux"][2, 3] == 0.0 and m["uy"][2, 3] == 0.0
    assert m["rho"][4, 5] == 0.0 and m["ux"][4, 5] == np.inf and m["uy"][4, 5] == np.inf
    if thermal:
        assert m["T"][2, 3] == 0.0 and np.isnan(m["T"][4, 5])
    for k in m:
        bad = ~np.isfinite(m[k])
        assert bad.sum() == bad[2, 3] + bad[4, 5]


@pytest.mark.parametrize("thermal", [True, False])
def test_sums_beyond_the_range_of_fp32(T, thermal):
    # populations that FP32 holds but whose sums it does not: moments and global sums are those of
    # FP64 arithmetic, nine and a few thousand terms of 2^-53 each
    nx, ny = 64, 48
    case, _ = W.random_periodic(nx, ny, seed=67, force="none", correction=thermal)
    case = dict(case, thermal=thermal)
    lat = T.Lattice(case)
    f, h = lat.populations()
    rng = np.random.default_rng(68)
    f[:, ::5, ::7] += 3e38 * rng.uniform(0.5, 1.0, f[:, ::5, ::7].shape)
    f[:, 1::5, ::7] *= 1e30 * rng.uniform(0.5, 1.0, f[:, 1::5, ::7].shape)
    if thermal:
        h[:, 2::5, ::7] += 3e38 * rng.uniform(0.5, 1.0, h[:, 2::5, ::7].shape)
    lat.set_populations(f, h)
    f, h = lat.populations()
    m, d = lat.moments(), lat.diagnostics()
    lat.snapshot_velocity()
    again = lat.diagnostics()
    p = lat.params
    lat.close()
    ex, ey = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    rho = f.sum(0)
    jx, jy = sum(e * v for e, v in zip(ex, f)), sum(e * v for e, v in zip(ey, f))
    assert rho.max() > 1e39 and np.isfinite(rho).all()
    scale = np.abs(f).sum(0)
    assert (np.abs(m["rho"] - rho) <= 2.0 ** -49 * scale).all()
    for k, j in (("ux", jx), ("uy", jy)):
        assert (np.abs(m[k] - j / rho) <= 2.0 ** -49 * scale / np.abs(rho)).all()
    tol = 2.0 ** -41
    for got, want, mag in ((d[0], rho.sum(), scale.sum()), (d[1], jx.sum(), scale.sum()), (d[2], jy.sum(), scale.sum())):
        assert abs(got - want) <= tol * mag
    uu = (jx / rho) ** 2 + (jy / rho) ** 2
    assert abs(d[7] - uu.sum()) <= tol * uu.sum()
    if thermal:
        assert abs(d[3] - h.sum()) <= tol * np.abs(h).sum()
        c = 2.0 / (2.0 / (p.gamma - 1.0) * p.R)
        E = h.sum(0) / rho
        assert (np.abs(m["T"] - c * (E - uu / 2)) <= 2.0 ** -47 * c * (np.abs(h).sum(0) / rho + uu)).all()
    assert abs(again[6]) <= 2.0 ** -40 * uu.sum() and again[7] == d[7]  # (the snapshot is FP32)


@pytest.mark.parametrize("what", ["moments", "populations"])
def test_host_outputs_stay_as_they_are_until_the_queued_work_is_done(T, what):
    # work queued earlier may still read an array that a call is about to overwrite in stream
    # order: while a few tenths of a second of steps run, a call waiting behind them on another
    # thread leaves every byte of its pageable outputs alone
    import threading

    import torch

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        lat = T.Lattice(*W.rayleigh_benard(512, 256, seed=69))
        lat.step(100)
        lat.moments(), lat.populations()
        lat.step(60000)
        done = torch.cuda.Event()
        done.record(stream)
    n = 512 * 256
    arrays = [np.full(n, 1.0 / 3.0) for _ in range(4)] if what == "moments" else [np.full(9 * n, 1.0 / 3.0) for _ in range(2)]
    call = (lambda: T.tclbm_moments(lat.handle, *[a.ctypes.data for a in arrays], 0)) if what == "moments" else \
        (lambda: T.tclbm_get_populations(lat.handle, *[a.ctypes.data for a in arrays], 0))
    thread = threading.Thread(target=call)
    thread.start()
    looks = 0
    while True:
        same = all((a == 1.0 / 3.0).all() for a in arrays)
        if done.query():
            break
        assert same
        looks += 1
    thread.join()
    assert looks > 3 and all((a != 1.0 / 3.0).all() for a in arrays)
    assert np.array_equal(arrays[0], (lat.moments()["rho"] if what == "moments" else lat.populations()[0]).ravel())
    lat.close()
