"""GPU parity of the CUDA library against the FP64 oracle (and closed forms).

Tolerances (per target body p, acceleration a_p from Eq. 1):
  FP64  : |a_gpu - a_ref| / |a_ref| <= 1e-13 per evaluation; positions within
          1e-10 AU of the oracle after 3650 steps of the 31-body system.
  mixed : |a_gpu - a_ref| / T_p <= 2e-6, with T_p = sum_j |term_pj| (the
          condition-free form), and |a_gpu - a_ref| / |a_ref| <= 2e-6 for every
          body whose sum is well conditioned (T_p / |a_p| <= 1e3); energy
          drift over 3650 steps within 2x the oracle's.
The FP64 bound comes from the arithmetic: each term is accurate to a few
ulps (binomial-series |d|^-3) and sums of <= 1e6 terms in FP64 keep ~1e-14.
The mixed bound is the FP32 unit roundoff (6e-8) times the few-ulp error of
the MUFU rsqrt seed, cubed, plus FP32 sub-sums of 64 terms.
"""
import numpy as np
import pytest

import oracle
from paper_2112_15079_gb300 import inputs

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-13
MIXED_TOL = 2e-6


@pytest.fixture(scope="module")
def nb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_15079_gb300 import build
    build.build()
    from paper_2112_15079_gb300 import nbody
    return nbody


def _make(nb, s, precision, tiles=None, graphs=True, offsets=None, small=True, pair_once=True):
    b = nb.NBody(s.r, s.v, s.m, offsets, G=s.G, dt=s.dt, precision=precision, graphs=graphs, small=small,
                 pair_once=pair_once)
    if tiles:
        t = b.tiles
        t.update(tiles)
        b.tiles = t
        b.reset()
    return b


def _rel_err(a, ref):
    return np.linalg.norm(a - ref, axis=0) / np.linalg.norm(ref, axis=0)


def _check_accel(precision, a, ref, tnorm):
    """Gate per body (module docstring); returns the figures of the mixed
    gate: bodies left out of the relative form (T_p / |a_p| > 1e3), the
    largest condition number, the worst relative error among the left-out
    bodies and among the rest, and the worst condition-free error."""
    d = np.linalg.norm(a - ref, axis=0)
    n = np.linalg.norm(ref, axis=0)
    cond = tnorm / n
    good = cond <= 1e3
    report = {"bodies": int(d.size), "excluded": int((~good).sum()), "max_cond": float(cond.max()),
              "worst_rel_excluded": float((d / n)[~good].max()) if (~good).any() else None,
              "worst_rel": float((d / n)[good].max()) if good.any() else None,
              "worst_condition_free": float((d / tnorm).max())}
    if precision == "fp64":
        assert np.max(d / n) <= FP64_TOL, np.max(d / n)
    else:
        assert np.max(d / tnorm) <= MIXED_TOL, np.max(d / tnorm)
        assert np.max((d / n)[good]) <= MIXED_TOL, np.max((d / n)[good])
    return report


def _t(threads, ipt, tj, jsplit, cps):
    return {"threads": threads, "ipt": ipt, "tj": tj, "jsplit": jsplit, "ctas_per_sm": cps}


# Work decompositions exercised per precision (None: the library's default).
TILES = {
    "fp64": [None, _t(64, 1, 64, 0, 1), _t(128, 2, 128, 2, 2), _t(256, 1, 192, 8, 3), _t(512, 1, 1024, 1, 1)],
    "mixed": [None, _t(128, 1, 64, 0, 1), _t(256, 2, 128, 2, 2), _t(512, 1, 192, 8, 2), _t(1024, 1, 2048, 1, 1),
              _t(512, 2, 512, 3, 1), _t(384, 2, 256, 0, 2), _t(768, 2, 1024, 0, 1), _t(128, 4, 512, 0, 2),
              _t(256, 4, 64, 2, 1)],
}
CASES = [(p, t) for p in ("fp64", "mixed") for t in TILES[p]]


@pytest.mark.parametrize("precision,tiles", CASES)
@pytest.mark.parametrize("n", [31, 2131, 5003])
def test_initial_accel_vs_oracle(nb, precision, tiles, n):
    s = inputs.solar_system(n, seed=100 + n)
    b = _make(nb, s, precision, tiles)
    a = b.accel().cpu().numpy()
    ref = oracle.accel(s.G, s.r, s.m, openmp=True)
    _check_accel(precision, a, ref, oracle.term_norm(s.G, s.r, s.m, openmp=True))


@pytest.mark.parametrize("precision,pair_once", [("fp64", True), ("fp64", False), ("mixed", False)])
def test_full_size_10425_accel_every_body(nb, precision, pair_once, record_property):
    """The 10,425-body Solar-System-shaped model, all bodies, default tiles
    (FP64: with the pair-once kernel, the default, and with the every-
    ordered-pair kernel; mixed: the every-ordered-pair kernel, its default at
    this size).  The mixed gate's exclusions are reported (no body of this
    model has T_p / |a_p| > 1e3: the Sun's pull dominates every sum)."""
    s = inputs.solar_system(10425)
    b = _make(nb, s, precision, pair_once=pair_once)
    assert b.pair_once == pair_once
    a = b.accel().cpu().numpy()
    ref = oracle.accel(s.G, s.r, s.m, openmp=True)
    rep = _check_accel(precision, a, ref, oracle.term_norm(s.G, s.r, s.m, openmp=True))
    record_property("mixed_gate", rep)
    print(precision, rep)
    assert rep["excluded"] == 0 and rep["max_cond"] < 10.0, rep


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_steps_then_reevaluate(nb, precision):
    """After GPU steps of the 10,425-body model, the GPU acceleration of the
    GPU-produced state equals the oracle's Eq. 1 at that state (the moons make
    long trajectories chaotic, so states are compared through Eq. 1)."""
    s = inputs.solar_system(10425, seed=7)
    b = _make(nb, s, precision)
    b.step(25)
    r = b.r.cpu().numpy()
    a = b.accel().cpu().numpy()
    ref = oracle.accel(s.G, r, s.m, openmp=True)
    _check_accel(precision, a, ref, oracle.term_norm(s.G, r, s.m, openmp=True))


def test_fp64_trajectory_31_bodies_3650_steps(nb):
    s = inputs.solar_system(31)
    b = _make(nb, s, "fp64")
    b.step(3650)
    r_ref, v_ref, _ = oracle.verlet(s.G, s.dt, 3650, s.r, s.v, s.m)
    r = b.r.cpu().numpy()
    assert np.abs(r - r_ref).max() <= 1e-10
    assert np.abs(b.v.cpu().numpy() - v_ref).max() <= 1e-10 * np.abs(v_ref).max()


@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 96])
def test_small_system_kernel_vs_general_and_oracle(nb, n):
    """One FP64 system of <= 96 bodies runs every step in one cluster launch
    (8 CTAs up to 32 bodies, 16 beyond; 4 warps per CTA up to 64 bodies, then
    one per 16 targets); it matches the oracle and the general two-kernel
    path."""
    s = inputs.solar_system(31, seed=70 + n) if n == 31 else None
    if n > 31:
        s = inputs.solar_system(n, seed=71, n_moons=0)
    if n == 2:
        r = np.array([[0.0, 1.0], [0.0, 0.0], [0.0, 0.0]])
        v = np.array([[0.0, 0.0], [0.0, 0.0172], [0.0, 0.0]])
        s = inputs.System(r=r, v=v, m=np.array([1.0, 3e-6]))
    steps = 1000
    small = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    gen = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64", small=False)
    for b in (small, gen):
        b.step(400)
        b.step(steps - 400)
        b.sync()
    r_ref, v_ref, a_ref = oracle.verlet(s.G, s.dt, steps, s.r, s.v, s.m)
    for b in (small, gen):
        assert np.abs(b.r.cpu().numpy() - r_ref).max() <= 1e-11 * max(1.0, np.abs(r_ref).max())
        assert np.abs(b.v.cpu().numpy() - v_ref).max() <= 1e-11 * np.abs(v_ref).max()
        a = b.accel().cpu().numpy()
        assert np.max(np.linalg.norm(a - a_ref, axis=0) / np.linalg.norm(a_ref, axis=0)) <= FP64_TOL
    assert np.abs(small.r.cpu().numpy() - gen.r.cpu().numpy()).max() <= 1e-11 * max(1.0, np.abs(r_ref).max())


@pytest.mark.parametrize("n,steps", [(97, 1000), (257, 1000), (521, 400), (1031, 200), (4096, 10)])
def test_grid_kernel_vs_general_and_oracle(nb, n, steps):
    """One FP64 system of 97 to 4,096 bodies runs every step of a call in one
    cooperative grid launch (one warp per target, positions exchanged through
    L2 behind a grid barrier); it matches the oracle and the general path,
    and a run split into two calls is bitwise the same as one call."""
    s = inputs.solar_system(n, seed=73, n_moons=0)
    grid = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    gen = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64", small=False)
    whole = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    for b in (grid, gen):
        b.step(steps // 3)
        b.step(steps - steps // 3)
        b.sync()
    whole.step(steps)
    whole.sync()
    assert np.array_equal(grid.state.cpu().numpy(), whole.state.cpu().numpy())
    r_ref, v_ref, a_ref = oracle.verlet(s.G, s.dt, steps, s.r, s.v, s.m, openmp=True)
    for b in (grid, gen):
        assert np.abs(b.r.cpu().numpy() - r_ref).max() <= 1e-11 * max(1.0, np.abs(r_ref).max())
        assert np.abs(b.v.cpu().numpy() - v_ref).max() <= 1e-11 * np.abs(v_ref).max()
        a = b.accel().cpu().numpy()
        assert np.max(np.linalg.norm(a - a_ref, axis=0) / np.linalg.norm(a_ref, axis=0)) <= FP64_TOL


@pytest.mark.parametrize("n", [152, 153, 305, 456, 457, 609, 1216, 1217, 1824, 1825])
def test_grid_kernel_shapes(nb, n):
    """The edges of the grid kernel's shapes (1 to 12 targets to a CTA, 4, 2
    or 1 warps to a target, on 152 SMs; 1,825 bodies take the general path)
    against the oracle, in the tolerance of the test above."""
    steps = 5
    s = inputs.solar_system(n, seed=74, n_moons=0)
    b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    b.step(steps)
    b.sync()
    r_ref, v_ref, a_ref = oracle.verlet(s.G, s.dt, steps, s.r, s.v, s.m, openmp=True)
    assert np.abs(b.r.cpu().numpy() - r_ref).max() <= 1e-11 * max(1.0, np.abs(r_ref).max())
    assert np.abs(b.v.cpu().numpy() - v_ref).max() <= 1e-11 * np.abs(v_ref).max()
    a = b.accel().cpu().numpy()
    assert np.max(np.linalg.norm(a - a_ref, axis=0) / np.linalg.norm(a_ref, axis=0)) <= FP64_TOL


@pytest.mark.parametrize("n", [31, 131, 521])
@pytest.mark.parametrize("r_scale, m_scale", [(2.0**230, 1.0), (2.0**-230, 1.0), (1.0, 2.0**-420)])
def test_small_systems_beyond_the_integer_path(nb, n, r_scale, m_scale):
    """Magnitudes whose |d|^-3 the FP64 series takes (the cluster and grid
    kernels, and the general path's first force): a power-of-two scale of a
    model must only scale its accelerations after a step that is too short
    to move it."""
    s = inputs.solar_system(n, n_moons=0)
    m = s.m.copy()
    m[20:] = 0.0
    b = nb.NBody(s.r * r_scale, 0.0 * s.v, m * m_scale, G=1.0, dt=1e-200, precision="fp64")
    ref = oracle.accel(1.0, s.r, m) * (m_scale / (r_scale * r_scale))
    for _ in range(2):
        a = b.accel().cpu().numpy()
        scale = np.abs(ref).max()
        assert np.max(np.linalg.norm((a - ref) / scale, axis=0) / np.linalg.norm(ref / scale, axis=0)) <= FP64_TOL
        b.step(1)
    b.close()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 96, 97, 131, 521, 1824])
def test_a_body_among_massless_ones_feels_nothing(nb, n):
    """Eq. 1 over massless bodies is exactly zero, and so is a single body's
    sum: the star of a system of test particles keeps a = 0 and its position to
    the bit in the single-launch kernels, whose lanes without a source take a
    massless stand-in."""
    s = inputs.solar_system(max(n, 31), seed=75, n_moons=0)
    r, v, m = s.r[:, :n].copy(), s.v[:, :n].copy(), np.zeros(n)
    m[0] = 1.0
    v[:, 0] = 0.0
    b = nb.NBody(r, v, m, G=s.G, dt=s.dt, precision="fp64")
    b.step(3)
    a = b.accel().cpu().numpy()
    assert np.array_equal(a[:, 0], np.zeros(3))
    assert np.array_equal(b.r.cpu().numpy()[:, 0], r[:, 0])
    if n > 1:
        d = b.r.cpu().numpy()[:, :1] - b.r.cpu().numpy()[:, 1:]
        ref = s.G * d / np.linalg.norm(d, axis=0) ** 3
        assert np.max(_rel_err(a[:, 1:], ref)) <= FP64_TOL
    b.close()


@pytest.mark.parametrize("n", [31, 131])
def test_single_launch_kernels_far_from_the_origin(nb, n):
    """Coordinates whose squares overflow (1e160; an ulp is 1e144 there, so every
    |d|^-3 underflows and Eq. 1 gives zeros): the massless stand-ins of the
    single-launch kernels must not turn them into NaN."""
    rng = np.random.default_rng(n)
    r = 1e160 + np.round(rng.uniform(-1.0, 1.0, (3, n)) * 2.0**20) * 2.0**486
    b = nb.NBody(r, 0.0 * r, rng.uniform(0.5, 1.0, n), G=1.0, dt=1e-200, precision="fp64")
    b.step(2)
    b.sync()
    assert np.array_equal(b.accel().cpu().numpy(), np.zeros((3, n)))
    b.close()


@pytest.mark.parametrize("n", [1, 2, 33, 131, 521])
def test_the_targets_own_pair_in_the_ordered_kernel(nb, n):
    """The FP64 ordered-pair kernel takes a target's own entry as a massless
    source a unit away: exactly nothing is added, also where the target is the
    only massive body, and its neighbours' sums keep the FP64 gate."""
    s = inputs.solar_system(max(n, 31), seed=76, n_moons=0)
    r, v = s.r[:, :n].copy(), s.v[:, :n].copy()
    for m in (np.where(np.arange(n) == 0, 1.0, 0.0), s.m[:n].copy()):
        b = nb.NBody(r, v, m, G=s.G, dt=s.dt, precision="fp64", small=False, pair_once=False)
        a = b.accel().cpu().numpy()
        b.close()
        if n == 1 or m[1] == 0.0:
            assert np.array_equal(a[:, 0], np.zeros(3))
        if n > 1:
            ref = oracle.accel(s.G, r, m)
            assert np.max(_rel_err(a[:, 1:], ref[:, 1:])) <= FP64_TOL


def test_grid_kernel_wait_timeout_reports_and_recovers(nb, monkeypatch):
    """NBODY_INJECT_WAIT_STALL=1 makes CTA 0 of the cooperative grid kernel
    (257 bodies) skip its first barrier arrival: every CTA's bounded wait
    runs out (about a second), the kernel winds down, nbody_sync reports
    ETIMEOUT, and after the state is restored and reset the context steps
    bitwise like a fresh one."""
    import time
    s = inputs.solar_system(257, seed=54, n_moons=0)
    fresh = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    fresh.step(50)
    want = fresh.state.cpu().numpy()
    monkeypatch.setenv("NBODY_INJECT_WAIT_STALL", "1")
    b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    monkeypatch.delenv("NBODY_INJECT_WAIT_STALL")
    t0 = time.time()
    b.step(10)
    with pytest.raises(nb.NBodyError) as ei:
        b.sync()
    assert ei.value.status == nb.NBODY_ETIMEOUT
    assert time.time() - t0 < 60
    torch = pytest.importorskip("torch")
    b.state[0:3].copy_(torch.tensor(s.r))
    b.state[3:6].copy_(torch.tensor(s.v))
    b.reset()
    b.step(50)
    assert np.array_equal(b.state.cpu().numpy(), want)


@pytest.mark.parametrize("sizes", [[1], [2], [33], [127], [128], [129], [1283], [40, 1, 300, 129, 7]])
@pytest.mark.parametrize("r_scale", [1.0, 2.0**210, 2.0**-210])
def test_energy_blocks(nb, sizes, r_scale):
    """The energy kernel's tiles and blocks (32 and 128 bodies), several
    systems in one context, massless bodies, and distances that the FP64
    series takes instead of the integer path.  Tolerance as above: a system's
    energy within 1e-13 of the sum of the magnitudes of its two parts."""
    parts = [inputs.solar_system(max(k, 31), seed=90 + i, n_moons=0) for i, k in enumerate(sizes)]
    r = [p.r[:, :k] * r_scale for p, k in zip(parts, sizes)]
    v = [p.v[:, :k] / np.sqrt(r_scale) for p, k in zip(parts, sizes)]
    m = [p.m[:k].copy() for p, k in zip(parts, sizes)]
    for t in m:
        t[3::5] = 0.0
    off = np.concatenate([[0], np.cumsum(sizes)])
    b = nb.NBody(np.concatenate(r, 1), np.concatenate(v, 1), np.concatenate(m), off, G=inputs.G_AU_DAY, dt=0.1,
                 precision="fp64")
    got = b.energy()
    b.close()
    for e, x, u, w in zip(got, r, v, m):
        kin, pot = oracle.energy(inputs.G_AU_DAY, np.ascontiguousarray(x), np.ascontiguousarray(u), w)
        assert abs(e - (kin + pot)) <= 1e-13 * (abs(kin) + abs(pot))


def test_mixed_energy_drift_31_bodies(nb):
    """Energy drift of the mixed path within 2x the oracle's (3650 steps)."""
    s = inputs.solar_system(31)
    E0 = sum(oracle.energy(s.G, s.r, s.v, s.m))
    b = _make(nb, s, "mixed")
    r, v, a = s.r, s.v, None
    drift_ref, drift_gpu = 0.0, 0.0
    for _ in range(73):
        r, v, a = oracle.verlet(s.G, s.dt, 50, r, v, s.m, a)
        drift_ref = max(drift_ref, abs(sum(oracle.energy(s.G, r, v, s.m)) - E0) / abs(E0))
        b.step(50)
        rg, vg = b.r.cpu().numpy(), b.v.cpu().numpy()
        drift_gpu = max(drift_gpu, abs(sum(oracle.energy(s.G, rg, vg, s.m)) - E0) / abs(E0))
    assert drift_gpu <= 2 * drift_ref, (drift_gpu, drift_ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_split_calls_and_graphs_bitwise(nb, precision):
    """On the general path (two launches per step): n steps in one call ==
    the same steps over several calls == without graphs: the kernels are
    deterministic and the drift is the same code."""
    s = inputs.solar_system(2131, seed=3)
    outs = []
    for graphs, chunks in ((True, [130]), (True, [64, 1, 65]), (False, [7, 123])):
        b = _make(nb, s, precision, graphs=graphs, small=False)
        for c in chunks:
            b.step(c)
        outs.append(b.state.cpu().numpy())
        b.close()
    assert np.array_equal(outs[0], outs[1])
    assert np.array_equal(outs[0], outs[2])
    b = _make(nb, s, precision, small=False)
    kt = b.kernel_times(130)  # the timed, unchained launches compute the same steps
    assert np.array_equal(b.state.cpu().numpy(), outs[0])
    assert kt["steps"] == 130 and kt["force_ms"] > 0 and kt["verlet_ms"] > 0
    assert kt["step_ms"] >= kt["force_ms"] + kt["verlet_ms"] - 1e-3
    b.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,seed", [(2131, 9), (10425, inputs.BASE_SEED), (10425, 9)])
def test_energy_vs_oracle(nb, precision, n, seed):
    """Total energy (FP64 in both precisions: the energy kernels take the FP64
    state), including the 10,425-body model, within 1e-13 relative."""
    s = inputs.solar_system(n, seed=seed)
    b = _make(nb, s, precision)
    e = b.energy()[0]
    ref = sum(oracle.energy(s.G, s.r, s.v, s.m))
    assert abs(e - ref) <= 1e-13 * abs(ref), (e, ref)


def test_fp64_two_body_systems_ulp(nb):
    """10^5 independent two-body systems in one FP64 context: body 0 at the
    origin, body 1 at d with |d| log-spaced over 1e-8 .. 1e3 AU in random
    directions, so each a_p is the single term G m_j d / |d|^3 (d exact).
    Against that term evaluated in extended precision, per element:
      GPU within 6 ulp.  The rounding count behind the bound: mu = fl(G m)
      (u), |d|^2 (3u, times 3/2 in |d|^-3), the series refinement of |d|^-3
      (2.5u: the rounding of y0^2 is corrected by the series itself), mu s
      and s d (u each) -- 11.5u = 5.75 ulp;
      the oracle within 6 ulp likewise, and GPU and oracle within 11 ulp of
      each other;
    and no bias: the mean signed error within 0.02 ulp and the mean
    magnitude below 1 ulp.  A refinement whose MUFU seed were worse than the
    2^-19 the series assumes would leave a same-signed error of many ulps."""
    L = np.longdouble
    if np.finfo(L).eps > 1e-18:
        pytest.skip("no extended precision on this host")
    n_sys = 100000
    rng = np.random.default_rng(5)
    mag = np.logspace(-8, 3, n_sys)
    u = rng.normal(size=(3, n_sys))
    u /= np.linalg.norm(u, axis=0)
    d = mag * u
    m0 = np.exp(rng.uniform(np.log(1e-6), np.log(1.0), n_sys))
    m1 = np.exp(rng.uniform(np.log(1e-12), np.log(1e-3), n_sys))
    r = np.zeros((3, 2 * n_sys))
    r[:, 1::2] = d
    m = np.empty(2 * n_sys)
    m[0::2] = m0
    m[1::2] = m1
    off = np.arange(0, 2 * n_sys + 1, 2, dtype=np.int64)
    G = inputs.G_AU_DAY
    b = nb.NBody(r, np.zeros_like(r), m, off, G=G, dt=0.1, precision="fp64")
    a = b.accel().cpu().numpy()
    b.close()
    dl = d.astype(L)
    r2 = (dl * dl).sum(axis=0)
    s3 = 1 / (r2 * np.sqrt(r2))
    exact = np.empty((3, 2 * n_sys), dtype=L)
    exact[:, 0::2] = L(G) * m1.astype(L) * s3 * dl
    exact[:, 1::2] = -(L(G) * m0.astype(L) * s3 * dl)
    ulp = np.spacing(np.abs(exact.astype(np.float64))).astype(L)
    err = ((a.astype(L) - exact) / ulp).astype(np.float64)
    assert np.abs(err).max() <= 6.0, np.abs(err).max()
    assert abs(err.mean()) <= 0.02 and np.abs(err).mean() <= 1.0, (err.mean(), np.abs(err).mean())
    samp = rng.choice(n_sys, 2000, replace=False)
    for k in samp:
        sl = slice(2 * k, 2 * k + 2)
        ora = oracle.accel(G, r[:, sl], m[sl])
        e_o = np.abs(((ora.astype(L) - exact[:, sl]) / ulp[:, sl]).astype(np.float64))
        assert e_o.max() <= 6.0, (k, e_o.max())
        assert np.abs(a[:, sl] - ora).max() <= 11.0 * float(ulp[:, sl].max()), k


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batched_uneven_systems(nb, precision):
    """Independent systems of uneven size (including 1- and 2-body systems)
    in one context: each equals the oracle run on its own.  Systems without
    moons are compared along the trajectory; systems with moons (whose
    shortest orbits are unresolved at dt = 0.1 day, so trajectories diverge
    chaotically) through Eq. 1 re-evaluated at the GPU state."""
    spec = [(31, 100), (1, 0), (700, 100), (2, 0), (1531, 0), (257, 0)]
    systems = []
    for k, (n, moons) in enumerate(spec):
        if n >= 31:
            systems.append(inputs.solar_system(n, seed=40 + k, n_moons=moons))
        else:
            r = np.array([[1.0, 2.5][:n], [0.0, 0.1][:n], [0.0, 0.0][:n]])
            v = np.array([[0.0, 0.0][:n], [0.01, -0.01][:n], [0.0, 0.001][:n]])
            systems.append(inputs.System(r=r, v=v, m=np.array([1e-3, 2e-3][:n])))
    off, r, v, m = inputs.concat(systems)
    G, dt = inputs.G_AU_DAY, inputs.DT_DAY
    b = nb.NBody(r, v, m, off, G=G, dt=dt, precision=precision)
    a = b.accel().cpu().numpy()
    b.step(20)
    rg, vg = b.r.cpu().numpy(), b.v.cpu().numpy()
    ag = b.accel().cpu().numpy()
    eg = b.energy()
    for k, sysk in enumerate(systems):
        sl = slice(off[k], off[k + 1])
        if sysk.n == 1:
            assert np.all(a[:, sl] == 0.0)
            np.testing.assert_allclose(rg[:, sl], sysk.r + 20 * dt * sysk.v, rtol=1e-14)
            continue
        _check_accel(precision, a[:, sl], oracle.accel(G, sysk.r, sysk.m), oracle.term_norm(G, sysk.r, sysk.m))
        _check_accel(precision, ag[:, sl], oracle.accel(G, rg[:, sl], sysk.m), oracle.term_norm(G, rg[:, sl], sysk.m))
        if sysk.info.get("n_moons", 0) == 0:
            r_ref, v_ref, _ = oracle.verlet(G, dt, 20, sysk.r, sysk.v, sysk.m)
            tol = 1e-12 if precision == "fp64" else 1e-7
            assert np.abs(rg[:, sl] - r_ref).max() <= tol * max(1.0, np.abs(r_ref).max())
        e_ref = sum(oracle.energy(G, rg[:, sl], vg[:, sl], sysk.m))
        assert abs(eg[k] - e_ref) <= 1e-12 * abs(e_ref) + 1e-300


@pytest.mark.parametrize("precision,n_ring", [("fp64", 4095), ("mixed", 262143), ("mixed", 1048575)])
def test_ring_closed_form_large_n(nb, precision, n_ring):
    """n-gon ring of equal masses m around a central mass Mc: every ring body
    is pulled inward with G Mc/R^2 + (G m/R^2) sum_k 1/(4 sin(pi k/n)) and
    feels no tangential force.  The error scale is the closed-form term norm
    T = G Mc/R^2 + (G m/(4R^2)) sum_k csc^2(pi k/n) = G Mc/R^2 + G m (n^2-1)/(12 R^2).
    The closed form holds for the exact polygon; rounding R cos, R sin to
    FP64 moves neighbours (2 pi R/n apart) by ~eps R, which shifts a_p by
    ~4 G m eps R (n / 2 pi R)^3 -- below 1e-13 T only for n of a few
    thousand, so the FP64 case uses n = 4095 (FP64 at large n is pinned by the
    integer-position chain below)."""
    G, R, m, Mc = 2.9591220828e-4, 2.0, 1e-8, 1.0
    th = 2 * np.pi * np.arange(n_ring) / n_ring
    r = np.concatenate([np.zeros((3, 1)), np.stack([R * np.cos(th), R * np.sin(th), 0 * th])], axis=1)
    mass = np.concatenate([[Mc], np.full(n_ring, m)])
    k = np.arange(1, n_ring)
    radial = G * Mc / R**2 + G * m / R**2 * np.sum(1.0 / (4.0 * np.sin(np.pi * k / n_ring)))
    T = G * Mc / R**2 + G * m * (n_ring**2 - 1) / (12 * R**2)
    b = nb.NBody(r, np.zeros_like(r), mass, G=G, dt=0.1, precision=precision)
    a = b.accel().cpu().numpy()
    ring = a[:, 1:]
    inward = -(ring[0] * np.cos(th) + ring[1] * np.sin(th))
    tangential = -ring[0] * np.sin(th) + ring[1] * np.cos(th)
    tol = FP64_TOL if precision == "fp64" else MIXED_TOL
    assert np.max(np.abs(inward - radial)) <= tol * T
    assert np.max(np.abs(tangential)) <= tol * T
    assert np.max(np.abs(a[:, 0])) <= tol * G * m * n_ring / R**2


@pytest.mark.parametrize("precision,n", [("fp64", 100003), ("mixed", 1048577)])
def test_collinear_chain_closed_form(nb, precision, n):
    """Unit masses at x = 0, 1, ..., n-1 (G = 1): body p feels
      a_p = H2(n-1-p) - H2(p),   with T_p = H2(n-1-p) + H2(p),
    H2(k) = sum_{i=1}^k 1/i^2 = pi^2/6 - psi_1(k+1) (trigamma).  The end
    bodies are perfectly conditioned, and a missing or doubled source tile
    anywhere shifts many a_p by far more than the tolerance."""
    special = pytest.importorskip("scipy.special")
    x = np.arange(n, dtype=np.float64)
    r = np.stack([x, 0 * x, 0 * x])
    b = nb.NBody(r, np.zeros_like(r), np.ones(n), G=1.0, dt=0.1, precision=precision)
    a = b.accel().cpu().numpy()
    p = np.arange(n)
    H2 = lambda k: np.pi**2 / 6 - special.polygamma(1, k + 1.0)
    want = H2(n - 1 - p) - H2(p)
    T = H2(n - 1 - p) + H2(p)
    tol = FP64_TOL if precision == "fp64" else MIXED_TOL
    # trigamma itself carries ~1e-15 relative error, well inside both bounds
    assert np.max(np.abs(a[0] - want) / T) <= tol
    assert np.all(a[1:] == 0.0)


def test_fp64_many_subulp_terms(nb):
    """A unit mass at distance 1 listed first, then n tiny masses on a
    half-circle of radius R: a_x = 1 + (m/R^2)/sin(pi/(2n)) exactly.  Each
    tiny term is below half an ulp of the running sum; a plain FP64 running
    sum over one chunk would miss them all (~3e-12 relative at n = 1e5)."""
    n, R = 100000, 2.0
    m = 5e-17 * R * R
    th = -np.pi / 2 + (np.arange(n) + 0.5) * np.pi / n
    x = np.concatenate([[0.0, 1.0], R * np.cos(th)])
    y = np.concatenate([[0.0, 0.0], R * np.sin(th)])
    mass = np.concatenate([[1.0, 1.0], np.full(n, m)])
    b = nb.NBody(np.stack([x, y, 0 * x]), np.zeros((3, n + 2)), mass, G=1.0, dt=0.1, precision="fp64")
    for tiles in (None, {"threads": 128, "ipt": 1, "tj": 256, "jsplit": 1, "ctas_per_sm": 2}):
        if tiles:
            b.tiles = tiles
            b.reset()
        a = b.accel()[:, 0].cpu().numpy()
        want = 1.0 + (m / R**2) / np.sin(np.pi / (2 * n))
        assert abs(a[0] - want) <= 1e-15 * want, (tiles, a[0] - want)
        assert abs(a[1]) <= 1e-20


def test_mixed_1m_sampled_rows(nb, record_property):
    """The N = 1,048,576 Solar-System-shaped model in the mixed path: sampled
    target rows against the oracle's Eq. 1 for those rows (the mixed gate's
    exclusions reported: none of these rows has T_p / |a_p| > 1e3)."""
    s = inputs.solar_system(1 << 20, seed=31)
    b = _make(nb, s, "mixed")
    a = b.accel().cpu().numpy()
    rng = np.random.default_rng(0)
    rows = np.concatenate([np.arange(0, 200), rng.choice(s.n, 56, replace=False), [s.n - 1]])
    ref = oracle.accel_rows(s.G, s.r, s.m, rows, openmp=True)
    tn = oracle.term_norm(s.G, s.r, s.m, rows, openmp=True)
    rep = _check_accel("mixed", a[:, rows], ref, tn)
    record_property("mixed_gate", rep)
    print(rep)
    assert rep["excluded"] == 0 and rep["max_cond"] < 10.0, rep


def test_fp64_1m_sampled_rows(nb):
    """The N = 1,048,576 model in the FP64 path (one ~31 s force evaluation at
    init, the bench's FP64 launch configuration): sampled rows against the
    oracle's Eq. 1 for those rows, to the FP64 tolerance."""
    s = inputs.solar_system(1 << 20, seed=32)
    b = _make(nb, s, "fp64")
    a = b.accel().cpu().numpy()
    rng = np.random.default_rng(1)
    rows = np.concatenate([np.arange(0, 131), rng.choice(s.n, 61, replace=False), [s.n - 1]])
    ref = oracle.accel_rows(s.G, s.r, s.m, rows, openmp=True)
    tn = oracle.term_norm(s.G, s.r, s.m, rows, openmp=True)
    _check_accel("fp64", a[:, rows], ref, tn)


def test_ensemble_full_size_sampled_rows(nb):
    """The 256-system uneven ensemble at full size (2.8M bodies, one context,
    mixed, the bench's configuration): Eq. 1 at init for sampled bodies of 16
    systems against the oracle run on each system alone."""
    ens = inputs.ensemble(256)
    off, r, v, m = inputs.concat(ens)
    b = nb.NBody(r, v, m, off, G=inputs.G_AU_DAY, dt=inputs.DT_DAY, precision="mixed")
    a = b.accel().cpu().numpy()
    rng = np.random.default_rng(2)
    for k in rng.choice(256, 16, replace=False):
        e = ens[k]
        rows = np.concatenate([np.arange(0, 131, 13), rng.choice(e.n, 20, replace=False), [e.n - 1]])
        ref = oracle.accel_rows(e.G, e.r, e.m, rows, openmp=True)
        tn = oracle.term_norm(e.G, e.r, e.m, rows, openmp=True)
        _check_accel("mixed", a[:, off[k] + rows], ref, tn)


def test_fp64_time_reversibility(nb):
    s = inputs.solar_system(131, seed=12, n_moons=0)  # resolved orbits only
    b = _make(nb, s, "fp64")
    b.step(300)
    back = nb.NBody(b.r, b.v, s.m, G=s.G, dt=-s.dt, precision="fp64")
    back.step(300)
    assert np.abs(back.r.cpu().numpy() - s.r).max() <= 1e-11 * np.abs(s.r).max()


def test_small_system_time_reversibility(nb):
    """The single-launch kernel (31 bodies, FP64): 3650 steps forward, then
    3650 with -dt from the end state, return to the start."""
    s = inputs.solar_system(31, seed=13)
    b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    b.step(3650)
    back = nb.NBody(b.r, b.v, s.m, G=s.G, dt=-s.dt, precision="fp64")
    back.step(3650)
    assert np.abs(back.r.cpu().numpy() - s.r).max() <= 1e-11 * np.abs(s.r).max()
    assert np.abs(back.v.cpu().numpy() - s.v).max() <= 1e-11 * np.abs(s.v).max()


@pytest.mark.parametrize("n,precision,integrator", [(31, "fp64", "verlet"), (2131, "mixed", "verlet"),
                                                    (2131, "fp64", "verlet"), (2131, "mixed", "rk4")])
def test_steps_captured_in_a_caller_graph(nb, n, precision, integrator):
    """A caller may capture nbody_step into its own CUDA graph (the call is
    asynchronous and allocates nothing): during capture the library launches
    its kernels directly (the single-launch cluster kernel for 31 bodies),
    and each replay advances the state exactly like a direct call."""
    torch = pytest.importorskip("torch")
    s = inputs.solar_system(n, seed=90 + n)
    k = 7
    ref = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision=precision, integrator=integrator)
    for _ in range(3):
        ref.step(k)
    ref.sync()
    side = torch.cuda.Stream()
    b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision=precision, integrator=integrator, stream=side)
    b.step(k)  # one direct call first, so the capture is not the first use of the context
    b.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        b.step(k)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    b.sync()
    assert np.array_equal(b.state.cpu().numpy(), ref.state.cpu().numpy())


def test_contexts_with_different_tiles_share_the_kernels(nb):
    """The force kernel's shared-memory limit belongs to the kernel instance,
    which every context of the process shares.  A context built later with
    smaller source tiles must not take away what an earlier one launches with
    (mixed: 1024 then 64 sources per stage), nor may a context take it from
    the allocation-free entry point (FP64, 256 sources per stage)."""
    torch = pytest.importorskip("torch")
    s = inputs.solar_system(2131, seed=95)
    big = {"threads": 512, "ipt": 1, "tj": 1024, "jsplit": 0, "ctas_per_sm": 2}
    small = dict(big, tj=64)
    want = {}
    for name, t in (("big", big), ("small", small)):
        r = _make(nb, s, "mixed", t)
        r.step(5)
        want[name] = r.state.cpu().numpy()
        r.close()
    a = _make(nb, s, "mixed", big)
    b = _make(nb, s, "mixed", small)  # built after a, needing less shared memory
    a.step(5)
    b.step(5)
    assert np.array_equal(a.state.cpu().numpy(), want["big"])
    assert np.array_equal(b.state.cpu().numpy(), want["small"])
    f = _make(nb, s, "fp64", {"threads": 128, "ipt": 1, "tj": 64, "jsplit": 0, "ctas_per_sm": 3})
    rt = torch.tensor(s.r, dtype=torch.float64, device="cuda")
    mt = torch.tensor(s.m, dtype=torch.float64, device="cuda")
    got = nb.accel_static(rt, mt, s.G).cpu().numpy()
    ref = f.accel().cpu().numpy()
    assert np.max(_rel_err(got, ref)) <= FP64_TOL


def test_edge_cases_and_errors(nb):
    torch = pytest.importorskip("torch")
    # single body: no force, straight-line motion
    one = nb.NBody(np.array([[1.0], [2.0], [3.0]]), np.array([[0.1], [0.0], [-0.2]]), np.array([1.0]),
                   G=1.0, dt=0.5, precision="fp64")
    assert np.all(one.accel().cpu().numpy() == 0.0)
    one.step(4)
    np.testing.assert_allclose(one.r.cpu().numpy()[:, 0], [1.2, 2.0, 2.6], rtol=1e-15)
    one.step(0)  # no-op
    with pytest.raises(nb.NBodyError) as ei:
        one.step(-1)
    assert ei.value.status == nb.NBODY_EINVAL
    # coincident bodies are rejected at init
    r = np.array([[0.0, 1.0, 1.0], [0.0, 0.0, 0.0], [0.0, 0.0, 0.0]])
    for prec in ("fp64", "mixed"):
        with pytest.raises(nb.NBodyError) as ei:
            nb.NBody(r, np.zeros((3, 3)), np.ones(3), G=1.0, dt=0.1, precision=prec)
        assert ei.value.status == nb.NBODY_EINVAL
    # non-finite state and negative mass
    r = np.array([[0.0, 1.0], [0.0, 0.0], [0.0, np.nan]])
    with pytest.raises(nb.NBodyError):
        nb.NBody(r, np.zeros((3, 2)), np.ones(2), G=1.0, dt=0.1)
    with pytest.raises(nb.NBodyError):
        nb.NBody(np.eye(3)[:, :2], np.zeros((3, 2)), np.array([1.0, -1.0]), G=1.0, dt=0.1)
    # bad options
    for kw in ({"G": 0.0, "dt": 0.1}, {"G": 1.0, "dt": 0.0}, {"G": float("inf"), "dt": 0.1}):
        with pytest.raises(nb.NBodyError):
            nb.NBody(np.eye(3)[:, :2], np.zeros((3, 2)), np.ones(2), **kw)
    # bad tiles
    b = nb.NBody(np.eye(3)[:, :2], np.zeros((3, 2)), np.ones(2), G=1.0, dt=0.1)
    with pytest.raises(nb.NBodyError):
        b.tiles = {"threads": 96, "ipt": 1, "tj": 64, "jsplit": 1, "ctas_per_sm": 1}
    with pytest.raises(nb.NBodyError):
        b.tiles = {"threads": 128, "ipt": 1, "tj": 100, "jsplit": 1, "ctas_per_sm": 1}
    # host pointers are rejected
    import ctypes
    h = np.zeros(2)
    ctx = ctypes.c_void_p()
    off = (ctypes.c_int64 * 2)(0, 2)
    opts = nb.nbody_opts(G=1.0, dt=0.1, precision=0, ckpt_every=0, flags=0, integrator=0)
    st = nb.nbody_init(ctypes.byref(ctx), 1, off, *([h.ctypes.data] * 7), ctypes.byref(opts), None)
    assert st == nb.NBODY_EINVAL and not ctx.value
    # a collision during the run surfaces as ENONFINITE on the next sync
    r = np.array([[0.0, 1.0], [0.0, 0.0], [0.0, 0.0]])
    v = np.array([[0.5, -0.5], [0.0, 0.0], [0.0, 0.0]])
    b = nb.NBody(r, v, np.zeros(2), G=1.0, dt=1.0, precision="fp64")  # massless: exact meeting
    b.step(1)
    with pytest.raises(nb.NBodyError) as ei:
        b.sync()
    assert ei.value.status == nb.NBODY_ENONFINITE
    del torch


def test_injected_allocation_failures(nb, monkeypatch):
    """NBODY_INJECT_ALLOC_FAIL=k fails a context's k-th device allocation with
    ENOMEM.  A failed init releases what it allocated; a failed set_tiles
    keeps the previous tiles and tables (still a matching pair, results
    unchanged); a failed first nbody_grad leaves the context able to run the
    next one, with the gradient of an undisturbed context."""
    torch = pytest.importorskip("torch")
    s = inputs.solar_system(1500, seed=9)
    ref = _make(nb, s, "mixed")
    ref.step(5)
    want = ref.state.cpu().numpy()
    gr = np.zeros((3, s.n))
    gr[:, :40] = 1.0
    want_g = [g.cpu().numpy() for g in ref.grad(3, gr)]
    ref.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]

    k = 1
    while True:  # every allocation of init in turn
        monkeypatch.setenv("NBODY_INJECT_ALLOC_FAIL", str(k))
        try:
            b = _make(nb, s, "mixed")
        except nb.NBodyError as e:
            assert e.status == nb.NBODY_ENOMEM and "injected" in str(e)
            k += 1
            assert k < 64
            continue
        break
    b.close()
    n_init = k - 1  # allocations init makes
    assert n_init >= 5

    new_tiles = {"threads": 512, "ipt": 2, "tj": 512, "jsplit": 0, "ctas_per_sm": 2}
    for j in range(1, 7):  # each allocation of a table rebuild
        monkeypatch.delenv("NBODY_INJECT_ALLOC_FAIL")
        b = _make(nb, s, "mixed")
        old = b.tiles
        monkeypatch.setenv("NBODY_INJECT_ALLOC_FAIL", str(n_init + j))
        with pytest.raises(nb.NBodyError) as ei:
            b.tiles = new_tiles
        assert ei.value.status == nb.NBODY_ENOMEM
        assert b.tiles == old
        b.step(5)
        assert np.array_equal(b.state.cpu().numpy(), want)
        b.close()

    j, failed = 1, 0
    while True:  # each allocation of the first nbody_grad
        monkeypatch.delenv("NBODY_INJECT_ALLOC_FAIL", raising=False)
        b = _make(nb, s, "mixed")
        monkeypatch.setenv("NBODY_INJECT_ALLOC_FAIL", str(n_init + j))
        try:
            got = b.grad(3, gr)
        except nb.NBodyError as e:
            assert e.status == nb.NBODY_ENOMEM
            failed += 1
            monkeypatch.delenv("NBODY_INJECT_ALLOC_FAIL")
            got = b.grad(3, gr)
            for x, y in zip(got, want_g):
                assert np.array_equal(x.cpu().numpy(), y)
            b.close()
            j += 1
            assert j < 64
            continue
        for x, y in zip(got, want_g):
            assert np.array_equal(x.cpu().numpy(), y)
        b.close()
        break
    assert failed >= 8
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert abs(torch.cuda.mem_get_info()[0] - free0) <= 16 << 20  # nothing leaked


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_autotune_restores_state_and_keeps_parity(nb, precision):
    """The autotuner times candidates on the bound state, puts the state back
    bitwise, and its winner is a valid decomposition: parity with the oracle
    and bitwise equal steps to a context given the same tiles."""
    s = inputs.solar_system(2131, seed=17)
    b = _make(nb, s, precision)
    b.step(3)
    before = b.state.cpu().numpy()
    tiles, ms = b.autotune(probe_steps=2)
    assert ms > 0 and b.tiles == tiles
    assert np.array_equal(b.state.cpu().numpy(), before)
    b.step(20)
    c = _make(nb, s, precision)
    c.step(3)
    c.tiles = tiles  # same history: default tiles for 3 steps, then the winner's
    c.step(20)
    assert np.array_equal(c.state.cpu().numpy(), b.state.cpu().numpy())
    d = _make(nb, s, precision, tiles)  # the winner's Eq. 1 against the oracle
    _check_accel(precision, d.accel().cpu().numpy(), oracle.accel(s.G, s.r, s.m, openmp=True),
                 oracle.term_norm(s.G, s.r, s.m, openmp=True))


def test_bounded_wait_timeout_reports_and_recovers(nb, monkeypatch):
    """A device wait that nothing completes: NBODY_INJECT_WAIT_STALL=k leaves
    the first source tile of CTA 0 unissued in the context's k-th adjoint
    product.  That CTA's bounded mbarrier wait runs out (~2 s), it drains and
    leaves, nbody_grad reports ETIMEOUT, and the context stays usable: the
    next gradient and the next steps equal a fresh context's bitwise."""
    import time
    torch = pytest.importorskip("torch")
    s = inputs.solar_system(2131, seed=51)
    gr = torch.ones((3, s.n), dtype=torch.float64)
    fresh = _make(nb, s, "mixed")
    want_g = [t.cpu().numpy() for t in fresh.grad(3, gr)]
    fresh.step(5)
    want_s = fresh.state.cpu().numpy()
    monkeypatch.setenv("NBODY_INJECT_WAIT_STALL", "2")  # the second product of the first gradient
    b = _make(nb, s, "mixed")
    monkeypatch.delenv("NBODY_INJECT_WAIT_STALL")
    t0 = time.time()
    with pytest.raises(nb.NBodyError) as ei:
        b.grad(3, gr)
    assert ei.value.status == nb.NBODY_ETIMEOUT
    assert time.time() - t0 < 60
    got = [t.cpu().numpy() for t in b.grad(3, gr)]
    for x, y in zip(got, want_g):
        assert np.array_equal(x, y)
    b.step(5)
    assert np.array_equal(b.state.cpu().numpy(), want_s)


def test_small_system_wait_timeout_reports_and_recovers(nb, monkeypatch):
    """The single-launch 31-body kernel exchanges positions through mbarrier
    waits.  NBODY_INJECT_WAIT_STALL=1 makes CTA 0 leave out one arrival in
    the first nbody_step call: its bounded wait runs out (~2 s), the other
    CTAs' next wait too, the kernel winds down, and nbody_sync reports
    ETIMEOUT.  After the state is restored and reset, the context steps
    bitwise like a fresh one."""
    import time
    s = inputs.solar_system(31, seed=52)
    fresh = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    fresh.step(100)
    want = fresh.state.cpu().numpy()
    monkeypatch.setenv("NBODY_INJECT_WAIT_STALL", "1")
    b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="fp64")
    monkeypatch.delenv("NBODY_INJECT_WAIT_STALL")
    t0 = time.time()
    b.step(10)
    with pytest.raises(nb.NBodyError) as ei:
        b.sync()
    assert ei.value.status == nb.NBODY_ETIMEOUT
    assert time.time() - t0 < 60
    torch = pytest.importorskip("torch")
    b.state[0:3].copy_(torch.tensor(s.r))
    b.state[3:6].copy_(torch.tensor(s.v))
    b.reset()
    b.step(100)
    assert np.array_equal(b.state.cpu().numpy(), want)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_reset_after_the_caller_changes_state_and_masses(nb, precision):
    """nbody_reset re-reads the bound state: new positions and masses (a third
    of them zero: test particles) give Eq. 1 at the new state, and the snapshot
    for nbody_grad is the new state."""
    torch = pytest.importorskip("torch")
    s = inputs.solar_system(2131, seed=61)
    b = _make(nb, s, precision)
    b.step(3)
    rng = np.random.default_rng(8)
    r2 = s.r * (1 + 1e-3 * rng.normal(size=s.r.shape))
    m2 = s.m.copy()
    m2[rng.choice(s.n, s.n // 3, replace=False)] = 0.0
    b.state[0:3].copy_(torch.tensor(r2))
    b.m.copy_(torch.tensor(m2))
    b.reset()
    ref = oracle.accel(s.G, r2, m2, openmp=True)
    _check_accel(precision, b.accel().cpu().numpy(), ref, oracle.term_norm(s.G, r2, m2, openmp=True))
    c = nb.NBody(b.r.cpu().numpy(), b.v.cpu().numpy(), m2, G=s.G, dt=s.dt, precision=precision)
    gr = torch.ones((3, s.n), dtype=torch.float64)
    for x, y in zip(b.grad(2, gr), c.grad(2, gr)):
        assert torch.equal(x, y)


def test_nondefault_stream(nb):
    torch = pytest.importorskip("torch")
    s = inputs.solar_system(700, seed=5)
    ref = _make(nb, s, "mixed")
    ref.step(10)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        b = _make(nb, s, "mixed")
        b.step(10)
        out = b.state.clone()
    st.synchronize()
    assert torch.equal(out, ref.state)


def _threshold_system(gap_over_threshold):
    """Two clusters on the x axis near x = 3 AU (one binade, ulp 2^-22):
    64 massless targets whose x = hi + 0.45 ulp, and 256 sources of mass
    1e-3 whose x = hi - 0.45 ulp, at a gap (between the clusters' hi boxes)
    of `gap_over_threshold` times the far threshold kappa (lo_w + lo_s),
    kappa = 2 / 1e-6 + 1.  y, z are multiples of 2^-14 (no lo part), so the
    lo parts the hi-only path drops are aligned with d: the worst case of
    its bound, an error of about 2 |lo_j - lo_p| / |d| = 1e-6 at the
    threshold.  Returns (system, indices of the targets, threshold)."""
    ulp = 2.0 ** -22
    lo = 0.45 * ulp
    kappa = 2.0 / 1e-6 + 1.0
    thr = kappa * (2 * lo)
    grid = 2.0 ** -14 * np.arange(16)
    yz = np.array([(a, b) for a in grid for b in grid])
    x0 = np.float32(3.0)
    xw = np.full(64, np.float64(x0)) + lo
    gap = gap_over_threshold * thr
    xs_hi = np.float64(np.float32(x0 + gap))
    xs = np.full(256, xs_hi) - lo
    r = np.zeros((3, 320))
    r[0, :64], r[1, :64], r[2, :64] = xw, yz[:64, 0], yz[:64, 1]
    r[0, 64:], r[1, 64:], r[2, 64:] = xs, yz[:256, 0], yz[:256, 1] + 2.0 ** -6
    m = np.concatenate([np.zeros(64), np.full(256, 1e-3)])
    return inputs.System(r=r, v=np.zeros_like(r), m=m), np.arange(64), thr


@pytest.mark.parametrize("ratio", [0.8, 1.25, 3.0])
def test_mixed_far_threshold_adversarial(nb, ratio):
    """Targets and sources placed just inside (0.8) and just outside (1.25,
    3) the distance beyond which the mixed kernel drops the lo parts, with
    the dropped parts aligned with d (worst case).  Inside: the hi/lo path,
    FP32-level error (<= 3e-7).  Outside: the hi-only path, whose error
    bound is 1e-6 at the threshold and falls as 1 / distance; the measured
    error must stay within that bound plus the FP32-level error, and (so the
    case really exercises the far path) exceed the FP32 level just outside.
    A threshold set too small would put pairs closer than it on the hi-only
    path with errors above the bound."""
    s, idx, thr = _threshold_system(ratio)
    b = nb.NBody(s.r, s.v, s.m, G=1.0, dt=0.1, precision="mixed")
    a = b.accel().cpu().numpy()[:, idx]
    ref = oracle.accel(1.0, s.r, s.m)[:, idx]
    err = np.linalg.norm(a - ref, axis=0) / np.linalg.norm(ref, axis=0)
    if ratio < 1.0:
        assert err.max() <= 3e-7, err.max()
    else:
        assert err.max() <= 1e-6 / ratio + 3e-7, (ratio, err.max())
        if ratio < 2.0:
            assert err.max() > 4e-7, (ratio, err.max())


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_reorder_keeps_parity(nb, precision):
    """nbody_reorder between steps (a new spatial order of the sources in
    the mixed path, a no-op in FP64) leaves the trajectory on the oracle's."""
    s = inputs.solar_system(2131, seed=81, n_moons=0)
    b = _make(nb, s, precision)
    b.step(30)
    b.reorder()
    b.step(30)
    r_ref, v_ref, _ = oracle.verlet(s.G, s.dt, 60, s.r, s.v, s.m, openmp=True)
    tol = 1e-12 if precision == "fp64" else 1e-7
    assert np.abs(b.r.cpu().numpy() - r_ref).max() <= tol * np.abs(r_ref).max()
    a = b.accel().cpu().numpy()
    r = b.r.cpu().numpy()
    _check_accel(precision, a, oracle.accel(s.G, r, s.m, openmp=True), oracle.term_norm(s.G, r, s.m, openmp=True))
    if precision == "fp64":  # no-op: bitwise the same as without
        c = _make(nb, s, precision)
        c.step(60)
        assert np.array_equal(c.state.cpu().numpy(), b.state.cpu().numpy())
