"""The mixed every-ordered-pair kernels at 2,131 bodies, where contexts run
pair-once blocks by default: pair_once=False, each test asserting that it has
reached them.  Tile decompositions (the mixed gate of the parity tests, every
body), the shared-memory limit that contexts of unlike tiles share, the
autotuner, the bounded waits of both kernels of the adjoint product, and the
two forms of its term."""
import time

import numpy as np
import pytest

import oracle
from paper_2112_15079_gb300 import inputs

pytestmark = pytest.mark.gpu

MIXED_TOL = 2e-6
N = 2131


@pytest.fixture(scope="module")
def nb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_15079_gb300 import build
    build.build()
    from paper_2112_15079_gb300 import nbody
    return nbody


def _t(threads, ipt, tj, jsplit, cps):
    return {"threads": threads, "ipt": ipt, "tj": tj, "jsplit": jsplit, "ctas_per_sm": cps}


def _ordered(nb, s, tiles=None):
    b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="mixed", pair_once=False)
    assert b.pair_once_block == 0
    if tiles:
        b.tiles = dict(b.tiles, **tiles)
        b.reset()
        assert b.pair_once_block == 0
    return b


def _gate(a, s):
    ref, t = oracle.accel(s.G, s.r, s.m, openmp=True), oracle.term_norm(s.G, s.r, s.m, openmp=True)
    d, n = np.linalg.norm(a - ref, axis=0), np.linalg.norm(ref, axis=0)
    good = t / n <= 1e3
    assert np.max(d / t) <= MIXED_TOL and np.max((d / n)[good]) <= MIXED_TOL


@pytest.mark.parametrize("tiles", [None, _t(128, 1, 64, 0, 1), _t(256, 2, 128, 2, 2), _t(512, 1, 192, 8, 2),
                                   _t(1024, 1, 2048, 1, 1), _t(512, 2, 512, 3, 1), _t(384, 2, 256, 0, 2),
                                   _t(768, 2, 1024, 0, 1), _t(128, 4, 512, 0, 2), _t(256, 4, 64, 2, 1)])
def test_tiles(nb, tiles):
    s = inputs.solar_system(N, seed=N)
    b = _ordered(nb, s, tiles)
    _gate(b.accel().cpu().numpy(), s)
    b.close()


def test_contexts_of_unlike_tiles_share_the_kernel(nb):
    """A context built later with smaller source tiles must not take away the
    shared memory that an earlier one launches with."""
    s = inputs.solar_system(N, seed=95)
    big, small = _t(512, 1, 1024, 0, 2), _t(512, 1, 64, 0, 2)
    want = {}
    for name, t in (("big", big), ("small", small)):
        r = _ordered(nb, s, t)
        r.step(5)
        want[name] = r.state.cpu().numpy()
        r.close()
    a, b = _ordered(nb, s, big), _ordered(nb, s, small)
    a.step(5)
    b.step(5)
    assert np.array_equal(a.state.cpu().numpy(), want["big"])
    assert np.array_equal(b.state.cpu().numpy(), want["small"])


def test_autotune(nb):
    """State restored, the winner current, steps bitwise a context's that was
    given the winner's tiles."""
    s = inputs.solar_system(N, seed=17)
    b = _ordered(nb, s)
    b.step(3)
    before = b.state.cpu().numpy()
    tiles, ms = b.autotune(probe_steps=2)
    assert ms > 0 and b.tiles == tiles and b.pair_once_block == 0
    assert np.array_equal(b.state.cpu().numpy(), before)
    b.step(20)
    c = _ordered(nb, s)
    c.step(3)
    c.tiles = tiles
    c.step(20)
    assert np.array_equal(c.state.cpu().numpy(), b.state.cpu().numpy())
    d = _ordered(nb, s, tiles)
    _gate(d.accel().cpu().numpy(), s)


def test_pair_once_context_leaves_tuned_tiles_in_the_cache(nb, tmp_path):
    """One cache key covers 4,200 bodies (pair-once blocks: no tiles to choose)
    and 5,003 (ordered pairs): autotuning the first must not replace what the
    second found; without an entry it writes its own."""
    path = tmp_path / "tune.json"
    mk = lambda n: nb.NBody(*(lambda s: (s.r, s.v, s.m))(inputs.solar_system(n, seed=5)), G=inputs.G_AU_DAY,  # noqa: E731
                            dt=inputs.DT_DAY, precision="mixed", tune_cache=str(path))
    once = mk(4200)
    assert once.pair_once_block == 128
    once.autotune(probe_steps=1)
    assert path.exists()
    path.unlink()
    a = mk(5003)
    assert a.pair_once_block == 0
    best, _ = a.autotune(probe_steps=1)
    doc = path.read_text()
    once.autotune(probe_steps=1)
    assert path.read_text() == doc
    assert mk(5003).tiles == best


@pytest.mark.parametrize("precision,pair_once,block", [("mixed", False, 0), ("mixed", True, 128), ("fp64", False, 0)])
def test_product_wait_timeout_reports_and_recovers(nb, precision, pair_once, block, monkeypatch):
    """NBODY_INJECT_WAIT_STALL=2 makes the second adjoint product's bounded wait
    run out: the ordered kernel's first source tile of CTA 0 stays unissued (the
    CTA drains its other copies and leaves), the pair-once kernel's CTA 0 leaves
    out an arrival.  nbody_grad reports ETIMEOUT, and the next gradient and
    steps are a fresh context's to the bit."""
    s = inputs.solar_system(N, seed=51)
    gr = np.ones((3, s.n))
    kw = dict(G=s.G, dt=s.dt, precision=precision, pair_once=pair_once)
    fresh = nb.NBody(s.r, s.v, s.m, **kw)
    assert fresh.pair_once_block == block
    want = [t.cpu().numpy() for t in fresh.grad(3, gr)]
    fresh.step(5)
    state = fresh.state.cpu().numpy()
    fresh.close()
    monkeypatch.setenv("NBODY_INJECT_WAIT_STALL", "2")
    b = nb.NBody(s.r, s.v, s.m, **kw)
    monkeypatch.delenv("NBODY_INJECT_WAIT_STALL")
    t0 = time.time()
    with pytest.raises(nb.NBodyError) as ei:
        b.grad(3, gr)
    assert ei.value.status == nb.NBODY_ETIMEOUT
    assert time.time() - t0 < 60
    for x, y in zip(b.grad(3, gr), want):
        assert np.array_equal(x.cpu().numpy(), y)
    b.step(5)
    assert np.array_equal(b.state.cpu().numpy(), state)
    b.close()


@pytest.mark.parametrize("n", [2049, 4352])
def test_both_forms_of_the_product(nb, n):
    """The pair-once product builds its term as f_q w_j - f_j w_q - 3 |d|^-2
    (f_q a + f_j b) d, the ordered one from u = mu_q w_j - mu_j w_q: the same
    rounding errors to a few FP32 ulps of the terms' magnitudes.  Against the
    FP64 gradient both keep the mixed gate, and the one's error stays within
    twice the other's in the root mean square over all elements (each 32-term
    sum rounds on its own, so the two differ by far less than that)."""
    s = inputs.solar_system(n, seed=23, moon_omega_dt_max=0.5)
    rng = np.random.default_rng(n)
    gr, gv = rng.normal(size=(3, n)), rng.normal(size=(3, n))
    ref = oracle.grad(s.G, s.dt, 2, s.r, s.v, s.m, gr, gv, openmp=True, magnitudes=True)
    rms = {}
    for once in (True, False):
        b = nb.NBody(s.r, s.v, s.m, G=s.G, dt=s.dt, precision="mixed", pair_once=once)
        assert b.pair_once_block == (128 if once else 0)
        got = [t.cpu().numpy() for t in b.grad(2, gr, gv)]
        b.close()
        for g, want, mag in zip(got, ref[:3], ref[3:]):
            assert np.all(np.abs(g - want) <= 1e-3 * mag)
        rms[once] = [np.sqrt(np.mean(((g - want) / mag) ** 2)) for g, want, mag in zip(got, ref[:3], ref[3:])]
    for a, b in zip(rms[True], rms[False]):
        assert a <= 2.0 * b, rms
