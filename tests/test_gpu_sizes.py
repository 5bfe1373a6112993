"""Sizes on both sides of the lines at which the kernels change how they split
their work, against the FP64 oracle (Sec. 2.2, Sec. 2.3, Appendix B).

Tolerances are those of the paths' own parity tests: FP64 1e-11 of the largest
magnitude (only summation orders differ); mixed 2e-5 for forces and
correlators, 1e-4 for the ionic per-particle energies and virials (sums of
large cancelling FP32 terms)."""
import numpy as np
import pytest

from paper_2503_07526_gb300 import synth
from test_gpu_corr import compare, series
from test_gpu_ionic import ALPHA, MASSES, reference, system  # noqa: F401 (fixture)
from test_gpu_ionic import params as ionic_params
from test_gpu_md import F_AT_RC, check_mixed_forces, jittered, params, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_07526_gb300 as pkg

    pkg.lib(build=True)
    return pkg


@pytest.mark.parametrize("skin", [0.05, 0.3])
@pytest.mark.parametrize("L", [32.0, 41.7])
def test_fp64_pairs_next_to_the_cutoff(pkg, oracle_mod, L, skin):
    """Dimers whose separations lie 1e-9, 1e-7 and 1e-5 rc inside and outside
    the cutoff, at every place of the box: the lists are selected in FP32 with
    an error band, the cutoff itself is decided in FP64."""
    k = np.arange(64)
    at = (np.stack([k % 4, k // 4 % 4, k // 16]) + 0.5) * (L / 4) + 0.5 * (synth.uniform01(3, 192).reshape(3, 64) - 0.5)
    u = synth.uniform01(4, 192).reshape(3, 64) - 0.5
    off = np.array([1e-9, -1e-9, 1e-7, -1e-7, 1e-5, -1e-5])[k % 6]
    b = at + u / np.sqrt((u ** 2).sum(0)) * 2.5 * (1.0 + off)
    r = np.mod(np.concatenate([at, b], axis=1), L)
    s = dict(n=128, L=L)
    g = pkg.System(params(pkg, s, precision=pkg.MD_PREC_FP64, skin=skin), r, np.zeros_like(r))
    got = g.particles()
    F, e, W = oracle_mod.lj_forces(r, L, method="cells")
    assert ((F ** 2).sum(0) > 0).sum() == 2 * (off < 0).sum()  # half of the dimers interact
    assert np.array_equal((got["F"] ** 2).sum(0) > 0, (F ** 2).sum(0) > 0)
    assert rel(got["F"], F) <= 1e-11
    assert np.abs(got["epot"] - e).max() <= 1e-11 * 2.5 * abs(F_AT_RC)
    assert rel(got["W"], W) <= 1e-11


@pytest.mark.parametrize("cells", [3, 16, 17, 18, 25, 27])
@pytest.mark.parametrize("kind", ["fp64", "tiles"])
def test_forces_and_reduction_over_sizes(pkg, oracle_mod, cells, kind):
    """108 atoms; 16,384 and 19,652 (the sort within one cluster ends at the
    first; the list build's warps per chunk and the tiles' CTAs change about
    there); 23,328, 62,500 and 78,732 (10, 15 and 16 cells per side, segments
    of unlike length): forces, energies, virials and the reduction after two
    steps, at the GPU's own positions."""
    s = jittered(cells, seed=cells, rho=0.8442 if cells > 3 else 0.15)
    if kind == "tiles":
        if cells == 3:
            s = jittered(5, seed=cells, rho=0.7)  # the tile path takes 3 cells per side at least
        p = params(pkg, s, precision=pkg.MD_PREC_MIXED, pair_mode=pkg.MD_PAIR_TILES)
    else:
        p = params(pkg, s, precision=pkg.MD_PREC_FP64)
    g = pkg.System(p, s["r"], s["v"])
    g.step(2)
    got, obs = g.particles(), g.observables()
    F, e, W = oracle_mod.lj_forces(got["r"], s["L"], method="cells")
    if kind == "fp64":
        assert rel(got["F"], F) <= 1e-11
        assert rel(got["epot"], e) <= 1e-11
        assert rel(got["W"], W) <= 1e-11
    else:
        check_mixed_forces(got["F"], F, got["r"], s["L"], oracle_mod)
    want = oracle_mod.observables(s["L"] ** 3, np.ones(s["n"]), got["v"], got["epot"], got["W"])
    assert obs["U"] == pytest.approx(want[0], rel=1e-10)
    assert rel(obs["sigma"], want[3:9]) <= 1e-10
    assert rel(obs["q"], want[9:12]) <= 1e-10


@pytest.mark.parametrize("kind", ["fp64", "tiles"])
def test_replicas_of_unlike_size_equal_replicas_run_alone(pkg, kind):
    """2,048 + 19,652 + 500 atoms in one handle: together they take the sort of
    several launches and the scan per replica, alone the small ones take the
    cluster's; the tile path agrees bit for bit, FP64 within summation order."""
    reps = []
    for k, (cells, rho) in enumerate(((8, 0.8), (17, 0.8442), (5, 0.7))):
        t = jittered(cells, seed=60 + k, rho=rho, T=1.2, amp=0.15)
        reps.append(dict(r=t["r"], v=t["v"], box=t["L"], n=t["n"]))
    kw = dict(precision=pkg.MD_PREC_FP64) if kind == "fp64" else dict(precision=pkg.MD_PREC_MIXED, pair_mode=pkg.MD_PAIR_TILES)
    kw.update(skin=0.2, stress=(6, 16, 2, 1), heatflux=(6, 16, 2, 1), vacf=None)
    b = pkg.System(pkg.make_params(1, 1.0, **kw), replicas=reps)
    b.step(20)
    got, a0 = b.particles(), 0
    for rp in reps:
        alone = pkg.System(pkg.make_params(rp["n"], rp["box"], **kw), rp["r"], rp["v"])
        alone.step(20)
        want = alone.particles()
        for key in ("r", "v", "F", "W"):
            x = got[key][..., a0:a0 + rp["n"]]
            assert np.array_equal(x, want[key]) if kind == "tiles" else rel(x, want[key]) <= 1e-13, key
        a0 += rp["n"]


_MESH = {}


@pytest.mark.parametrize("precision,copies,order", [(0, 1, 4), (0, 2, 6), (0, 3, 8), (0, 4, 6),
                                                    (1, 1, 6), (1, 2, 4), (1, 3, 8), (1, 4, 4)])
def test_ionic_sizes_and_orders_match_oracle(pkg, system, precision, copies, order):  # noqa: F811
    """1,728 to 110,592 ions: 32, 64 and 128 ions per chunk of the spread and
    gather, spline orders 4, 6 and 8.  The larger systems are the small one
    copied side by side on a mesh as many times finer, whose forces, energies
    and virials are the small one's."""
    from oracle import ewald

    s = system
    if order not in _MESH:
        q = np.where(s["types"] == 0, 1.0, -1.0)
        r = np.mod(s["r"], s["L"])
        base = reference(s, 16)  # real-space and self terms; its mesh terms are exchanged for this order's
        F8, E8, W8, _, _ = ewald.spme_reciprocal(r, q, s["L"], alpha=ALPHA, K=16, order=8)
        Fk, Ek, Wk, _, _ = ewald.spme_reciprocal(r, q, s["L"], alpha=ALPHA, K=16, order=order)
        _MESH[order] = dict(F=base["F"] - F8 + Fk, epot=base["epot"] - E8 + Ek, W=base["W"] - W8 + Wk)
    ref, c = _MESH[order], copies
    shift = s["L"] * np.stack(np.meshgrid(*[np.arange(c)] * 3, indexing="ij")).reshape(3, -1).astype(float)
    r = (np.mod(s["r"], s["L"])[:, None, :] + shift[:, :, None]).reshape(3, -1)
    big = dict(n=s["n"] * c ** 3, L=s["L"] * c)
    p = ionic_params(pkg, big, precision, mesh=16 * c)
    p.order = order
    g = pkg.System(p, r, np.tile(s["v"], (1, c ** 3)), types=np.tile(s["types"], c ** 3))
    got = g.particles()
    g.close()
    for key, t in (("F", 1e-11 if precision == 0 else 2e-5), ("epot", 1e-11 if precision == 0 else 1e-4),
                   ("W", 1e-11 if precision == 0 else 1e-4)):
        want = np.tile(ref[key], (1, c ** 3) if ref[key].ndim == 2 else c ** 3)
        assert rel(got[key], want) <= t, key


def chunk_volumes(r, L, mesh, order, chunk=32):
    """Mesh points of the box that each 32 consecutive ions of a cell row reach,
    in the order of the sort (cells of rc + skin = 11 A, x fastest, then octant
    and number)."""
    nc = int(L // 11.0)
    e = L / nc
    c = np.minimum((r / e).astype(int), nc - 1)
    octant = ((r >= (c + 0.5) * e) * np.array([[1], [2], [4]])).sum(0)
    row = c[2] * nc + c[1]
    at = np.lexsort((np.arange(r.shape[1]), octant, c[0], row))
    u = np.floor(r * (mesh / L)).astype(int)
    out = []
    for k in range(nc * nc):
        mine = at[row[at] == k]
        for a in range(0, len(mine), chunk):
            x = u[:, mine[a:a + chunk]]
            out.append(np.prod(x.max(1) - x.min(1) + order))
    return np.array(out)


@pytest.mark.parametrize("order", [4, 6, 8])
@pytest.mark.parametrize("precision", [0, 1])
def test_ionic_meshes_too_fine_for_the_tiles(pkg, system, precision, order):  # noqa: F811
    """192 mesh points over three cells: every chunk reaches more points than the
    largest shared tile of the spread (160 KB, a value a point) and of the gather
    (two) holds, so charges go straight to the global mesh and are read from
    there: forces, energies and virials against the oracle, and two runs bit for
    bit.  The mixed form's virials carry the FP32 rounding of the mesh times
    second derivatives of the weights, that is (K / L)^2: the bound of the tests
    with 32 points times (K / 32)^2."""
    from oracle import ewald

    s, K = system, 192
    r = np.mod(s["r"], s["L"])
    assert chunk_volumes(r, s["L"], K, order).min() > 160 * 1024 / 4
    if (K, order) not in _MESH:
        q = np.where(s["types"] == 0, 1.0, -1.0)
        base = reference(s, 16)  # real-space and self terms; its mesh terms are exchanged
        F8, E8, W8, _, _ = ewald.spme_reciprocal(r, q, s["L"], alpha=ALPHA, K=16, order=8)
        Fk, Ek, Wk, _, _ = ewald.spme_reciprocal(r, q, s["L"], alpha=ALPHA, K=K, order=order)
        _MESH[K, order] = dict(F=base["F"] - F8 + Fk, epot=base["epot"] - E8 + Ek, W=base["W"] - W8 + Wk)
    want = _MESH[K, order]
    p = ionic_params(pkg, s, precision, mesh=K)
    p.order = order
    after = []
    for _ in range(2):
        g = pkg.System(p, s["r"], s["v"], types=s["types"])
        got = g.particles()
        for key, t in (("F", 1e-11 if precision == 0 else 2e-5), ("epot", 1e-11 if precision == 0 else 1e-4),
                       ("W", 1e-11 if precision == 0 else 1e-4 * (K / 32) ** 2)):
            assert rel(got[key], want[key]) <= t, key
        g.step(5)
        after.append(g.particles())
        g.close()
    for key in ("r", "v", "F", "W", "epot"):
        assert np.array_equal(after[0][key], after[1][key]), key


@pytest.mark.parametrize("b,p,m,ns,gs,prec,S", [
    (4, 16, 2, 4864, 2432, 0, 100), (4, 16, 2, 4865, 973, 0, 100), (3, 32, 2, 4864, 1216, 1, 90),
    (3, 32, 4, 4866, 811, 1, 90), (2, 16, 2, 300002, 150001, 1, 40), (2, 16, 2, 600000, 200000, 1, 40),
    (2, 8, 2, 300000, 100000, 0, 24)])
def test_corr_push_over_series_counts(pkg, oracle_mod, b, p, m, ns, gs, prec, S):
    """A warp per series up to 4,864 series, a thread per one, two or four
    series above (by the count and its divisibility)."""
    x = series(ns, S, seed=ns)
    g = pkg.Corr.create(b, p, m, ns, gs, False, prec)
    o = oracle_mod.Corr(b, p, m, ns, gs, False)
    for t in range(S):
        g.push(x[t])
        o.push(x[t])
    compare(pkg, g, o, ns // gs, prec)
    g.close()


def dilute(n, cells, seed):
    """n atoms on a jittered cubic lattice in a box of `cells` cells per side."""
    L = 2.8 * cells * 1.001
    k = int(np.ceil(n ** (1.0 / 3.0) - 1e-9))
    at = np.linspace(0, k ** 3 - 1, n).astype(np.int64)
    r = (np.stack([at % k, at // k % k, at // (k * k)]) + 0.5) * (L / k)
    r = r + 0.2 * (synth.uniform01(seed, 3 * n).reshape(3, n) - 0.5)
    return dict(r=np.ascontiguousarray(np.mod(r, L)), v=synth.maxwell_velocities(n, 1.5, seed), L=L, n=n)


@pytest.mark.parametrize("kind", ["fp64", "verlet", "tiles"])
@pytest.mark.parametrize("n,cells", [(3000, 10), (3000, 11), (257, 24), (16384, 10), (16384, 32)])
def test_sort_of_dilute_systems(pkg, oracle_mod, n, cells, kind):
    """1,000 cells (the last sort within one cluster is at 1,024) and 1,331 to
    32,768, most of them empty in the larger boxes: forces after steps with
    rebuilds, at the GPU's own positions."""
    s = dilute(n, cells, seed=cells)
    kw = dict(fp64=dict(precision=pkg.MD_PREC_FP64), verlet=dict(precision=pkg.MD_PREC_MIXED),
              tiles=dict(precision=pkg.MD_PREC_MIXED, pair_mode=pkg.MD_PAIR_TILES))[kind]
    g = pkg.System(params(pkg, s, vacf=None, dt=0.02, **kw), s["r"], s["v"])
    g.step(12)
    got = g.particles()
    assert g.observables()["rebuilds"] >= 2
    g.close()
    F, e, W = oracle_mod.lj_forces(got["r"], s["L"], method="cells")
    if not F.any():  # the 257 atoms of the largest cells per atom: no pair in range
        assert not got["F"].any()
    elif kind == "fp64":
        assert rel(got["F"], F) <= 1e-11
        assert rel(got["W"], W) <= 1e-11
    else:
        check_mixed_forces(got["F"], F, got["r"], s["L"], oracle_mod)


def test_dilute_sort_time_has_no_step_at_the_small_sort(pkg):
    """16,384 atoms in 96^3 cells are on one side of the small sort's line by
    atoms, 16,385 on the other: a step takes the same time on both (it took
    four times as long below the line when cells did not count)."""
    import time

    best = []
    for n in (16384, 16385):
        s = dilute(n, 96, seed=3)
        g = pkg.System(params(pkg, s, vacf=None, precision=pkg.MD_PREC_MIXED), s["r"], s["v"])
        took = []
        for _ in range(5):
            t = time.perf_counter()
            g.step(32)
            g.observables()
            took.append(time.perf_counter() - t)
        best.append(min(took))
        g.close()
    assert best[0] <= 2.0 * best[1]


@pytest.mark.parametrize("p,m,ns", [(2, 2, 1216), (2, 2, 1217), (4, 2, 1216), (4, 2, 1217), (4, 4, 4864), (4, 2, 4865),
                                    (6, 2, 4864)])
@pytest.mark.parametrize("cross", [False, True])
@pytest.mark.parametrize("prec", [0, 1])
def test_corr_push_of_few_lags(pkg, oracle_mod, p, m, ns, cross, prec):
    """Up to four lags a warp per series ends at 1,216 series in FP64, else at
    4,864."""
    x, y = series(ns, 70, seed=ns + p), series(ns, 70, seed=ns + p + 1)
    g = pkg.Corr.create(4, p, m, ns, cross=cross, precision=prec)
    o = oracle_mod.Corr(4, p, m, ns, 1, cross)
    for t in range(70):
        g.push(x[t], y[t] if cross else None)
        o.push(x[t], y[t] if cross else None)
    gv, gc, gu = g.raw()
    ov, oc, ou = o.raw()
    assert gu == ou and np.array_equal(gc, oc)
    gv, ov = np.reshape(gv, -1), np.reshape(ov, -1)
    assert np.abs(gv - ov).max() <= (1e-11 if prec == 0 else 2e-5) * np.abs(ov).max()
    g.close()


def test_push_time_of_few_lags_has_no_step_at_the_warps_line(pkg):
    """FP64 correlators of two lags with 4,864 and 4,865 series take the same
    time a push (7.5 and 5.7 us where the warps went on to 4,864 at any number
    of lags)."""
    import time

    import torch

    best = []
    for ns in (4864, 4865):
        g = pkg.Corr.create(4, 2, 2, ns, precision=0)
        rows = list(torch.randn(256, ns, device="cuda", dtype=torch.float64))
        took = []
        for _ in range(12):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for row in rows:
                g.push(row)
            torch.cuda.synchronize()
            took.append(time.perf_counter() - t)
        best.append(min(took))
        g.close()
    assert best[0] <= 1.15 * best[1]
