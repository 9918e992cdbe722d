"""One update, several kernels: node pairs, two steps per launch, grouped
launches and the tile lists give each node the same bits as one node per
thread, at the sizes and walls where they could differ (odd widths, ragged
blocks, every kind of wall on every side); and the diagnostics' FP64 sums
against the fields they are made of."""
import numpy as np
import pytest

from paper_1701_00702_gb300 import inputs

pytestmark = pytest.mark.gpu
W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


@pytest.fixture(scope="module")
def lbm():
    from paper_1701_00702_gb300 import lbm as m
    return m


def random_run(lbm, nx, ny, prec, seed, qt=5, **over):
    p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, thermal_q=qt, L_char=100.0, Ra=1e7, **over)
    p["nx"] = nx
    F, G, H, dT = inputs.random_state(nx, ny, qt, seed=seed, H_range=(0.0, 1.6), f_base=W9[:, 0, 0])
    s = lbm.Solver(p)
    s.set_state(F - W9, G, H, dT)
    return s


def twin(lbm, s, form):
    t = lbm.Solver(s.params).set_step_form(form)
    t.load(s.save())
    return t


@pytest.mark.parametrize("kinds", [(0, 0, 1, 1), (1, 1, 0, 0), (1, 1, 1, 1), (1, 0, 0, 1), (0, 1, 1, 0)])
@pytest.mark.parametrize("shape", [(3, 3, 0, 0), (4, 3, 0, 0), (31, 13, 0, 0), (64, 12, 0, 0), (33, 8, 0, 1), (130, 7, 0, 1),
                                   (66, 9, 1, 0), (2, 5, 1, 0)])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_step_forms_give_the_same_bits(lbm, shape, kinds, prec):
    """Forms 1 (one step per launch), 2 (node pairs) and 3 (two steps per launch)
    from a random state, four steps: equal checkpoints."""
    nx, ny, px, py = shape
    s = random_run(lbm, nx, ny, prec, seed=nx * 31 + ny, periodic_x=px, periodic_y=py, wall_kind=list(kinds),
                   wall_T=[1.0, 0.0, 0.3, 0.6])
    runs = [twin(lbm, s, form) for form in (1, 2, 3)]
    for r in runs:
        r.step(4)
        assert r.status() == 0
    want = runs[0].save()
    for r in runs[1:]:
        assert np.array_equal(want, r.save())


@pytest.mark.parametrize("shape", [(287, 301), (320, 320), (334, 303), (65, 1400), (256, 242)])
@pytest.mark.parametrize("prec,q,eq9", [(1, 5, 0), (1, 9, 0), (2, 5, 0), (2, 9, 0), (3, 5, 1)])
def test_two_step_builds_of_tall_tiles(lbm, shape, prec, q, eq9):
    """Tiles of 12 to 15 rows: two per SM at registers capped for it (16-bit,
    D2Q9), one per SM, and the many-tiles build, against one step per launch."""
    s = random_run(lbm, *shape, prec, seed=9, qt=q, **(dict(ks_over_kl=0.7) if eq9 else {}))
    a, b = twin(lbm, s, 1), twin(lbm, s, 3)
    a.step(4)
    b.step(4)
    assert b.status() == 0 and np.array_equal(a.save(), b.save())


@pytest.mark.parametrize("shape,prec,q,form,bounce", [
    ((769, 701), 1, 5, 1, 0), ((641, 643), 1, 9, 1, 0), ((900, 874), 1, 5, 3, 0), ((1011, 999), 2, 5, 1, 0),
    ((1301, 1210), 2, 5, 2, 0), ((1000, 803), 3, 9, 1, 0), ((1000, 1003), 3, 5, 1, 1)])
def test_reads_marked_evict_first(lbm, shape, prec, q, form, bounce):
    """Grids whose state is about L2's size, where lbm_step marks its reads
    evict-first, against a batch of one run, which does not."""
    s = random_run(lbm, *shape, prec, seed=3, qt=q, solid_scheme=bounce)
    a, b = twin(lbm, s, form), twin(lbm, s, 1)
    batch = lbm.Batch([b], autotune=False).configure(128, 3)
    a.step(4)
    batch.step(64)   # (the graph's launches)
    a.step(60)
    assert a.status() == 0 and np.array_equal(a.save(), b.save())
    batch.close()


@pytest.mark.parametrize("prec,q,mapping,shape", [(2, 5, 4, (701, 720)), (1, 5, 5, (501, 524)), (1, 5, 4, (501, 524)),
                                                 (3, 9, 4, (611, 600)), (1, 9, 5, (433, 480))])
def test_grouped_reads_marked_evict_first(lbm, prec, q, mapping, shape):
    """Two runs whose states are about L2's size together, in grouped launches
    that mark their reads, against lbm_step on each, which does not."""
    runs = [random_run(lbm, *shape, prec, seed=k, qt=q) for k in (1, 2)]
    twins = [twin(lbm, s, 1) for s in runs]
    b = lbm.Batch(runs, autotune=False).configure(128, mapping)
    b.step(66)
    for s, t in zip(runs, twins):
        t.step(66)
        assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()


@pytest.mark.parametrize("shape", [(1025, 768), (900, 874)])
def test_two_steps_with_prefetch_beyond_l2(lbm, shape):
    """FP32 grids of at least 786,432 nodes, whose two-step tiles prefetch rows
    ahead: ragged chunks and a last tile row, against one step per launch."""
    s = random_run(lbm, *shape, 1, seed=5)
    a, b = twin(lbm, s, 1), twin(lbm, s, 3)
    a.step(4)
    b.step(4)
    assert b.status() == 0 and np.array_equal(a.save(), b.save())


@pytest.mark.parametrize("prec", [2, 3])
def test_plain_pairs_at_their_threshold(lbm, prec):
    """16-bit runs of 131,072 nodes and more take node pairs in one step per
    launch; pairs with the prefetch kernel's form give the same bits."""
    for nx, ny in ((512, 256), (513, 256), (511, 256)):
        s = random_run(lbm, nx, ny, prec, seed=nx)
        a, b = twin(lbm, s, 1), twin(lbm, s, 2)
        a.step(3)
        b.step(3)
        assert np.array_equal(a.save(), b.save())


@pytest.mark.parametrize("prec,mapping", [(0, 4), (1, 4), (1, 5), (2, 4), (2, 5), (3, 4), (1, 0), (2, 1)])
@pytest.mark.parametrize("count", [1, 3, 9, 27])
def test_batches_follow_their_runs_bit_for_bit(lbm, prec, mapping, count):
    """Groups of every size class (one run, few, one group's worth and more),
    odd sides, a bounce-back run among the others, graph replays and the steps
    outside them, a run whose step form changes and one that steps alone in
    between (the kept launches are dropped): each run equals lbm_step's."""
    rng = np.random.default_rng(count)
    runs, twins = [], []
    for k in range(count):
        nx, ny = int(rng.integers(3, 90)), int(rng.integers(3, 40))
        s = random_run(lbm, nx, ny, prec, seed=k, periodic_y=k % 2, solid_scheme=1 if k == 2 else 0)
        runs.append(s)
        twins.append(twin(lbm, s, 1))
    b = lbm.Batch(runs, autotune=False).configure(128, mapping)

    def both(n):
        b.step(n)
        for t in twins:
            t.step(n)

    both(5)
    both(131)
    runs[0].set_step_form(1)
    both(6)
    runs[-1].step(1)
    twins[-1].step(1)
    both(7)
    for s, t in zip(runs, twins):
        assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (3, 3, 0, 0), (127, 5, 0, 1), (129, 300, 0, 0), (640, 410, 0, 0), (1030, 515, 0, 1)])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_diagnostics_are_the_sums_of_the_fields(lbm, shape, prec):
    """One, four and eight rows per thread, with and without walls: melt
    fraction, enthalpy, mass and the wall's Nusselt number against numpy sums of
    the fields.  The fields of the FP32 and 16-bit forms are rounded to FP32
    (2^-24 each), the diagnostics' terms are not; the Nusselt number's flux
    takes differences of temperatures (3, -4, 1)."""
    nx, ny, px, py = shape
    s = random_run(lbm, nx, ny, prec, seed=ny, periodic_x=px, periodic_y=py)
    s.step(2)
    f = {k: v.astype(np.float64) for k, v in s.fields(device=False).items()}
    d, c, p = s.diag(), s.derived(), s.params
    phi, tol = p["porosity"], 1e-13 if prec == 0 else 2.0 ** -23
    E = phi * f["H_f"].sum() + (1 - phi) * c["rho_m"] * f["T_s"].sum()
    assert abs(d["melt_frac"] - f["f_l"].mean()) <= 1e-13
    assert abs(d["enthalpy"] - E) <= tol * (phi * np.abs(f["H_f"]).sum() + (1 - phi) * c["rho_m"] * np.abs(f["T_s"]).sum())
    assert abs(d["mass"] - f["rho"].sum()) <= tol * nx * ny
    if px:
        assert np.isnan(d["nu_hot"])
    else:
        g = [0.5 * (3 * f[k][:, 0] - 4 * f[k][:, 1] + f[k][:, 2]) for k in ("T_f", "T_s")]
        k_e = phi * p["k_f"] + (1 - phi) * c["k_m"]
        nu = p["L_char"] / k_e * (phi * p["k_f"] * g[0] + (1 - phi) * c["k_m"] * g[1]).mean()
        assert abs(d["nu_hot"] - nu) <= 1e-11 * max(1.0, abs(nu))


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (3, 3, 0, 0), (31, 5, 0, 1), (33, 4, 1, 0), (200, 4, 0, 1), (97, 100, 0, 0),
                                   (608, 16, 0, 1), (609, 16, 0, 1)])
@pytest.mark.parametrize("kinds", [(0, 0, 1, 1), (1, 0, 0, 1)])
def test_conduction_lanes_equal_one_node_per_thread(lbm, shape, kinds):
    """FP64 runs without flow up to 9,728 nodes step with two lanes per node; the
    tile-list batch steps one node per thread.  Equal checkpoints after five
    steps, on both sides of the limit and with either wall on every side."""
    nx, ny, px, py = shape
    p = inputs.conduction_1d(nx, ny, periodic_x=px, periodic_y=py, wall_kind=list(kinds), wall_T=[1.0, 0.0, 0.4, 0.7],
                             T_solidus=0.29, T_liquidus=0.31, L_char=100.0)
    _, G, H, dT = inputs.random_state(nx, ny, 5, seed=nx + ny, H_range=(0.0, 1.6))
    s = lbm.Solver(p)
    s.set_state(None, G, H, dT)
    t = twin(lbm, s, 0)
    b = lbm.Batch([t], autotune=False).configure(128, 0)
    s.step(5)
    b.step(5)
    assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()
