"""Edges of the launch rules and of the node update, compared with the general
path: block edges, sizes about a rule's line, special values."""
import numpy as np
import pytest

from paper_1701_00702_gb300 import inputs

pytestmark = pytest.mark.gpu
W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.fixture(scope="module")
def lbm():
    from paper_1701_00702_gb300 import lbm as m
    return m


def twin(lbm, s, form=0):
    t = lbm.Solver(s.params).set_step_form(form)
    t.load(s.save())
    return t


@pytest.mark.parametrize("nx", [3, 15, 16, 17, 31, 32, 33, 47, 48, 49, 65, 200])
def test_conduction_lanes_beyond_the_grid(lbm, nx):
    """Widths whose last block has lanes beyond the grid: in the last node's warp,
    in the block's other warp (nx mod 32 from 1 to 16: a whole warp without a
    node, which may touch no history) and none.  Hundreds of steps, graph
    replays among them, equal those of one thread per node."""
    p = inputs.conduction_1d(nx, 37, wall_kind=[0, 0, 1, 1], wall_T=[1.0, 0.0, 0.4, 0.7], T_solidus=0.29,
                             T_liquidus=0.31, L_char=100.0)
    _, G, H, dT = inputs.random_state(nx, 37, 5, seed=nx, H_range=(0.0, 1.6))
    s = lbm.Solver(p)
    s.set_state(None, G, H, dT)
    t = twin(lbm, s)
    b = lbm.Batch([t], autotune=False).configure(128, 0)
    s.step(197)
    b.step(197)
    assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()


@pytest.mark.parametrize("shape", [(512, 256), (513, 256), (545, 545), (577, 579), (1025, 1026), (1601, 1030)])
@pytest.mark.parametrize("prec,eq9", [(2, 0), (3, 0), (2, 1)])
def test_pairs_equal_one_node_per_thread(lbm, shape, prec, eq9):
    """16-bit runs about and above the sizes where automatic single steps take
    node pairs, with and without the prefetch and the evict-first reads: forms 0
    and 2 against form 1, which steps one node per thread, from a random state."""
    nx, ny = shape
    p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, L_char=100.0, Ra=1e7, wall_kind=[0, 1, 1, 0],
                      **(dict(ks_over_kl=0.7, cps_over_cpl=0.9) if eq9 else {}))
    p["nx"] = nx
    F, G, H, dT = inputs.random_state(nx, ny, 5, seed=nx, H_range=(0.0, 1.6), f_base=W9)
    s = lbm.Solver(p)
    s.set_state(F - W9[:, None, None], G, H, dT)
    runs = [twin(lbm, s, form) for form in (1, 0, 2)]
    for r in runs:
        r.step(3)
        assert r.status() == 0
    want = runs[0].save()
    assert np.array_equal(want, runs[1].save()) and np.array_equal(want, runs[2].save())


@pytest.mark.parametrize("shapes", [[(401, 333), (300, 290), (512, 200), (333, 300), (65, 900), (129, 64)],
                                    [(401, 333), (300, 290), (129, 64)]])
@pytest.mark.parametrize("prec,eq9", [(2, 0), (3, 1)])
def test_grouped_launches_on_both_sides_of_the_pair_rule(lbm, shapes, prec, eq9):
    """Map 4 over 558,000 and 235,000 nodes in 16-bit storage (node pairs, one
    node per thread), a bounce-back run among them: each run equals lbm_step's."""
    runs, twins = [], []
    for k, (nx, ny) in enumerate(shapes):
        p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, L_char=100.0, Ra=1e7, solid_scheme=1 if k == 1 else 0,
                          **(dict(ks_over_kl=0.7) if eq9 and k else {}))
        p["nx"] = nx
        F, G, H, dT = inputs.random_state(nx, ny, 5, seed=k, H_range=(0.0, 1.6), f_base=W9)
        s = lbm.Solver(p)
        s.set_state(F - W9[:, None, None], G, H, dT)
        runs.append(s)
        twins.append(twin(lbm, s, 1))
    b = lbm.Batch(runs, autotune=False).configure(128, 4)
    b.step(67)
    for s, t in zip(runs, twins):
        t.step(67)
        assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()


@pytest.mark.parametrize("prec,mapping", [(1, 3), (1, 4), (2, 3), (2, 4), (3, 4)])
def test_d2q9_batches_equal_their_runs(lbm, prec, mapping):
    """The register-capped D2Q9 kernels of single runs and of grouped launches,
    runs with Eq. 9 and with constant properties together: each equals lbm_step's."""
    runs, twins = [], []
    for k in range(10):
        nx, ny = 17 + 13 * k, 70 - 6 * k
        p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, thermal_q=9, L_char=100.0, Ra=1e7,
                          **(dict(ks_over_kl=0.7, cps_over_cpl=0.9) if k % 3 == 0 else {}))
        p["nx"] = nx
        F, G, H, dT = inputs.random_state(nx, ny, 9, seed=k, H_range=(0.0, 1.6), f_base=W9)
        s = lbm.Solver(p)
        s.set_state(F - W9[:, None, None], G, H, dT)
        runs.append(s)
        twins.append(twin(lbm, s, 1))
    b = lbm.Batch(runs, autotune=False).configure(128, mapping)
    b.step(67)
    for s, t in zip(runs, twins):
        t.step(67)
        assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()


@pytest.mark.parametrize("mapping", [0, 1, 2])
@pytest.mark.parametrize("prec,qt,flow", [(0, 5, 1), (0, 9, 1), (1, 5, 1), (1, 9, 1), (2, 5, 1), (2, 9, 1), (3, 5, 1), (3, 9, 1),
                                          (0, 5, 0), (1, 5, 0), (2, 9, 0)])
def test_tile_lists_equal_their_runs(lbm, prec, qt, flow, mapping):
    """Maps 0 to 2 in every storage type, lattice and with flow or without, runs
    with Eq. 9 and with constant properties together (the kernel with per-node
    rates serves both): each equals lbm_step's bit for bit."""
    runs, twins = [], []
    for k in range(7):
        nx, ny = 9 + 21 * k, 60 - 7 * k
        over = dict(ks_over_kl=0.7, cps_over_cpl=0.9) if k % 2 else {}
        p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, thermal_q=qt, L_char=100.0, Ra=1e7, flow=flow,
                          periodic_y=int(k == 2), **over)
        p["nx"] = nx
        F, G, H, dT = inputs.random_state(nx, ny, qt, seed=k, H_range=(0.0, 1.6), f_base=W9)
        s = lbm.Solver(p)
        s.set_state(F - W9[:, None, None] if flow else None, G, H, dT)
        runs.append(s)
        twins.append(twin(lbm, s, 1))
    b = lbm.Batch(runs, autotune=False).configure(64, mapping)
    b.step(69)
    for s, t in zip(runs, twins):
        t.step(69)
        assert s.status() == 0 and np.array_equal(s.save(), t.save())
    b.close()


@pytest.mark.parametrize("prec,flow", [(0, 1), (0, 0), (1, 1), (2, 1)])
def test_the_tallest_grid_steps(lbm, prec, flow):
    """65,536 rows, one more than a grid has blocks along y: single steps, graph
    replays and map 3 with one-row blocks equal the tile list."""
    p = inputs.cavity(100, precision=prec, flow=flow, L_char=100.0)
    p["nx"], p["ny"] = 3, 65536
    runs = [lbm.Solver(p) for _ in range(3)]
    lists = lbm.Batch([runs[1]], autotune=False).configure(128, 0)
    chain = lbm.Batch([runs[2]], autotune=False).configure(128, 3).set_block(0, 256, 1)
    runs[0].step(67)
    lists.step(67)
    chain.step(67)
    want = runs[0].save()
    assert all(r.status() == 0 for r in runs)
    assert all(np.array_equal(want, r.save()) for r in runs[1:])
    d = runs[0].diag()
    assert np.isfinite([d["melt_frac"], d["enthalpy"], d["mass"], d["nu_hot"]]).all()
    lists.close(), chain.close()


@pytest.mark.parametrize("nx,ny,prec,flow", [(577, 300, 2, 1), (200, 4, 0, 0)])
def test_block_shapes_of_runs_with_a_kernel_of_their_own(lbm, nx, ny, prec, flow):
    """Map 3 with a shape set for a run that otherwise takes node pairs or two
    lanes per node, the graph's steps and those outside it, against lbm_step."""
    p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, flow=flow, L_char=100.0, periodic_y=1 - flow)
    p["nx"] = nx
    s = lbm.Solver(p)
    for block in ((32, 8), (256, 1), (32, 2)):
        r = twin(lbm, s)
        b = lbm.Batch([r], autotune=False).configure(128, 3).set_block(0, *block)
        assert b.blocks() == [block]
        t = twin(lbm, s)
        b.step(131)
        t.step(131)
        assert np.array_equal(r.save(), t.save())
        b.close()


@pytest.mark.parametrize("kinds", [(0, 0, 1, 1), (1, 1, 0, 0)])
@pytest.mark.parametrize("shape", [(3, 3), (4, 5), (34, 21), (130, 8)])
@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("eq9", [0, 1])
def test_pairs_on_walls_round_as_single_nodes(lbm, shape, kinds, prec, eq9):
    """Fast flow next to walls, where the wall rule subtracts products: node pairs
    and two steps per launch against one node per thread, bit for bit."""
    nx, ny = shape
    p = inputs.cavity(max(nx, ny), ny=ny, precision=prec, L_char=100.0, Ra=1e7, wall_kind=list(kinds), porosity=0.85,
                      wall_T=[1.0, 0.0, 0.9, 0.1], **(dict(ks_over_kl=0.7, cps_over_cpl=0.9) if eq9 else {}))
    p["nx"] = nx
    F, G, H, dT = inputs.random_state(nx, ny, 5, seed=nx + eq9, H_range=(0.9, 1.9), u_amp=0.3, f_base=W9)
    s = lbm.Solver(p)
    s.set_state(F - W9[:, None, None], G, H, dT)
    runs = [twin(lbm, s, form) for form in (1, 2, 3)]
    for r in runs:
        r.step(4)
        assert r.status() == 0
    want = runs[0].save()
    assert np.array_equal(want, runs[1].save()) and np.array_equal(want, runs[2].save())
