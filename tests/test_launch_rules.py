"""The one-step kernel's launch rules on the CPU: which kernel and blocks a run
takes, from the library's own rule (tests/launch_rules.cu calls it)."""
import ctypes
import subprocess

import pytest

from paper_1701_00702_gb300 import build


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    lib = build.build()
    out = tmp_path_factory.mktemp("rules") / "launch_rules.so"
    src = build.ROOT / "tests" / "launch_rules.cu"
    subprocess.run([build.nvcc(), *build.GENCODE, "-std=c++20", "-O1", "-shared", "-Xcompiler", "-fPIC", "-I",
                    str(build.CSRC), "-o", str(out), str(src), str(lib), f"-Xlinker=-rpath={lib.parent}"],
                   check=True, capture_output=True)
    L = ctypes.CDLL(str(out))

    def step(nx, ny, prec, form=0, qt=5, flow=1, bounce=0, block=(0, 0)):
        o = (ctypes.c_int * 4)()
        L.rule_step(prec, qt, flow, bounce, nx, ny, form, *block, o)
        return tuple(o)

    step.lib = L
    return step


def takes_pairs(launch, nx):
    """Blocks of 32 x 4 threads that cover two columns each (no rule gives one
    node per thread blocks of 32 x 4)."""
    gx, _, bx, by = launch
    return (bx, by) == (32, 4) and gx == -(-nx // 64)


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("shape", [(512, 256), (577, 577), (1024, 1024), (1600, 1024), (2048, 2048)])
def test_single_is_one_node_per_thread(rules, shape, prec):
    """Form 1 keeps one node per thread at every size, form 2 pairs."""
    assert not takes_pairs(rules(*shape, prec, form=1), shape[0])
    assert takes_pairs(rules(*shape, prec, form=2), shape[0])


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("shape", [(577, 577), (640, 640), (1024, 1024), (2048, 2048)])
def test_automatic_single_steps_take_pairs(rules, shape, prec):
    for form in (0, 3):
        assert takes_pairs(rules(*shape, prec, form=form), shape[0])
        assert not takes_pairs(rules(*shape, prec, form=form, bounce=1), shape[0])
        assert not takes_pairs(rules(*shape, prec, form=form, qt=9), shape[0])
        assert not takes_pairs(rules(*shape, 1, form=form), shape[0])


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("shape,pairs", [
    # within a wave of one-node blocks, by the blocks of the busiest SM
    ((363, 361), 0), ((512, 256), 0), ((448, 300), 0), ((512, 340), 0), ((514, 256), 0), ((600, 240), 1), ((600, 300), 1),
    ((1000, 180), 1), ((900, 160), 1),
    # beyond it
    ((1000, 200), 1), ((512, 512), 1), ((128, 2000), 1), ((1024, 1024), 1), ((1606, 1000), 1),
    # odd widths: a second chain in the last node's warp, unless it is alone there
    ((333, 700), 0), ((593, 411), 0), ((515, 511), 0), ((777, 501), 1), ((1201, 301), 1), ((865, 801), 1),
    ((513, 300), 1), ((577, 577), 1), ((65, 3000), 1),
])
def test_automatic_pairs_where_they_are_the_faster(rules, shape, pairs, prec):
    assert takes_pairs(rules(*shape, prec), shape[0]) == bool(pairs)


@pytest.mark.parametrize("prec", [2, 3])
def test_grouped_launches_take_pairs_where_nodes_abound(rules, prec):
    """Batches whose grouped runs have few nodes together step one node per
    thread: there one warp's chain is the time, which pairs lengthen."""
    pairs = lambda nodes, prec=prec, qt=5, flow=1: rules.lib.rule_group_pairs(prec, qt, flow, ctypes.c_longlong(nodes))
    assert not any(pairs(n) for n in (9, 17416, 114024, 284456, 380495))
    assert all(pairs(n) for n in (560742, 1 << 20, 1 << 30))
    assert not pairs(1 << 20, prec=1) and not pairs(1 << 20, qt=9) and not pairs(1 << 20, flow=0)


SHAPES = [(0, 0), (128, 2), (64, 4), (32, 8), (256, 1), (128, 1), (64, 2), (32, 4), (64, 1), (32, 2)]


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(3, 65536), (128, 65536), (1000, 65536), (128, 65535), (65536, 3)])
def test_grids_stay_within_the_launch_limits(rules, nx, ny, prec):
    """65,536 rows are admitted, 65,535 blocks along y: the run's own block shape
    and every shape a batch may choose cover the grid within the limit."""
    for qt, flow in ((5, 1), (5, 0), (9, 1)):
        for form in (0, 1, 2):
            for block in SHAPES:
                launch = rules(nx, ny, prec, form=form, qt=qt, flow=flow, block=block)
                gx, gy, bx, by = launch
                assert gy <= 65535 and gy * by >= ny and bx * by <= 256
                assert gx * bx * (2 if takes_pairs(launch, nx) else 1) >= nx


@pytest.mark.parametrize("block", SHAPES[1:])
def test_a_chosen_block_shape_is_the_one_launched(rules, block):
    """One node per thread in the chosen shape, also in runs whose own kernel
    would be node pairs or two lanes per node; pairs by form or size stay."""
    bx, by = block
    for nx, ny, prec, form, flow in ((512, 512, 2, 0, 1), (1024, 1000, 3, 0, 1), (600, 600, 2, 1, 1), (256, 256, 1, 0, 1),
                                     (200, 4, 0, 0, 0), (700, 700, 0, 0, 1)):
        assert rules(nx, ny, prec, form=form, flow=flow, block=block) == (-(-nx // bx), -(-ny // by), bx, by)
    for nx, ny, form in ((2048, 2048, 0), (256, 256, 2)):
        assert takes_pairs(rules(nx, ny, 2, form=form, block=block), nx)


@pytest.mark.parametrize("shape,block", [
    ((64, 64), (64, 2)), ((200, 200), (64, 2)), ((256, 256), (128, 1)), ((360, 360), (128, 1)), ((160, 300), (128, 1)),
    ((137, 689), (32, 2)), ((290, 420), (64, 1)), ((190, 660), (64, 1)), ((24, 2000), (32, 2)), ((400, 390), (32, 2)),
    ((512, 512), (128, 1)),
])
def test_blocks_leave_few_columns_idle_beyond_a_wave(rules, shape, block):
    """Where blocks of 128 x 1 are more than a wave, by nodes or by idle columns,
    the widest of 128, 64 and 32 that leaves the fewest columns idle."""
    for prec, qt in ((1, 5), (1, 9), (2, 9)):
        assert rules(*shape, prec, form=1, qt=qt)[2:] == block
