"""The resident loop's plan, built and checked on the host: every link, face row and
writer of its tiles, the symmetry that its exchange relies on, and its limits."""
import pytest

from paper_1812_00390_gb300 import meshgen as mg


@pytest.fixture(scope="module")
def fv():
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1812_00390_gb300 import fvlbm
    return fvlbm


# tiles per SM (152 SMs, of a GB300 or when no GPU answers) and tile size; 0: none
CASES = [
    ("fp32", lambda: mg.two_triangles(), 1, 128), ("fp32", lambda: mg.couette(40, 1), 1, 128),
    ("fp32", lambda: mg.channel(nx=30, ny=17, top_bottom="symmetry"), 1, 128),
    ("fp32", lambda: mg.cavity(128, 20.0), 1, 256), ("fp16", lambda: mg.cavity(200, 20.0), 2, 256),
    ("fp32", lambda: mg.cylinder_hybrid(), 3, 256), ("bf16", lambda: mg.cavity(300, 20.0), 4, 256),
    ("fp32", lambda: mg.cavity(310, 20.0), 4, 256), ("fp32", lambda: mg.cavity(321, 20.0), 0, 0),
    ("fp32", lambda: mg.periodic_tri(235, 235, lx=235.0, ly=235.0), 4, 256),
    ("fp32", lambda: mg.bricks(160, 80), 1, 128), ("fp32", lambda: mg.bricks(460, 230), 2, 256),
    ("fp64", lambda: mg.two_triangles(periodic=True), 1, 64), ("fp64", lambda: mg.couette(), 1, 64),
    ("fp64", lambda: mg.cavity(64, 20.0), 1, 64), ("fp64", lambda: mg.cavity(75, 20.0), 0, 0),
    ("fp64", lambda: mg.bricks(130, 65), 1, 64),
    ("fp64", lambda: mg.periodic_tri(53, 53, lx=53.0, ly=53.0), 1, 64),
]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_resident_plan_checks(fv, k):
    prec, make, per_sm, tile = CASES[k]
    m = make()
    p = fv.make_params(0.1, scheme="rk2", precision=prec)
    i = fv.plan_info(fv.Mesh(m), p, resident=True)
    assert i["violations"] == 0, i.get("first_violation")
    assert i["stage_kernel"] == tile and -(-i["n_tiles"] // 152) == per_sm
    if tile:
        assert i["n_tiles"] * i["mean_tile_cells"] == pytest.approx(m.n_cell)
        assert i["mean_tile_cells"] + i["mean_ring1_cells"] <= tile
        assert i["max_local_cells"] <= 3 * tile // 2 + 64
    none = fv.plan_info(fv.Mesh(m), fv.make_params(0.1, scheme="rk2", precision=prec, kernel=128), resident=True)
    assert none["stage_kernel"] == 0 and none["n_tiles"] == 0 and none["violations"] == 0


def test_tiles_of_the_length_asked_for_are_not_short(fv):
    """28,800 triangles on 152 SMs: every tile is an SM's share of the cells, none was cut
    by the capacity; nearly full, they serve the stage kernels of the automatic choice too."""
    h = fv.Mesh(mg.periodic_tri(120, 120, lx=120.0, ly=120.0))
    p = fv.make_params(0.1, scheme="rk2", precision="fp32")
    for resident in (False, True):
        i = fv.plan_info(h, p, resident=resident)
        assert i["stage_kernel"] == 256 and i["n_tiles"] == 152 and i["short_tiles"] == 0


def test_stage_kernels_have_full_tiles_where_the_loop_has_short_ones(fv):
    h = fv.Mesh(mg.cavity(128, 20.0))
    auto, own = (fv.plan_info(h, fv.make_params(0.1, scheme="rk2", precision="fp32", kernel=k)) for k in (0, 256))
    assert auto == own and auto["mean_tile_cells"] > 150
    assert fv.plan_info(h, fv.make_params(0.1, scheme="rk2", precision="fp32"), resident=True)["mean_tile_cells"] < 110
