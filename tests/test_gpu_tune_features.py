"""The features that the autotuner hands to its cost model are those of the launches a call makes:
d3 tile by the momenta's classes in the FP64 form, row-factored columns by the call's own momenta and
grouped spin terms in the Ozaki form (index 6: slabs, index 7: units per SM, index 9: padded columns)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M9 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0)]
PAIRS = [(0, 1, 0), (1, 0, 0), (2, 3, 2), (3, 2, 2)]


def tune(form, L, nd, mom, options):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)

    def gauss(*shape):
        return torch.complex(*(torch.randn(*shape, generator=gen, dtype=torch.float64, device="cuda") for _ in "ri"))

    V, phi = gauss(1, 4, L ** 3, 3), [gauss(1, 16, nd) for _ in range(3)]
    out = torch.empty((1, len(mom), nd, nd, nd), dtype=torch.complex128, device="cuda")
    ctx = bb.bblock_create(L, 4, nd, form)
    for k, v in options.items():
        bb.bblock_set_option(ctx, k, v)
    rep = bb.bblock_autotune(ctx, V, *phi, mom, PAIRS, [0.5, -0.5, 0.5, -0.5], out, repeats=1)
    bb.bblock_destroy(ctx)
    return rep


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_narrow_d3_tiles_of_two_classes_make_twice_the_units(form):
    one = [(0, 0, 0), (1, 1, 1), (-1, -1, -1), (1, 0, 1), (-1, 1, 0), (0, -1, 1)]
    two = one + [(2, 2, 2), (-2, -2, -2), (2, -2, 2), (-2, 2, 1), (1, 2, -2)]
    tiles = [{round(8 * float(r["features"][7]) - 12 * float(r["features"][6]), 3) for r in tune(form, 16, 64, m, {})}
             for m in (one, two)]      # log2 of tiles per SM, the same for every slab count
    assert len(tiles[0]) == len(tiles[1]) == 1
    assert abs(tiles[1].pop() - tiles[0].pop() - 1.0) < 1e-2


def test_row_factored_columns_of_the_first_call():
    rep = tune("ozaki", 6, 40, M9, {"tc_rows": 1, "tc_cluster": 1})
    for r in rep:                      # 3 distinct n0: 120 columns in 3 tiles of 48
        assert abs(float(r["features"][9]) - 0.2) < 1e-6
