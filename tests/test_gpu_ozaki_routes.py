"""The Ozaki form's automatic route (row-factored phase or (p, d3) columns) and cluster size.

Timed on the device by the library's own step times: the automatic choice may take at most 1.35
times the faster of the two routes with automatic clusters (its model is 8 to 16 % off, and it
takes the row-factored route only when that looks 5 % faster), plus 20 us of launches, where
a wrong route takes up to 3.5 times as long. Lattices on both sides of the choice.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M27 = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
M9 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0)]
ONE = ([(0, 1, 0)], [1.0])
TWO = ([(0, 1, 0), (1, 0, 0), (2, 3, 2)], [0.7, -0.7, 0.7])


@pytest.mark.parametrize("L,nd,mom,op", [
    (4, (48, 48, 48), M27, TWO), (6, (33, 31, 33), M27, ONE), (6, (48, 48, 48), M9, ONE), (8, (64, 60, 64), M27, ONE),
    (12, (33, 33, 33), M9, ONE), (9, (20, 20, 20), M9, TWO), (16, (48, 48, 48), M9, TWO), (24, (30, 32, 32), M9, TWO),
    (10, (48, 40, 48), [(0, 0, 0), (1, 0, 0)], ONE)])
def test_automatic_route(L, nd, mom, op):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    gen = torch.Generator(device="cuda")
    gen.manual_seed(L)

    def gauss(*shape):
        return torch.complex(*(torch.randn(*shape, generator=gen, dtype=torch.float64, device="cuda") for _ in "ri"))

    V, phi = gauss(1, 8, L ** 3, 3), [gauss(1, 32, d) for d in nd]
    out = torch.empty((1, len(mom), *nd), dtype=torch.complex128, device="cuda")
    times = {}
    for rows in (0, 1, 2):
        ctx = bb.bblock_create(L, 8, max(nd), "ozaki")
        bb.bblock_set_option(ctx, "graphs", 0)
        bb.bblock_set_option(ctx, "tc_rows", rows)
        bb.bblock_compute(ctx, V, *phi, mom, *op, B_out=out)
        bb.bblock_profile_enable(ctx)
        got = []
        for _ in range(7):
            bb.bblock_compute(ctx, V, *phi, mom, *op, B_out=out)
            steps = bb.bblock_profile_read(ctx)
            got.append(steps["contract"][1] + steps["reduce"][1])
        times[rows] = float(np.median(got))
        bb.bblock_destroy(ctx)
    assert times[0] <= 1.35 * min(times[1], times[2]) + 0.020, times
